// The backward kernel of sorted nodes alone, in a file of its own (see backward_leaves.cu).
#include "backward.cuh"

namespace hyperattn {

cudaError_t launch_bwd_nodes(const BwdArgs& b, const BwdMaps& maps, unsigned grid, int* status, cudaStream_t st) {
  auto go = [&](auto d) {
    constexpr int D = decltype(d)::value;
    using C = Cfg<D, 8>;
    const cudaError_t e = allow_smem<bwd_kernel<D, kNodes, 8>>(C::kTotal);
    return e != cudaSuccess ? e : launch(bwd_kernel<D, kNodes, 8>, grid, C::kThreads, C::kTotal, st, b, maps, status);
  };
  return b.a.g.d == 64 ? go(std::integral_constant<int, 64>{}) : go(std::integral_constant<int, 128>{});
}

}  // namespace hyperattn
