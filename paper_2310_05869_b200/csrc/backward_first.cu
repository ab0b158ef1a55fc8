// The backward kernel of leaves that write dK and dV, in a file of its own (see backward_leaves.cu).
#include "backward.cuh"

namespace hyperattn {

cudaError_t launch_bwd_first(const BwdArgs& b, const BwdMaps& maps, int results_warps, unsigned grid, int* status, cudaStream_t st) {
  auto go = [&](auto d, auto rw) {
    constexpr int D = decltype(d)::value, RW = decltype(rw)::value;
    using C = Cfg<D, RW>;
    const cudaError_t e = allow_smem<bwd_kernel<D, kFirst, RW>>(C::kTotal);
    return e != cudaSuccess ? e : launch(bwd_kernel<D, kFirst, RW>, grid, C::kThreads, C::kTotal, st, b, maps, status);
  };
  using std::integral_constant;
  if (b.a.g.d == 128) return go(integral_constant<int, 128>{}, integral_constant<int, 8>{});
  return results_warps == 4 ? go(integral_constant<int, 64>{}, integral_constant<int, 4>{}) : go(integral_constant<int, 64>{}, integral_constant<int, 8>{});
}

}  // namespace hyperattn
