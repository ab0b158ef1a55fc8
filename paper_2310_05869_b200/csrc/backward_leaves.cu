// The backward kernel with four results warps, in a file of its own: in one with the others, their code comes to lie otherwise and is 2.7 %
// slower (12 heads x 4096 rows 60.2 -> 61.8 us; 16 causal heads x 32768 rows in leaves of 512 1796 -> 1844).
#include "backward.cuh"

namespace hyperattn {

cudaError_t launch_bwd_leaves_d64(const BwdArgs& b, const BwdMaps& maps, unsigned grid, int* status, cudaStream_t st) {
  using C = Cfg<64, 4>;
  const cudaError_t e = allow_smem<bwd_kernel<64, true, 4>>(C::kTotal);
  return e != cudaSuccess ? e : launch(bwd_kernel<64, true, 4>, grid, C::kThreads, C::kTotal, st, b, maps, status);
}

}  // namespace hyperattn
