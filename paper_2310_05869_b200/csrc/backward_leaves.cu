// The backward kernel with four results warps, in a file of its own.  In one with the others all of them are slower, from the same source with the
// same registers and spills; why is not known (their code comes to lie otherwise), so measure it again with another compiler.  nvcc 12.9, the pass,
// us, own file -> one file: 12 heads x 4096 rows 60.2 -> 61.4, 32 x 4096 131 -> 133, 16 causal heads x 32768 rows in leaves of 512 1767 -> 1846, of
// 4096 1675 -> 1722, 128 leaves of 4096 rows 968 -> 994; d = 128, 32 heads x 32768 rows 1602 -> 1623.
#include "backward.cuh"

namespace hyperattn {

cudaError_t launch_bwd_leaves_d64(const BwdArgs& b, const BwdMaps& maps, unsigned grid, int* status, cudaStream_t st) {
  using C = Cfg<64, 4>;
  const cudaError_t e = allow_smem<bwd_kernel<64, kBoxes, 4>>(C::kTotal);
  return e != cudaSuccess ? e : launch(bwd_kernel<64, kBoxes, 4>, grid, C::kThreads, C::kTotal, st, b, maps, status);
}

}  // namespace hyperattn
