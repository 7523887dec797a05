// Finite-difference update with variable heat capacities (c_p,k(T) polynomials), 2-D and 3-D,
// FP32 and FP64: compiled apart from the constant-c_p kernels so that both build in parallel.
#include "fd_kernel.cuh"
namespace hlbm {
// The registers of an FP32 cell with variable heat capacities: 64 (4 blocks per SM, 700 bytes spilled)
// hide more latency, 80 (3 blocks, 368 bytes) run fewer instructions. The second wins until the blocks
// make many waves (swirl burner, 4 / 3 blocks: 61x27x37 29.1 / 23.1 us, 96x48x48 57.0 / 45.5,
// 192x96x96 251 / 238, 256x128x128 542 / 534, 320x160x160 900 / 919, 384x192x192 1575 / 1607; 2 blocks
// 44.3 at 96x48x48 and 286 at 192x96x96).
constexpr int VCP_3_BLOCKS_MAX = 5000000;
template <int D, typename R> cudaError_t launch_fd_vcp(const FDArgs<R>& a, cudaStream_t st) {
  const dim3 grid = fd_grid<D>(a.geo), block(FDShape<D>::X, FDShape<D>::Y, FDShape<D>::Z);
  // polynomial degree: linear c_p (the common case) or the full quartic
  const bool lin = a.c.varcp == 1;
  if (a.c.K == 6 && a.c.nrx == 2) {
    if (sizeof(R) == 4 && a.geo.N <= VCP_3_BLOCKS_MAX) {
      if (lin) fd_step_kernel<D, R, 6, 2, 1, false, 3><<<grid, block, 0, st>>>(a);
      else fd_step_kernel<D, R, 6, 2, 4, false, 3><<<grid, block, 0, st>>>(a);
    } else if (lin) fd_step_kernel<D, R, 6, 2, 1><<<grid, block, 0, st>>>(a);
    else fd_step_kernel<D, R, 6, 2, 4><<<grid, block, 0, st>>>(a);
  } else {
    if (lin) fd_step_kernel<D, R, 0, 0, 1><<<grid, block, 0, st>>>(a);
    else fd_step_kernel<D, R, 0, 0, 4><<<grid, block, 0, st>>>(a);
  }
  return cudaGetLastError();
}
template cudaError_t launch_fd_vcp<2, float>(const FDArgs<float>&, cudaStream_t);
template cudaError_t launch_fd_vcp<2, double>(const FDArgs<double>&, cudaStream_t);
template cudaError_t launch_fd_vcp<3, float>(const FDArgs<float>&, cudaStream_t);
template cudaError_t launch_fd_vcp<3, double>(const FDArgs<double>&, cudaStream_t);
}  // namespace hlbm
