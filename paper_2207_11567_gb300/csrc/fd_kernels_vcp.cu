// Finite-difference update with variable heat capacities (c_p,k(T) polynomials), 2-D and 3-D,
// FP32 and FP64: compiled apart from the constant-c_p kernels so that both build in parallel.
#include "fd_kernel.cuh"
namespace hlbm {
// Registers of an FP32 cell with variable heat capacities: 80 (3 blocks per SM; 64 at 4 blocks spill twice
// as much). Swirl burner, 4 / 3 blocks: 96x48x48 52.1 / 36.7 us, 192x96x96 228 / 206, 256x128x128 495 / 468,
// 384x192x192 1455 / 1439.
constexpr int VCP_BLOCKS = 3;
template <int D, typename R> cudaError_t launch_fd_vcp(const FDArgs<R>& a, cudaStream_t st) {
  const dim3 grid = fd_grid<D>(a.geo), block(FDShape<D>::X, FDShape<D>::Y, FDShape<D>::Z);
  // polynomial degree: linear c_p (the common case) or the full quartic
  const bool lin = a.c.varcp == 1;
  if (a.c.K == 6 && a.c.nrx == 2) {
    if (lin) fd_step_kernel<D, R, 6, 2, 1, false, VCP_BLOCKS><<<grid, block, 0, st>>>(a);
    else fd_step_kernel<D, R, 6, 2, 4, false, VCP_BLOCKS><<<grid, block, 0, st>>>(a);
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
