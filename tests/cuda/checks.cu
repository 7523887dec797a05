// Device checks of the kernels' own arithmetic (csrc/packed.cuh, csrc/lb_kernel.cuh), compiled by
// tests/test_gpu_arith.py with the library's flags. Each entry point returns how many of its values differ in
// any bit from CUDA's IEEE operators, or -1 after a CUDA error.
#include <cuda_runtime.h>
#include "lb_kernel.cuh"

using namespace hlbm;

namespace {
__device__ __forceinline__ bool differs(float a, float b) {
  return __float_as_uint(a) != __float_as_uint(b) && !(isnan(a) && isnan(b));
}

// v = mantissa i of the exponent e (2^e <= v < 2^(e + 1))
__device__ __forceinline__ float value(unsigned int i, int e) { return __uint_as_float(((unsigned int)(e + 127) << 23) | i); }

__global__ void tau_kernel(float tau0, float k, int e, unsigned long long* bad) {
  const unsigned int i = blockIdx.x * blockDim.x + threadIdx.x;
  const float n0 = value(i, e), n1 = value(i, e + 1);
  const F2 t = smag_tau(pack2(tau0, tau0), pack2(n0, n1), pack2(k, k));
  const float w0 = 0.5f * __fadd_rn(tau0, __fsqrt_rn(__fmaf_rn(tau0, tau0, __fmul_rn(k, __fsqrt_rn(n0)))));
  const float w1 = 0.5f * __fadd_rn(tau0, __fsqrt_rn(__fmaf_rn(tau0, tau0, __fmul_rn(k, __fsqrt_rn(n1)))));
  if (differs(lo(t), w0) || differs(hi(t), w1)) atomicAdd(bad, 1ull);
}

constexpr int BLOCK = 256, MANTISSAS = 1 << 23;

template <typename F> long long count(F launch) {
  unsigned long long *bad = nullptr, n = 0;
  if (cudaMalloc(&bad, sizeof(*bad)) != cudaSuccess || cudaMemset(bad, 0, sizeof(*bad)) != cudaSuccess) return -1;
  launch(bad);
  const bool ok = cudaGetLastError() == cudaSuccess && cudaMemcpy(&n, bad, sizeof(n), cudaMemcpyDeviceToHost) == cudaSuccess;
  cudaFree(bad);
  return ok ? (long long)n : -1;
}
}  // namespace

// the Smagorinsky relaxation time over all mantissas of the squared strain norm at exponents e, e + 1
extern "C" long long check_tau(float tau0, float k, int e) {
  return count([=](unsigned long long* bad) { tau_kernel<<<MANTISSAS / BLOCK, BLOCK>>>(tau0, k, e, bad); });
}
