// Device checks of the kernels' own arithmetic (csrc/packed.cuh, csrc/lb_kernel.cuh), compiled by
// tests/test_gpu_arith.py with the library's flags. Each entry point returns how many of its values differ in
// any bit from CUDA's IEEE operators, or -1 after a CUDA error.
#include <cuda_runtime.h>
#include "fd_kernel.cuh"
#include "lb_kernel.cuh"

using namespace hlbm;

namespace {
// other bits, but for the sign of a zero and a NaN's payload
__device__ __forceinline__ bool differs(float a, float b) { return a != b && !(isnan(a) && isnan(b)); }

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

// reciprocals and roots of every mantissa at the exponents e and e + 1, alone and in pairs, both signs
__global__ void rcp_kernel(int e, unsigned long long* bad) {
  const unsigned int i = blockIdx.x * blockDim.x + threadIdx.x;
  const float x = value(i, e), y = -value(i, e + 1);
  const F2 p = rcp_(pack2(x, y));
  const float a = __frcp_rn(x), b = __frcp_rn(y);
  if (differs(rcp_(x), a) || differs(rcp_(y), b) || differs(lo(p), a) || differs(hi(p), b)) atomicAdd(bad, 1ull);
}

__global__ void sqrt_kernel(int e, unsigned long long* bad) {
  const unsigned int i = blockIdx.x * blockDim.x + threadIdx.x;
  const float x = value(i, e), y = value(i, e + 1);
  const F2 p = sqrt_pos(pack2(x, y)), q = sqrt_rn(pack2(x, y));
  const float a = __fsqrt_rn(x), b = __fsqrt_rn(y);
  if (differs(lo(p), a) || differs(hi(p), b) || differs(lo(q), a) || differs(hi(q), b)) atomicAdd(bad, 1ull);
}

// 32 pseudo-random bits of n (multiply-xorshift mixing)
__device__ __forceinline__ unsigned int mix(unsigned int n) {
  n = (n ^ (n >> 16)) * 0x45d9f3bu;
  n = (n ^ (n >> 15)) * 0x2c1b3c6du;
  return n ^ (n >> 16);
}

// quotients of random pairs, a in 2^ea_lo .. 2^ea_hi, |b| in 2^-20 .. 2^20; off: units in the last place allowed
__global__ void div_kernel(int ea_lo, int ea_hi, int off, unsigned long long* bad) {
  const unsigned int i = blockIdx.x * blockDim.x + threadIdx.x;
  const unsigned int ma = mix(3 * i), mb = mix(3 * i + 1), me = mix(3 * i + 2);
  const float a = value(ma & 0x7fffffu, ea_lo + (int)((me >> 8) % (unsigned)(ea_hi - ea_lo)));
  const float b = ((me >> 31) ? -1.0f : 1.0f) * value(mb & 0x7fffffu, (int)(me & 0xffu) % 40 - 20);
  const float q = div_(a, b, rcp_(b)), w = __fdiv_rn(a, b);
  const int d = (int)(__float_as_uint(q) & 0x7fffffffu) - (int)(__float_as_uint(w) & 0x7fffffffu);
  if (d < -off || d > off || signbit(q) != signbit(w)) atomicAdd(bad, 1ull);
}

// flame sensor at temperatures of a cell that holds no gas yet (0) or has blown up
__global__ void sensor_kernel(const float* T, int n, float* out) {
  FDConst<float> c{};
  c.F = 8.0f;
  c.sensor_Ta = 8400.0f;
  c.sensor_beta = 10.0f;
  c.inv_wref = 1e5f;
  if ((int)threadIdx.x < n) out[threadIdx.x] = sensor_floc<float>(c, T[threadIdx.x], 0.04f, 0.2f);
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

extern "C" long long check_rcp(int e) {
  return count([=](unsigned long long* bad) { rcp_kernel<<<MANTISSAS / BLOCK, BLOCK>>>(e, bad); });
}
extern "C" long long check_sqrt(int e) {
  return count([=](unsigned long long* bad) { sqrt_kernel<<<MANTISSAS / BLOCK, BLOCK>>>(e, bad); });
}
extern "C" long long check_div(int ea_lo, int ea_hi, int off) {
  return count([=](unsigned long long* bad) { div_kernel<<<(1 << 24) / BLOCK, BLOCK>>>(ea_lo, ea_hi, off, bad); });
}
// F_loc at the n <= 32 temperatures T (device arrays)
extern "C" int sensor(const float* T, int n, float* out) {
  sensor_kernel<<<1, 32>>>(T, n, out);
  return (int)cudaDeviceSynchronize();
}
