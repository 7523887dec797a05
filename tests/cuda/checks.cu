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

// One thermal D3Q27 stream-collide at the default rates with one thread per cell (two = 0) or two cells per
// thread (two = 1), populations of FP16 (half = 1) or FP32; bc: low and high code of x, y, z; device arrays.
__device__ PthState g_pth;
__device__ int g_flag;

template <typename S> cudaError_t stream_collide_of(int two, const LBArgs<float>& a) {
  if (two) return launch_pair<3, S, true, false>(a, 0, false);
  const dim3 grid((a.geo.nx + LB_BLOCK - 1) / LB_BLOCK, a.geo.ny, a.geo.nz);
  return launch_ex<LBArgs<float>>(lb_step_kernel<3, S, float, true, COLL_CUMULANT_FULL, false>, grid, dim3(LB_BLOCK), 0, false, a);
}

extern "C" int stream_collide(int two, int half, const int* n, const int* bc, const void* g_in, const unsigned int* links,
                              const float* rho, const float* lam, const float* T, const float* inlet, const float* u_in,
                              float lb_lam, float omega_b, float smag_k, float P_ref, void* g_out, float* u_out,
                              float* ph) {
  LBArgs<float> a{};
  a.geo = Geo{n[0], n[1], n[2], n[0] * n[1] * n[2], {bc[0], bc[2], bc[4]}, {bc[1], bc[3], bc[5]}};
  PthState p{};
  p.lb_lam = lb_lam;
  if (cudaMemcpyToSymbol(g_pth, &p, sizeof(p)) != cudaSuccess) return -1;
  void *pth = nullptr, *flag = nullptr;
  if (cudaGetSymbolAddress(&pth, g_pth) != cudaSuccess || cudaGetSymbolAddress(&flag, g_flag) != cudaSuccess) return -1;
  a.g_in = g_in;
  a.g_out = g_out;
  a.links = links;
  a.rho = rho;
  a.lam = lam;
  a.T = T;
  a.inlet_u = inlet;
  a.u_in = u_in;
  a.u = u_out;
  a.write_u = 1;
  a.ph_out = ph;
  a.pth = (const PthState*)pth;
  a.flag = (int*)flag;
  a.nu_lat = 0.002f;
  a.T_ref_inv = 1.0f / 300.0f;
  a.mu_exp = 0.7f;
  a.smag_k = smag_k;
  a.P_ref = P_ref;
  a.omega_b = omega_b;
  a.om3 = a.om4 = a.om5 = a.om6 = 1.0f;
  const cudaError_t e = half ? stream_collide_of<__half>(two, a) : stream_collide_of<float>(two, a);
  return e != cudaSuccess ? (int)e : (int)cudaDeviceSynchronize();
}
