// Finite-difference update of small 2-D FP64 grids (the planar flame), one warp per field.
//
// What bounds it: FP64 instructions. GB300 runs 1.18 TFLOP/s of FP64 FMA, about one lane per clock and
// SM sub-partition, so a warp holds its sub-partition for 32 clocks per instruction and the ~3400 FP64
// instructions of one cell's update (powers, exponentials, divisions) take 55 us however few cells
// there are; fd_step_kernel's blocks of 256 cells also leave most SMs empty (256x8 cells: 8 of 152).
// Here a block owns 32 cells with one warp per field (T, Y_k). The powers of the face viscosities and of
// the rate law are independent tasks, dealt out to the warps and passed through shared memory; then
// each warp does the faces, diffusion and sources of its own field. Formulas as in fd_cell, with the
// shared reciprocals formed once per cell.
// Measured on 256x8 cells, 4 species, one reaction, one run alone: FD + stream-collide 122 -> 34 us per step
// (FD update 113 us in 8 blocks of fd_step_kernel).
// Taken up to FD_SPLIT_MAX cells, six blocks per SM: with a seventh on some of them the warps, which all form
// the shared quantities, cost more than fd_step_kernel's blocks of 256 cells with every SM busy. Whole step,
// fd_step_kernel / this: 6 species (2 reactions) 16,384 cells 156.7 / 101.5 us, 24,576 161.8 / 148.4, 29,184
// 161.8 / 151.6, 30,208 164.5 / 187.3, 32,768 166.2 / 193.1; 4 species (1 reaction) 16,384 116.9 / 74.8,
// 24,576 121.9 / 120.7, 29,184 122.0 / 122.1, 32,768 126.0 / 128.3; 8 species 28,672 185.8 / 175.7, 32,768
// 190.4 / 206.2.
#include "fd_kernel.cuh"
#include "launch.h"

namespace hlbm {

namespace {
constexpr int SPLIT_MU = 5;                          // tasks: mu at r, -x, +x, -y, +y
constexpr int SPLIT_RATE = MAX_RX * (1 + MAX_ORD);   // then per reaction its exponential and its powers
constexpr int SPLIT_WARPS = MAX_SP + 1;

__global__ void __launch_bounds__(32 * SPLIT_WARPS) fd_split_kernel(const FDArgs<double> a) {
  __shared__ double s_fm[SPLIT_MU][32], s_rate[SPLIT_RATE][32], s_na[SPLIT_WARPS][32], s_new[SPLIT_WARPS][32];
  const FDConst<double>& c = a.c;
  const Geo& g = a.geo;
  const int N = g.N, K = c.K, lane = threadIdx.x, f = threadIdx.y, nw = K + 1;
  const int r = blockIdx.x * 32 + lane;
  const uint32_t sw = r < N ? __ldg(a.sword + r) : 0u;
  const bool active = (sw >> 31) != 0u;
  const int x = r % g.nx, y = r / g.nx;
  // neighbour kinds and indices of the radius-2 stencil (as in fd_cell's general copy)
  int k1[2][2], k2[2][2], i1[2][2], i2[2][2];
  double Tr = 1.0, Fr = c.F, sW = 0.0, Yf = 0.0;
  if (active) {
    const int pos[2] = {x, y}, dims[2] = {g.nx, g.ny}, strides[2] = {1, g.nx};
#pragma unroll
    for (int ax = 0; ax < 2; ++ax)
#pragma unroll
      for (int sd = 0; sd < 2; ++sd) {
        const int sg = sd ? 1 : -1;
        const uint32_t bits = (sw >> (4 * (2 * ax + sd))) & 15u;
        k1[ax][sd] = (int)(bits & 3u);
        k2[ax][sd] = (int)(bits >> 2);
        int p1 = pos[ax] + sg;
        p1 = p1 < 0 ? p1 + dims[ax] : (p1 >= dims[ax] ? p1 - dims[ax] : p1);
        int p2 = p1 + sg;
        p2 = p2 < 0 ? p2 + dims[ax] : (p2 >= dims[ax] ? p2 - dims[ax] : p2);
        i1[ax][sd] = k1[ax][sd] == NB_FLUID ? r + (p1 - pos[ax]) * strides[ax] : r;
        i2[ax][sd] = k2[ax][sd] == 0 ? r + (p2 - pos[ax]) * strides[ax] : i1[ax][sd];
      }
    Tr = ldg(a.T + r);
    if (a.Floc) Fr = ldg(a.Floc + r);
    for (int k = 0; k < K; ++k) {
      const double v = ldg(a.Y + (size_t)k * N + r);
      sW += v * c.inv_W[k];
      if (k == f - 1) Yf = v;
    }
  }
  const double fdr = a.pth->fd_rho_d, sT = sW * Tr;
  const double rho = active ? fdr / sT : 1.0;       // lattice units, P_th W / (R T rho_ref)
  const double rho_phys = rho * c.rho_ref_f;
  // ---- powers and exponentials, one task per warp at a time
  for (int t = f; t < SPLIT_MU + SPLIT_RATE; t += nw) {
    if (!active) continue;
    if (t < SPLIT_MU) {
      double Tn = Tr, Fn = Fr;
      if (t > 0) {
        const int ax = (t - 1) >> 1, sd = (t - 1) & 1, kk = k1[ax][sd], j = i1[ax][sd];
        if (kk == NB_FLUID) {
          Tn = ldg(a.T + j);
          if (a.Floc) Fn = ldg(a.Floc + j);
        } else if (kk == NB_INLET) {
          Tn = c.T_in;
        }
      }
      s_fm[t][lane] = Fn * (c.nu_lat * pow(Tn * c.T_ref_inv, c.mu_exp));
    } else {
      const int j = (t - SPLIT_MU) / (1 + MAX_ORD), m = (t - SPLIT_MU) % (1 + MAX_ORD) - 1;
      if (j >= c.nrx || m >= c.nord[j]) continue;
      double v;
      if (m < 0) {
        v = c.A[j] * exp(-c.ER_hi[j] / Tr);
        if (c.beta[j] != 0.0) v *= pow(Tr, c.beta[j]);
      } else {
        const int k = c.ord_k[j][m];
        const double n = c.ord_n[j][m];
        const double conc = rho_phys * fmax(ldg(a.Y + (size_t)k * N + r), 0.0) * c.inv_W[k];
        v = n == 1.0 ? conc : pow(conc, n);
      }
      s_rate[t - SPLIT_MU][lane] = v;
    }
  }
  __syncthreads();
  // ---- the warp's field
  double ur[2] = {0.0, 0.0};
  const double inv_T = active ? 1.0 / Tr : 0.0;
  if (active) {
    double q[MAX_RX], qdot = 0.0;
#pragma unroll
    for (int j = 0; j < MAX_RX; ++j) {
      q[j] = 0.0;
      if (j >= c.nrx) continue;
      q[j] = s_rate[j * (1 + MAX_ORD)][lane];
      for (int m = 0; m < c.nord[j]; ++m) q[j] *= s_rate[j * (1 + MAX_ORD) + 1 + m][lane];
      qdot += c.heat[j] * q[j];
    }
    const double inv_rho = sT / fdr, inv_rpF = inv_rho * c.inv_rho_ref / Fr;
    const double* phi = f == 0 ? a.T : a.Y + (size_t)(f - 1) * N;
    const double phin = f == 0 ? c.T_in : c.Y_in[f - 1], eps = f == 0 ? c.eps_T : c.eps_Y;
    const double pr = f == 0 ? Tr : Yf, fm0 = s_fm[0][lane];
    double adv = 0.0, dif = 0.0;
#pragma unroll
    for (int ax = 0; ax < 2; ++ax) {
      ur[ax] = ldg(a.u + (size_t)ax * N + r);
      double uf[2], ff[2];
#pragma unroll
      for (int sd = 0; sd < 2; ++sd) {
        const int kk = k1[ax][sd];
        double un = 0.0;
        if (kk == NB_FLUID) un = ldg(a.u + (size_t)ax * N + i1[ax][sd]);
        else if (kk == NB_INLET) un = ldg(a.inlet_u + ax * g.ny + y);
        else if (kk == NB_OUTLET) un = ur[ax];
        uf[sd] = 0.5 * (ur[ax] + un);
        ff[sd] = 0.5 * (fm0 + s_fm[1 + 2 * ax + sd][lane]);
      }
      const double m1 = k1[ax][0] == NB_INLET ? phin : ldg(phi + i1[ax][0]);
      const double m2 = k2[ax][0] == 2 ? phin : ldg(phi + i2[ax][0]);
      const double p1 = k1[ax][1] == NB_INLET ? phin : ldg(phi + i1[ax][1]);
      const double p2 = k2[ax][1] == 2 ? phin : ldg(phi + i2[ax][1]);
      const double dm2 = m1 - m2, dm1 = pr - m1, dp1 = p1 - pr, dp2 = p2 - p1;
      const double sm1 = fma(dm1, dm1, eps), sp1 = fma(dp1, dp1, eps), tm1 = sm1 * sm1, tp1 = sp1 * sp1;
      // upwind-far difference of each face (see fd_cell): face + v0 + (t_c d_f + 2 t_f d_c) / (2 (t_c + 2 t_f))
      const bool up = uf[1] >= 0.0, um = uf[0] >= 0.0;
      const double fP = up ? dm1 : -dp2, cP = up ? dp1 : -dp1, fM = um ? dm2 : -dp1, cM = um ? dm1 : -dm1;
      const double sfP = fma(fP, fP, eps), sfM = fma(fM, fM, eps), tfP = sfP * sfP, tfM = sfM * sfM;
      const double fp = (up ? pr : p1) + 0.5 * ((tp1 * fP + 2.0 * tfP * cP) / (tp1 + 2.0 * tfP));
      const double fm = (um ? m1 : pr) + 0.5 * ((tm1 * fM + 2.0 * tfM * cM) / (tm1 + 2.0 * tfM));
      adv += ur[ax] * (fp - fm);
      dif += ff[1] * dp1 - ff[0] * dm1;
    }
    double src;
    if (f == 0) {
      dif *= c.inv_Pr * inv_rho;
      src = c.dt_phys * qdot * inv_rpF * c.inv_cp + a.pth->fd_dT_d * inv_rho;
    } else {
      dif *= c.inv_Pr * c.inv_Le[f - 1] * inv_rho;
      double om = 0.0;
#pragma unroll
      for (int j = 0; j < MAX_RX; ++j)
        if (j < c.nrx) om += c.nu[j][f - 1] * q[j];
      src = c.dt_phys * c.W[f - 1] * om * inv_rpF;
    }
    const double NA = dif + src, pn = pr - adv + NA;
    s_na[f][lane] = NA;
    s_new[f][lane] = pn;
    if (f == 0) a.T_out[r] = pn;
    else a.Y_out[(size_t)(f - 1) * N + r] = pn;
  }
  __syncthreads();
  // ---- sums over the fields: Lambda and rho (warp 0), the sensor (warp 1), the P_th partial (last warp)
  if (f == 0 && active) {
    const double W = 1.0 / sW;
    double lam = s_na[0][lane] * inv_T;
    for (int k = 0; k < K; ++k) lam += W * c.inv_W[k] * s_na[1 + k][lane];
    a.lam_out[r] = lam;
    a.rho_out[r] = rho;
  }
  if (f == 1 && active && a.Floc_out)
    a.Floc_out[r] = sensor_floc<double>(c, s_new[0][lane], s_new[1 + c.sensor_species][lane],
                                        s_new[1 + c.sensor_oxidizer][lane]);
  if (!c.closed || f != K) return;
  double vI = 0.0, vM = 0.0;
  if (active) {
    double sWn = 0.0;
    for (int k = 0; k < K; ++k) sWn += s_new[1 + k][lane] * c.inv_W[k];
    vI = c.I_scale / (sWn * s_new[0][lane]);
    if (x == 0 && g.bc_lo[0] == BC_INLET) vM += c.M_scale * a.pth->rho_in_d * ldg(a.inlet_u + y);
    if (x == g.nx - 1 && g.bc_hi[0] == BC_OUTLET) vM -= c.M_scale * rho * ur[0];
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    vI += __shfl_down_sync(0xffffffffu, vI, o);
    vM += __shfl_down_sync(0xffffffffu, vM, o);
  }
  if (lane == 0) {
    double* out = (double*)a.partials;
    out[2 * blockIdx.x] = vI;
    out[2 * blockIdx.x + 1] = vM;
  }
}
}  // namespace

int fd_split_blocks(const Geo& g) { return (g.N + 31) / 32; }

cudaError_t launch_fd_split(const FDArgs<double>& a, cudaStream_t st) {
  fd_split_kernel<<<fd_split_blocks(a.geo), dim3(32, a.c.K + 1), 0, st>>>(a);
  return cudaGetLastError();
}

}  // namespace hlbm
