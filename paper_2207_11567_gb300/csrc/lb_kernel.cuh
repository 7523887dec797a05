// Fused pull-stream + collide kernels of the pressure/momentum lattice Boltzmann solver
// (Section 2.1-2.2), one or two cells per thread, lattice units (c_s^2 = 1/3).
//
// Per fluid cell:
//   stream   g_i(r) = g*_i(r - c_i) (Eq. 1, pull), bounce-back g_i = g*_{Q-1-i}(r) on links
//            marked in the cell's link word, plus 2 w_i rho (c_i . u_w) on low-x inlet links;
//   moments  P_h = sum g + rho Lambda / 6, u = 3 sum c g / rho (Eq. 7);
//   source   Xi_i = w_i [ (c.u/cs2 + (c.u)^2/(2 cs4) - u^2/(2 cs2)) cs2 (c_i - u).grad rho
//            + rho cs2 Lambda ] (Eq. 2 with Eq. 4 inserted);
//   precond  f'_i = 3 (g_i + Xi_i / 2) / rho (Eq. 13); p' = sum f'; h = f' - (p' - 1) w;
//   collide  cumulants of h about u (central moments by the axis-by-axis transform), shear rate
//            1/tau with tau from Eq. 12 plus the Smagorinsky closure, trace rate omega_b,
//            orders 3..6 with omega_hi; or the single-rate (BGK) relaxation of h to f^eq(1, u);
//   post     g*_i = rho/3 (h*_i + (p' - 1) w_i) + Xi_i / 2 (Eq. 8), stored shifted as
//            (g* - w P_ref) / w.
// Arithmetic is arranged so that no O(1) offset is ever added and cancelled again (which costs
// FP32 its precision): with q_i = g_i / w_i - P_ref, xi_i = Xi_i / w_i, s_i = q_i + xi_i / 2 and
// S = sum_j w_j s_j, one has h_i / w_i - 1 = 3 (s_i - S) / rho and
// g*_i / w_i - P_ref = rho/3 (h*_i / w_i - 1) + S + xi_i / 2; the cumulant collision works on
// h - h_eq with h_eq the product-form equilibrium, whose central moments are known exactly.
#pragma once
#include "packed.cuh"

namespace hlbm {

// central-moment transform of one line of three values (c = -1, 0, +1) about velocity u
template <typename R> __device__ __forceinline__ void chim_fwd(R& a, R& b, R& c, const R u) {
  const R m0 = a + b + c;
  const R d = c - a;
  const R s = c + a;
  a = m0;
  b = d - u * m0;
  c = s - R(2) * u * d + u * u * m0;
}
template <typename R> __device__ __forceinline__ void chim_bwd(R& a, R& b, R& c, const R u) {
  const R m0 = a, m1 = b, m2 = c;
  const R k1 = m1 + u * m0;
  const R k2 = m2 + R(2) * u * m1 + u * u * m0;
  a = R(0.5) * (k2 - k1);
  b = m0 - k2;
  c = R(0.5) * (k2 + k1);
}

// x^y for x > 0: FP32 via the hardware log2 / exp2 (relative error a few 1e-7), FP64 with pow
template <typename R> __device__ __forceinline__ R pw(R x, R y);
template <> __device__ __forceinline__ float pw<float>(float x, float y) { return exp2f(y * __log2f(x)); }
template <> __device__ __forceinline__ double pw<double>(double x, double y) { return pow(x, y); }

// Cumulant relaxation in deviation form. n[] holds the central moments (slot a + 3b [+ 9c])
// of e = h - h_eq, where h_eq is the product-form equilibrium at the cell velocity; the central
// moments of h_eq are exactly 0 for any odd index and (1/3)^k for k indices equal to 2, so the
// full central moments are kappa = kappa_eq + n. All formulas below are the cumulant relations
// (partition formula, unit density) rewritten in n, so that every FP32 quantity is small.
template <bool FULL, typename R>
__device__ __forceinline__ void cumulant_relax2(R* n, const R om, const R omb, const R om3, const R om4) {
  const R third = R(1) / R(3);
  const R n20 = n[2], n02 = n[6], n11 = n[4];
  const R C22 = FULL ? R(0) : n[8] - third * (n20 + n02) - n20 * n02 - R(2) * n11 * n11;
  const R tr = R(0.5) * (n20 + n02);
  const R o1 = R(1) - om, ob = R(1) - omb;
  const R s20 = o1 * (n20 - tr) + ob * tr;
  const R s02 = o1 * (n02 - tr) + ob * tr;
  const R s11 = o1 * n11;
  n[2] = s20; n[6] = s02; n[4] = s11;
  if constexpr (FULL) {
    n[5] = R(0);
    n[7] = R(0);
    n[8] = third * (s20 + s02) + s20 * s02 + R(2) * s11 * s11;
  } else {
    n[5] *= (R(1) - om3);
    n[7] *= (R(1) - om3);
    n[8] = (R(1) - om4) * C22 + third * (s20 + s02) + s20 * s02 + R(2) * s11 * s11;
  }
}

template <bool FULL, typename R>
__device__ __forceinline__ void cumulant_relax3(R* n, const R om, const R omb, const R om3,
                                                const R om4, const R om5, const R om6) {
#define K(a, b, c) n[(a) + 3 * (b) + 9 * (c)]
  const R third = R(1) / R(3), ninth = R(1) / R(9);
  const R a = K(2, 0, 0), b = K(0, 2, 0), c = K(0, 0, 2);
  const R n110 = K(1, 1, 0), n101 = K(1, 0, 1), n011 = K(0, 1, 1);
  const R n210 = K(2, 1, 0), n201 = K(2, 0, 1), n120 = K(1, 2, 0);
  const R n021 = K(0, 2, 1), n102 = K(1, 0, 2), n012 = K(0, 1, 2), n111 = K(1, 1, 1);
  const R n211 = K(2, 1, 1), n121 = K(1, 2, 1), n112 = K(1, 1, 2);
  const R n220 = K(2, 2, 0), n202 = K(2, 0, 2), n022 = K(0, 2, 2);
  // forward cumulants of order 4, 5, 6 (not needed when those orders relax fully)
  R C211 = R(0), C121 = R(0), C112 = R(0), C220 = R(0), C202 = R(0), C022 = R(0);
  R C221 = R(0), C212 = R(0), C122 = R(0), C222 = R(0);
  if constexpr (!FULL) {
    C211 = n211 - third * n011 - a * n011 - R(2) * n110 * n101;
    C121 = n121 - third * n101 - b * n101 - R(2) * n110 * n011;
    C112 = n112 - third * n110 - c * n110 - R(2) * n101 * n011;
    C220 = n220 - third * (a + b) - a * b - R(2) * n110 * n110;
    C202 = n202 - third * (a + c) - a * c - R(2) * n101 * n101;
    C022 = n022 - third * (b + c) - b * c - R(2) * n011 * n011;
    C221 = K(2, 2, 1) - ((third + a) * n021 + (third + b) * n201 + R(4) * n110 * n111 +
                                 R(2) * n101 * n120 + R(2) * n011 * n210);
    C212 = K(2, 1, 2) - ((third + a) * n012 + (third + c) * n210 + R(4) * n101 * n111 +
                                 R(2) * n110 * n102 + R(2) * n011 * n201);
    C122 = K(1, 2, 2) - ((third + c) * n120 + (third + b) * n102 + R(4) * n011 * n111 +
                                 R(2) * n101 * n021 + R(2) * n110 * n012);
    C222 = K(2, 2, 2) + ninth * (a + b + c) - third * (n022 + n202 + n220) -
                   (a * n022 + b * n202 + c * n220) -
                   R(4) * (n110 * n112 + n101 * n121 + n011 * n211) -
                   (R(2) * (n210 * n012 + n201 * n021 + n120 * n102) + R(4) * n111 * n111) +
                   R(2) * third * (a * b + b * c + c * a) + R(2) * a * b * c +
                   R(4) * ((third + a) * n011 * n011 + (third + b) * n101 * n101 + (third + c) * n110 * n110) +
                   R(16) * n110 * n101 * n011;
  }
  // second order: trace deviation (rate omega_b) and deviatoric part (rate omega)
  const R tr = third * (a + b + c);
  const R o1 = R(1) - om, ob = R(1) - omb;
  const R s200 = o1 * (a - tr) + ob * tr;
  const R s020 = o1 * (b - tr) + ob * tr;
  const R s002 = o1 * (c - tr) + ob * tr;
  const R s110 = o1 * n110, s101 = o1 * n101, s011 = o1 * n011;
  const R o3 = FULL ? R(0) : R(1) - om3;
  const R s210 = FULL ? R(0) : o3 * n210, s201 = FULL ? R(0) : o3 * n201, s120 = FULL ? R(0) : o3 * n120;
  const R s021 = FULL ? R(0) : o3 * n021, s102 = FULL ? R(0) : o3 * n102, s012 = FULL ? R(0) : o3 * n012;
  const R s111 = FULL ? R(0) : o3 * n111;
  const R o4 = FULL ? R(0) : R(1) - om4, o5 = FULL ? R(0) : R(1) - om5, o6 = FULL ? R(0) : R(1) - om6;
  const R D211 = FULL ? R(0) : o4 * C211, D121 = FULL ? R(0) : o4 * C121, D112 = FULL ? R(0) : o4 * C112;
  const R D220 = FULL ? R(0) : o4 * C220, D202 = FULL ? R(0) : o4 * C202, D022 = FULL ? R(0) : o4 * C022;
  // back to central moments (deviation form)
  K(2, 0, 0) = s200; K(0, 2, 0) = s020; K(0, 0, 2) = s002;
  K(1, 1, 0) = s110; K(1, 0, 1) = s101; K(0, 1, 1) = s011;
  K(2, 1, 0) = s210; K(2, 0, 1) = s201; K(1, 2, 0) = s120;
  K(0, 2, 1) = s021; K(1, 0, 2) = s102; K(0, 1, 2) = s012; K(1, 1, 1) = s111;
  K(2, 1, 1) = D211 + (third + s200) * s011 + R(2) * s110 * s101;
  K(1, 2, 1) = D121 + (third + s020) * s101 + R(2) * s110 * s011;
  K(1, 1, 2) = D112 + (third + s002) * s110 + R(2) * s101 * s011;
  K(2, 2, 0) = D220 + third * (s200 + s020) + s200 * s020 + R(2) * s110 * s110;
  K(2, 0, 2) = D202 + third * (s200 + s002) + s200 * s002 + R(2) * s101 * s101;
  K(0, 2, 2) = D022 + third * (s020 + s002) + s020 * s002 + R(2) * s011 * s011;
  K(2, 2, 1) = (FULL ? R(0) : o5 * C221) + (third + s200) * s021 + (third + s020) * s201 + R(4) * s110 * s111 +
               R(2) * s101 * s120 + R(2) * s011 * s210;
  K(2, 1, 2) = (FULL ? R(0) : o5 * C212) + (third + s200) * s012 + (third + s002) * s210 + R(4) * s101 * s111 +
               R(2) * s110 * s102 + R(2) * s011 * s201;
  K(1, 2, 2) = (FULL ? R(0) : o5 * C122) + (third + s002) * s120 + (third + s020) * s102 + R(4) * s011 * s111 +
               R(2) * s101 * s021 + R(2) * s110 * s012;
  const R A = (third + s200) * D022 + (third + s020) * D202 + (third + s002) * D220;
  const R B = R(4) * (s110 * D112 + s101 * D121 + s011 * D211);
  const R C3 = R(2) * (s210 * s012 + s201 * s021 + s120 * s102) + R(4) * s111 * s111;
  const R Dd = ninth * (s200 + s020 + s002) + third * (s200 * s020 + s020 * s002 + s002 * s200) +
               s200 * s020 * s002 +
               R(2) * ((third + s200) * s011 * s011 + (third + s020) * s101 * s101 + (third + s002) * s110 * s110) +
               R(8) * s110 * s101 * s011;
  K(2, 2, 2) = (FULL ? R(0) : o6 * C222) + A + B + C3 + Dd;
#undef K
}

// Central moments of the product-form equilibrium minus those of the rest weights w, both
// about u, for the moment (a, b, c): prod ke - prod (ke + dl) with ke = (1, 0, 1/3) and
// dl = (0, -u, u^2) per axis, expanded so that only small terms are formed.
template <int D, int J, typename R>
__device__ __forceinline__ R delta_eq(const R* dx, const R* dy, const R* dz) {
  constexpr int a = J % 3, b = (J / 3) % 3, c = J / 9;
  const R kx = a == 0 ? R(1) : (a == 1 ? R(0) : R(1) / R(3));
  const R ky = b == 0 ? R(1) : (b == 1 ? R(0) : R(1) / R(3));
  const R kz = c == 0 ? R(1) : (c == 1 ? R(0) : R(1) / R(3));
  const R ex = dx[a], ey = dy[b], ez = (D == 3) ? dz[c] : R(0);
  if constexpr (D == 2) return -(ex * ky + kx * ey + ex * ey);
  return -(ex * ky * kz + kx * ey * kz + kx * ky * ez + ex * ey * kz + ex * ky * ez + kx * ey * ez + ex * ey * ez);
}

// m[J] += sign * delta_eq for the moments whose order a + b + c lies in [LO, HI]
template <int D, typename R, int J, int LO = 0, int HI = 6>
__device__ __forceinline__ void add_delta_eq(R* m, const R* dx, const R* dy, const R* dz, const R sign) {
  if constexpr (J < Lat<D>::Q) {
    constexpr int order = J % 3 + (J / 3) % 3 + J / 9;
    if constexpr (order >= LO && order <= HI) m[J] += sign * delta_eq<D, J, R>(dx, dy, dz);
    add_delta_eq<D, R, J + 1, LO, HI>(m, dx, dy, dz, sign);
  }
}

// Relaxation time with the Smagorinsky closure: n2 = Pi : Pi of the deviator, k = smag_k. Both roots are
// rounded as the IEEE ones (a hardware root of the norm, one unit off, gained no time: cold swirl
// 256x128x128, 20 steps with it / with this, FP32 2826 / 2826 us, FP16 2082 / 2084).
template <typename V> __device__ __forceinline__ V smag_tau(V tau0, V n2, V k) {
  return splat<V>(0.5) * (tau0 + sqrt_pos(fma_(tau0, tau0, k * sqrt_rn(n2))));
}

// ------------------------------------------------------------------ collision, full relaxation
// Cumulant collision with full relaxation of the orders 3..6 (the default rates), Eq. 2, 7, 13 and
// 9-12 of one cell, for V = float, double or F2 (two cells): q[] comes in as the pulled populations
// q_i = g_i / w_i - P_ref and goes out as the new stored ones. It works on sums over the lattice
// instead of per-population terms, one axis at a time:
// * The ten raw moments M_0, M_a, M_ab = 6^D sum_i w_i q_i (1, c_a, c_a c_b): per line of three
//   (1/6, 2/3, 1/6)(q_-, q_0, q_+) the sums q_- + 4 q_0 + q_+, q_+ - q_-, q_+ + q_-, so that no
//   weight is multiplied in.
// * u_a = M_a / (2^D m), m = rho 3^(D-1): the reciprocal and one residual correction, which
//   keeps the momentum of the stored populations (they are rebuilt from u with the same m) free of
//   a rounding that would repeat every step. With G = u . grad rho and L = rho cs2 Lambda, the
//   closed forms of the source's moments (k_0 = L + G/3, k_ab = L u_a u_b + (g_a u_b + g_b u_a)/9
//   [+ L/3 + G/9 for a = b]) leave for the second central moments of h - h_eq
//     n_ab = (3/rho) (A_ab - delta_ab A_0 / 3) - u_a u_b (1 + G / (2 rho)) + (g_a u_b + g_b u_a)/(6 rho)
//   (A = M / 6^D; L cancels).
// * Relaxed to s_ab (deviator at 1/tau, trace at omega_b), the populations h* have unit mass,
//   velocity u, covariance 1/3 + s_ab and no cumulants beyond: their raw moments follow from
//   Isserlis' theorem, written as deviations from those of the rest weights so that every quantity
//   is small.
// * Back to populations one axis at a time, (m_2 - m_1, m_0 - m_2, m_2 + m_1); the factors 1/2 of
//   that inverse, 1 / w_i and rho / 3 together are m / 2^(number of zero components of c_i).
// * The half source xi_i / 2 of Eq. 8 is, along x, a polynomial of degree 2 in c_x (c_x^3 = c_x)
//   whose coefficients are formed once per line and added there.
// About 480 operations per cell of D3Q27, against about 1080 with the transforms of all 27 central
// moments and per-population source terms. Taken by isothermal and 2-D runs from lb_pair_kernel and by
// FP64 (planar flame 256x8: stream-collide 22.8 -> 16.5 us); error of u after 20 steps of the cold swirl
// against 64-bit values 2.4e-7 before, 1.5e-7 with it.
template <int D, typename V, bool THERMAL> struct LBCell {
  V rho, lam;           // density, Lambda (with the thermodynamic-pressure term)
  V gx, gy, gz;         // density gradient
  V u[3], usq;          // out: velocity, its square
  V psum, rl3;          // out: sum of g - P_ref, rho cs2 Lambda
};

template <int D, typename V, bool THERMAL, typename R>
__device__ __forceinline__ void collide_full(V* q, LBCell<D, V, THERMAL>& c, const V nu3, const LBArgs<R>& a) {
  constexpr int Q = Lat<D>::Q;
  const V one = splat<V>(1.0), two = splat<V>(2.0), four = splat<V>(4.0), half = splat<V>(0.5);
  const V third = splat<V>(1.0 / 3.0), zero = splat<V>(0.0);
  // raw moments: x lines, then y, then z; slot a + 3 b (+ 9 c) of m[]
#pragma unroll
  for (int j = 0; j < Q / 3; ++j) {
    const V s = q[3 * j] + q[3 * j + 2], d = q[3 * j + 2] - q[3 * j];
    q[3 * j] = fma_(four, q[3 * j + 1], s);
    q[3 * j + 1] = d;
    q[3 * j + 2] = s;
  }
#pragma unroll
  for (int k = 0; k < Q / 9; ++k) {
    V* p = q + 9 * k;
    {
      const V s = p[0] + p[6], d = p[6] - p[0];
      p[0] = fma_(four, p[3], s);
      p[3] = d;
      p[6] = s;
    }
    {
      const V s = p[1] + p[7], d = p[7] - p[1];
      p[1] = fma_(four, p[4], s);
      p[4] = d;
    }
    p[2] = fma_(four, p[5], p[2] + p[8]);
  }
  V M0, M[3], Md[3], Mo[3];  // Md: xx, yy, zz; Mo: xy, xz, yz
  if constexpr (D == 3) {
    const V s0 = q[0] + q[18];
    M0 = fma_(four, q[9], s0);
    M[2] = q[18] - q[0];
    Md[2] = s0;
    M[0] = fma_(four, q[10], q[1] + q[19]);
    Mo[1] = q[19] - q[1];
    M[1] = fma_(four, q[12], q[3] + q[21]);
    Mo[2] = q[21] - q[3];
    Md[0] = fma_(four, q[11], q[2] + q[20]);
    Md[1] = fma_(four, q[15], q[6] + q[24]);
    Mo[0] = fma_(four, q[13], q[4] + q[22]);
  } else {
    M0 = q[0];
    M[0] = q[1];
    M[1] = q[3];
    M[2] = Md[2] = Mo[1] = Mo[2] = zero;
    Md[0] = q[2];
    Md[1] = q[6];
    Mo[0] = q[4];
  }
  // velocity and pressure
  const V mm = splat<V>(D == 3 ? 9.0 : 3.0) * c.rho, m4 = splat<V>(D == 3 ? 8.0 : 4.0) * mm;
  const V im4 = rcp_(m4);
#pragma unroll
  for (int d = 0; d < D; ++d) {
    const V t = M[d] * im4;
    c.u[d] = fma_(fma_(zero - m4, t, M[d]), im4, t);
  }
  if constexpr (D == 2) c.u[2] = zero;
  const V ux = c.u[0], uy = c.u[1], uz = c.u[2];
  const V uxx = ux * ux, uyy = uy * uy, uzz = D == 3 ? uz * uz : zero;
  c.usq = D == 3 ? uxx + uyy + uzz : uxx + uyy;
  // 6^-D in two parts: the sum must not lose or gain a fixed fraction each step
  constexpr double sc = D == 3 ? 1.0 / 216.0 : 1.0 / 36.0;
  const V sc_hi = splat<V>(sc);
  c.psum = sizeof(R) == 4 ? fma_(M0, splat<V>(sc - (double)(float)sc), M0 * sc_hi) : M0 * sc_hi;
  V S = c.psum;
  c.rl3 = zero;
  V G = zero, hL = zero, c1 = one, c2 = zero;
  if constexpr (THERMAL) {
    c.rl3 = c.rho * c.lam * third;
    G = fma_(ux, c.gx, uy * c.gy);
    if constexpr (D == 3) G = fma_(uz, c.gz, G);
    hL = half * c.rl3;
    S = fma_(splat<V>(1.0 / 6.0), G, S + hL);
    c2 = splat<V>(D == 3 ? 12.0 : 2.0) * im4;  // 1 / (6 rho)
    c1 = fma_(splat<V>(3.0) * c2, G, one);     // 1 + G / (2 rho)
  }
  // second central moments of h - h_eq. (3/rho) / 6^D = im4 (D3Q27: 3 / (216 rho) = 1 / (72 rho);
  // D2Q9: 3 / (36 rho) = 1 / (12 rho))
  const V M0t = M0 * third;
  V nd[3], no[3];  // xx, yy, zz; xy, xz, yz
  {
    const V vx = c1 * ux, vy = c1 * uy, vz = c1 * uz;
    V b[3] = {ux * vx, uy * vy, uz * vz}, bo[3] = {ux * vy, ux * vz, uy * vz};
    if constexpr (THERMAL) {
      const V hx = c2 * c.gx, hy = c2 * c.gy, hz = c2 * c.gz;
      const V tx = two * hx, ty = two * hy, tz = two * hz;
      b[0] = b[0] - tx * ux;
      b[1] = b[1] - ty * uy;
      bo[0] = bo[0] - fma_(hx, uy, hy * ux);
      if constexpr (D == 3) {
        b[2] = b[2] - tz * uz;
        bo[1] = bo[1] - fma_(hx, uz, hz * ux);
        bo[2] = bo[2] - fma_(hy, uz, hz * uy);
      }
    }
#pragma unroll
    for (int d = 0; d < D; ++d) nd[d] = fma_(im4, Md[d] - M0t, zero - b[d]);
    if constexpr (D == 2) nd[2] = zero;
    no[0] = fma_(im4, Mo[0], zero - bo[0]);
    no[1] = D == 3 ? fma_(im4, Mo[1], zero - bo[1]) : zero;
    no[2] = D == 3 ? fma_(im4, Mo[2], zero - bo[2]) : zero;
  }
  const V tr = (D == 3 ? third : half) * (D == 3 ? nd[0] + nd[1] + nd[2] : nd[0] + nd[1]);
#pragma unroll
  for (int d = 0; d < D; ++d) nd[d] = nd[d] - tr;
  // relaxation time (Eq. 12) with the Smagorinsky closure on the deviator
  const V inv_rho = splat<V>(D == 3 ? 72.0 : 12.0) * im4;
  const V tau0 = THERMAL ? fma_(nu3, inv_rho, half) : nu3 + half;
  V tau = tau0;
  if (a.smag_k > R(0)) {
    V n2 = fma_(nd[0], nd[0], nd[1] * nd[1]), o2 = no[0] * no[0];
    if constexpr (D == 3) {
      n2 = fma_(nd[2], nd[2], n2);
      o2 = fma_(no[1], no[1], fma_(no[2], no[2], o2));
    }
    n2 = fma_(two, o2, n2);
    tau = smag_tau(tau0, n2, splat<V>(a.smag_k));
  }
  const V o1 = one - rcp_(tau);
  const V obt = splat<V>(R(1) - a.omega_b) * tr;
  // relaxed covariance deviations s and raw second moments P = s + u u, T = 1/3 + P
  const V sxx = fma_(o1, nd[0], obt), syy = fma_(o1, nd[1], obt), sxy = o1 * no[0];
  const V Pxx = sxx + uxx, Pyy = syy + uyy, uxy = ux * uy, Pxy = sxy + uxy;
  const V Txx = third + Pxx, Tyy = third + Pyy;
  const V ux2 = two * ux, uy2 = two * uy;
  // raw moments of h* minus those of the rest weights, slots a + 3 b + 9 c
  q[1] = ux; q[3] = uy; q[2] = Pxx; q[6] = Pyy; q[4] = Pxy;
  q[5] = fma_(uy, Txx, ux2 * sxy);
  q[7] = fma_(ux, Tyy, uy2 * sxy);
  q[8] = fma_(two * sxy, fma_(two, Pxy, zero - sxy), fma_(Txx, Pyy, third * Pxx));
  if constexpr (D == 3) {
    const V szz = fma_(o1, nd[2], obt), sxz = o1 * no[1], syz = o1 * no[2];
    const V Pzz = szz + uzz, uxz = ux * uz, uyz = uy * uz, Pxz = sxz + uxz, Pyz = syz + uyz;
    const V Tzz = third + Pzz, uz2 = two * uz;
    const V sxy2 = two * sxy, sxz2 = two * sxz, syz2 = two * syz;
    q[9] = uz; q[18] = Pzz; q[10] = Pxz; q[12] = Pyz;
    q[11] = fma_(uz, Txx, ux2 * sxz);  // xxz
    q[15] = fma_(uz, Tyy, uy2 * syz);  // yyz
    q[19] = fma_(ux, Tzz, uz2 * sxz);  // xzz
    q[21] = fma_(uy, Tzz, uz2 * syz);  // yzz
    q[13] = fma_(ux, Pyz, fma_(uy, sxz, uz * sxy));  // xyz
    q[20] = fma_(sxz2, fma_(two, Pxz, zero - sxz), fma_(Txx, Pzz, third * Pxx));  // xxzz
    q[24] = fma_(syz2, fma_(two, Pyz, zero - syz), fma_(Tyy, Pzz, third * Pyy));  // yyzz
    q[14] = fma_(sxz2, Pxy, fma_(sxy2, uxz, Txx * Pyz));  // xxyz
    q[16] = fma_(syz2, Pxy, fma_(sxy2, uyz, Tyy * Pxz));  // xyyz
    q[22] = fma_(syz2, Pxz, fma_(sxz2, uyz, Tzz * Pxy));  // xyzz
    const V ninth = splat<V>(1.0 / 9.0);
    q[17] = fma_(uz, ninth + q[8], fma_(sxz2, q[7], syz2 * q[5]));    // xxyyz
    q[23] = fma_(uy, ninth + q[20], fma_(sxy2, q[19], syz2 * q[11]));  // xxyzz
    q[25] = fma_(ux, ninth + q[24], fma_(sxy2, q[21], sxz2 * q[15]));  // xyyzz
    q[26] = fma_(uz, q[17], fma_(sxz2, q[16], fma_(syz2, q[14], fma_(ninth, szz, (third + szz) * q[8]))));
    // back along z: slots of equal (a, b); the mass moment is zero
#pragma unroll
    for (int j = 0; j < 9; ++j) {
      const V m1 = q[j + 9], m2 = q[j + 18];
      q[j + 9] = j == 0 ? zero - m2 : q[j] - m2;
      q[j] = m2 - m1;
      q[j + 18] = m2 + m1;
    }
  }
  // back along y
#pragma unroll
  for (int k = 0; k < Q / 9; ++k)
#pragma unroll
    for (int x = 0; x < 3; ++x) {
      V* p = q + 9 * k + x;
      const V m1 = p[3], m2 = p[6];
      const bool mass = D == 2 && x == 0;
      p[3] = mass ? zero - m2 : p[0] - m2;
      p[0] = m2 - m1;
      p[6] = m2 + m1;
    }
  // back along x, with the scale to stored populations, S and the half source
  V fac[D + 1];  // by number of nonzero components
  fac[D] = mm;
#pragma unroll
  for (int k = D - 1; k >= 0; --k) fac[k] = half * fac[k + 1];
  V hgx = zero, hgy = zero, hgz = zero, hG = zero, e2 = zero, eb = zero;
  if constexpr (THERMAL) {
    hgx = half * c.gx;
    hgy = half * c.gy;
    hgz = half * c.gz;
    hG = half * G;
    e2 = splat<V>(1.5) * uxx;
    eb = splat<V>(-0.5) * c.usq;
    S = S + hL;
  }
#pragma unroll
  for (int j = 0; j < Q / 3; ++j) {
    const int jy = j % 3 - 1, jz = D == 3 ? j / 3 - 1 : 0;
    const int k = (jy != 0) + (jz != 0);
    const V m0 = q[3 * j], m1 = q[3 * j + 1], m2 = q[3 * j + 2];
    V p0 = S, p1 = zero, p02 = S;
    if constexpr (THERMAL) {
      // xi / 2 = e (c . g - G) / 2 with e = e0 + e1 c_x + e2 c_x^2 and c . g - G = b + g_x c_x
      V e0 = eb, e1 = ux, b = zero - hG;
      if (k) {
        const V ay = jy > 0 ? uy : zero - uy, az = jz > 0 ? uz : zero - uz;
        const V au = jy ? (jz ? (jz > 0 ? ay + uz : ay - uz) : ay) : az;
        e0 = fma_(au, fma_(splat<V>(1.5), au, one), eb);
        e1 = ux * fma_(splat<V>(3.0), au, one);
        if (jy) b = jy > 0 ? b + hgy : b - hgy;
        if (jz) b = jz > 0 ? b + hgz : b - hgz;
      }
      p0 = fma_(e0, b, S);
      p1 = fma_(e0 + e2, hgx, e1 * b);
      p02 = fma_(e1, hgx, fma_(e2, b, p0));
    }
    const V A = fma_(fac[k + 1], m2, p02);
    const V B = THERMAL ? fma_(fac[k + 1], m1, p1) : fac[k + 1] * m1;
    q[3 * j] = A - B;
    q[3 * j + 1] = fma_(fac[k], m0 - m2, p0);
    q[3 * j + 2] = A + B;
  }
}

// ------------------------------------------------------------ collision of two cells, D3Q27 thermal
// The update of collide_full with central moments (axis-by-axis transform of all of them), operation by operation
// in the arithmetic of the one-cell kernel's FP32 form: same order, same products fused into an add,
// so that its results are the same bits (tests/test_gpu_pair_bits.py). Why here: a reacting flow turns rounding into differences
// of another size (a fuel fraction of order 1/2 crossing zero, a face velocity changing sign: 1e-8 in u
// becomes 1e-3 of the pressure fluctuation in 20 steps), so the arithmetic of reacting 3-D runs does not
// change with the kernel that carries it.
// ptxas fuses a packed product into the packed add that uses it, whatever the rounding modifiers and
// -fmad say; mul_rn keeps a product's own rounding where it feeds an add: a fused multiply-add with a
// -0 that ptxas cannot see through (constant memory).
static __constant__ unsigned long long k_minus_zero2 = 0x8000000080000000ull;
__device__ __forceinline__ F2 mul_rn(F2 a, F2 b) {
  F2 z;
  z.v = k_minus_zero2;
  return fma_(a, b, z);
}

// One line of central moments about u (nu = -u, n2u = -2 u, uu = u u), forwards.
__device__ __forceinline__ void line_fwd(F2& a, F2& b, F2& c, const F2 nu, const F2 n2u, const F2 uu) {
  const F2 m0 = (a + b) + c, d = c - a, s = c + a;
  a = m0;
  b = fma_(nu, m0, d);
  c = fma_(uu, m0, fma_(n2u, d, s));
}
// Back (u2 = 2 u), with the outer two values left at twice their size (exact; the final scale makes up
// for it). RN: where the one-cell form rounds 2 u m1 by itself.
template <bool RN>
__device__ __forceinline__ void line_bwd(F2& a, F2& b, F2& c, const F2 u, const F2 u2, const F2 uu) {
  const F2 m0 = a, m1 = b, m2 = c;
  const F2 k1 = fma_(u, m0, m1);
  const F2 k2 = fma_(uu, m0, RN ? m2 + mul_rn(u2, m1) : fma_(u2, m1, m2));
  a = k2 - k1;
  b = m0 - k2;
  c = k2 + k1;
}

// Moments of order (A, B, C) of h_eq - w about u, to be subtracted: the seven terms of delta_eq.
// e1, e2: -u_a and u_a u_a per axis.
template <int J>
__device__ __forceinline__ F2 delta_sum(const F2* e1, const F2* e2) {
  constexpr int A = J % 3, B = J / 3 % 3, C = J / 9;
  const F2 k3 = splat<F2>((double)(1.0f / 3.0f));
  const F2 ex = A == 2 ? e2[0] : e1[0], ey = B == 2 ? e2[1] : e1[1], ez = C == 2 ? e2[2] : e1[2];
  if constexpr (J == 8) return (mul_rn(ex, k3) + mul_rn(ey, k3)) + mul_rn(ex, ey);
  F2 acc = splat<F2>(0.0);
  bool any = false;
  auto add = [&](F2 p, F2 r) {
    acc = any ? fma_(p, r, acc) : p * r;
    any = true;
  };
  if constexpr (A > 0 && B != 1 && C != 1) {
    if constexpr (B == 2 && C == 2) add(ex * k3, k3);
    else add(ex, k3);  // one of B, C is 2 in every order that comes here
  }
  if constexpr (B > 0 && A != 1 && C != 1) {
    if constexpr (A == 2 && C == 2) add(ey * k3, k3);
    else add(ey, k3);
  }
  if constexpr (C > 0 && A != 1 && B != 1) {
    if constexpr (A == 2 && B == 2) add(ez, splat<F2>((double)((1.0f / 3.0f) * (1.0f / 3.0f))));
    else add(ez, k3);
  }
  if constexpr (A > 0 && B > 0 && C != 1) {
    if constexpr (C == 2) add(ex * ey, k3);
    else add(ex, ey);
  }
  if constexpr (A > 0 && C > 0 && B != 1) {
    if constexpr (B == 2) add(ex * k3, ez);
    else add(ex, ez);
  }
  if constexpr (B > 0 && C > 0 && A != 1) {
    if constexpr (A == 2) add(ey * k3, ez);
    else add(ey, ez);
  }
  if constexpr (A > 0 && B > 0 && C > 0) add(ex * ey, ez);
  return acc;
}

__device__ __forceinline__ void collide_central(F2* q, LBCell<3, F2, true>& c, const F2 nu3, const LBArgs<float>& a) {
  typedef F2 V;
  const V one = splat<V>(1.0), two = splat<V>(2.0), half = splat<V>(0.5), zero = splat<V>(0.0);
  const V third = splat<V>((double)(1.0f / 3.0f)), ninth = splat<V>((double)(1.0f / 9.0f));
  // weights by number of nonzero components of c_i
  constexpr float W4[4] = {(float)wgt<3>(13), (float)wgt<3>(12), (float)wgt<3>(9), (float)wgt<3>(0)};
  // their reciprocals times 1 / 2 per nonzero component (see line_bwd)
  constexpr float F4[4] = {(float)(1.0 / wgt<3>(13)), 0.5f * (float)(1.0 / wgt<3>(12)),
                           0.25f * (float)(1.0 / wgt<3>(9)), 0.125f * (float)(1.0 / wgt<3>(0))};
  // ---- moments (Eq. 7)
  V psum = zero, mx = zero, my = zero, mz = zero;
#pragma unroll
  for (int i = 0; i < 27; ++i) {
    const double w = (double)(float)wgt<3>(i);
    psum = fma_(splat<V>(w), q[i], psum);
    if (cx(i)) mx = fma_(splat<V>(cx(i) * w), q[i], mx);
    if (cy(i)) my = fma_(splat<V>(cy(i) * w), q[i], my);
    if (cz(i)) mz = fma_(splat<V>(cz(i) * w), q[i], mz);
  }
  const V rho = c.rho, gx = c.gx, gy = c.gy, gz = c.gz, three = splat<V>(3.0);
  const V inv_rho = rcp_(rho);
  const V ux = mul_rn(three * mx, inv_rho), uy = mul_rn(three * my, inv_rho), uz = mul_rn(three * mz, inv_rho);
  const V uxx = mul_rn(ux, ux), uyy = mul_rn(uy, uy), uzz = mul_rn(uz, uz);
  const V usq = (uxx + uyy) + uzz;
  const V udg = fma_(uz, gz, fma_(uy, gy, ux * gx));
  const V rl3 = mul_rn(rho * c.lam, third);  // rho cs2 Lambda
  const V k0 = fma_(third, udg, rl3);
  const V S = fma_(half, k0, psum);
  c.u[0] = ux;
  c.u[1] = uy;
  c.u[2] = uz;
  c.usq = usq;
  c.psum = psum;
  c.rl3 = rl3;
  const V tau0 = fma_(nu3, inv_rho, half);
  // ---- central moments of w d about u
  const V nux = zero - ux, nuy = zero - uy, nuz = zero - uz;
  {
    const V t3 = three * inv_rho, n2ux = two * nux;
    V tw[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) tw[k] = t3 * splat<V>(W4[k]);
#pragma unroll
    for (int j = 0; j < 9; ++j) {
      const int k = (j % 3 != 1) + (j / 3 != 1);
      const V xa = q[3 * j] - S, xb = q[3 * j + 1] - S, xc = q[3 * j + 2] - S;
      const V A = tw[k + 1] * xa;
      const V m0 = fma_(tw[k + 1], xc, fma_(tw[k], xb, A));
      const V d = fma_(tw[k + 1], xc, zero - A), s = fma_(tw[k + 1], xc, A);
      q[3 * j] = m0;
      q[3 * j + 1] = fma_(nux, m0, d);
      q[3 * j + 2] = fma_(uxx, m0, fma_(n2ux, d, s));
    }
    const V n2uy = two * nuy, n2uz = two * nuz;
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
      for (int x = 0; x < 3; ++x) line_fwd(q[x + 9 * k], q[x + 3 + 9 * k], q[x + 6 + 9 * k], nuy, n2uy, uyy);
#pragma unroll
    for (int j = 0; j < 9; ++j) line_fwd(q[j], q[j + 9], q[j + 18], nuz, n2uz, uzz);
  }
  // ---- half source (pre-conditioning) in moments of order 0..2
  const V uxy = mul_rn(ux, uy), uxz = mul_rn(ux, uz), uyz = mul_rn(uy, uz);
  {
    const V h = splat<V>(1.5) * inv_rho;
    const V u3[3] = {ux, uy, uz}, n3[3] = {nux, nuy, nuz}, g3[3] = {gx, gy, gz}, uu[3] = {uxx, uyy, uzz};
    q[0] = fma_(h, k0, q[0]);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const int ja = i == 0 ? 1 : (i == 1 ? 3 : 9);
      q[ja] = fma_(h, n3[i] * k0, q[ja]);
      const V X = uu[i] + third, Z = fma_(two * g3[i], u3[i], udg);
      q[2 * ja] = fma_(h, fma_(rl3, X, ninth * Z), q[2 * ja]);
#pragma unroll
      for (int b = i + 1; b < 3; ++b) {
        const int jb = b == 1 ? 3 : 9;
        const V Y = fma_(g3[i], u3[b], g3[b] * u3[i]);
        q[ja + jb] = fma_(h, fma_(rl3 * u3[i], u3[b], ninth * Y), q[ja + jb]);
      }
    }
  }
  // deviation from the equilibrium, order 2
  q[2] = q[2] + uxx;
  q[6] = q[6] + uyy;
  q[18] = q[18] + uzz;
  q[4] = q[4] + uxy;
  q[10] = q[10] + uxz;
  q[12] = q[12] + uyz;
  const V sum = (q[2] + q[6]) + q[18];
  const V tr = mul_rn(third, sum);
  // ---- relaxation time (Eq. 12, Smagorinsky)
  V tau = tau0;
  if (a.smag_k > 0.0f) {
    const V nt = zero - third;
    const V e0 = fma_(nt, sum, q[2]), e1 = fma_(nt, sum, q[6]), e2 = fma_(nt, sum, q[18]);
    const V o2 = fma_(q[12], q[12], fma_(q[4], q[4], q[10] * q[10]));
    const V n2 = fma_(two, o2, fma_(e2, e2, fma_(e0, e0, e1 * e1)));
    tau = smag_tau(tau0, n2, splat<V>(a.smag_k));
  }
  const V o1 = one - rcp_(tau), ob = splat<V>(1.0f - a.omega_b);
  // ---- relaxed second-order moments and the higher ones without cumulants
  const V sxx = fma_(ob, tr, mul_rn(o1, q[2] - tr)), syy = fma_(ob, tr, mul_rn(o1, q[6] - tr));
  const V szz = fma_(ob, tr, mul_rn(o1, q[18] - tr));
  const V sxy = mul_rn(o1, q[4]), sxz = mul_rn(o1, q[10]), syz = mul_rn(o1, q[12]);
  const V tx = third + sxx, ty = third + syy, tz = third + szz;
  const V s2xy = two * sxy, s2xz = two * sxz, sxxyy = mul_rn(sxx, syy);
  const V e1[3] = {nux, nuy, nuz}, e2[3] = {uxx, uyy, uzz};
  V Dd = fma_(ninth, (sxx + syy) + szz, third * fma_(szz, sxx, fma_(syy, szz, sxxyy)));
  Dd = fma_(sxxyy, szz, Dd);
  Dd = fma_(two, fma_(tz * sxy, sxy, fma_(tx * syz, syz, (ty * sxz) * sxz)), Dd);
  Dd = fma_((splat<V>(8.0) * sxy) * sxz, syz, Dd);
  q[26] = Dd - delta_sum<26>(e1, e2);
  q[2] = sxx - uxx;
  q[6] = syy - uyy;
  q[18] = szz - uzz;
  q[4] = sxy - uxy;
  q[10] = sxz - uxz;
  q[12] = syz - uyz;
  q[5] = zero - delta_sum<5>(e1, e2);
  q[7] = zero - delta_sum<7>(e1, e2);
  q[11] = zero - delta_sum<11>(e1, e2);
  q[13] = zero - delta_sum<13>(e1, e2);
  q[15] = zero - delta_sum<15>(e1, e2);
  q[19] = zero - delta_sum<19>(e1, e2);
  q[21] = zero - delta_sum<21>(e1, e2);
  q[14] = fma_(s2xy, sxz, tx * syz) - delta_sum<14>(e1, e2);
  q[16] = fma_(s2xy, syz, ty * sxz) - delta_sum<16>(e1, e2);
  q[22] = fma_(s2xz, syz, tz * sxy) - delta_sum<22>(e1, e2);
  q[8] = fma_(s2xy, sxy, mul_rn(third, sxx + syy) + sxxyy) - delta_sum<8>(e1, e2);
  q[20] = fma_(s2xz, sxz, fma_(sxx, szz, third * (sxx + szz))) - delta_sum<20>(e1, e2);
  q[24] = fma_(two * syz, syz, fma_(syy, szz, third * (syy + szz))) - delta_sum<24>(e1, e2);
  q[17] = zero - delta_sum<17>(e1, e2);
  q[23] = zero - delta_sum<23>(e1, e2);
  q[25] = zero - delta_sum<25>(e1, e2);
  // ---- back to populations
  {
    const V u2x = two * ux, u2y = two * uy, u2z = two * uz;
#pragma unroll
    for (int j = 0; j < 9; ++j) line_bwd<false>(q[j], q[j + 9], q[j + 18], uz, u2z, uzz);
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
      for (int x = 0; x < 3; ++x) {
        if (k == 1) line_bwd<false>(q[x + 9 * k], q[x + 3 + 9 * k], q[x + 6 + 9 * k], uy, u2y, uyy);
        else line_bwd<true>(q[x + 9 * k], q[x + 3 + 9 * k], q[x + 6 + 9 * k], uy, u2y, uyy);
      }
#pragma unroll
    for (int j = 0; j < 9; ++j) {
      if (j % 3 == 1) line_bwd<false>(q[3 * j], q[3 * j + 1], q[3 * j + 2], ux, u2x, uxx);
      else line_bwd<true>(q[3 * j], q[3 * j + 1], q[3 * j + 2], ux, u2x, uxx);
    }
  }
  // ---- post-collision (Eq. 8): scale, S and the half source
  V fac[4];
  {
    const V rho3 = rho * third;
#pragma unroll
    for (int k = 0; k < 4; ++k) fac[k] = rho3 * splat<V>(F4[k]);
  }
  const V hu = splat<V>(-0.5) * usq, ngx = zero - gx, ngy = zero - gy, ngz = zero - gz;
  auto out = [&](int i, int k, V t, V cu, V cg) {
    const V e = k ? fma_(t, cu, cu) + hu : hu;
    const V E = fma_(e, cg - udg, rl3);
    q[i] = fma_(half, E, fma_(fac[k], q[i], S));
  };
  out(13, 0, zero, zero, zero);
#pragma unroll
  for (int i = 0; i < 13; ++i) {
    // direction i and its opposite, which share the product 1.5 c.u
    const int k = (cx(i) != 0) + (cy(i) != 0) + (cz(i) != 0);
    V cu = zero, cg = zero, nu_ = zero, ng = zero;
    bool any = false;
    auto add = [&](int s, V u, V nu, V g, V n) {
      const V pu = s > 0 ? u : nu, mu = s > 0 ? nu : u, pg = s > 0 ? g : n, mg = s > 0 ? n : g;
      cu = any ? cu + pu : pu;
      nu_ = any ? nu_ + mu : mu;
      cg = any ? cg + pg : pg;
      ng = any ? ng + mg : mg;
      any = true;
    };
    if (cx(i)) add(cx(i), ux, nux, gx, ngx);
    if (cy(i)) add(cy(i), uy, nuy, gy, ngy);
    if (cz(i)) add(cz(i), uz, nuz, gz, ngz);
    const V t = splat<V>(1.5) * cu;
    out(i, k, t, cu, cg);
    const V e = fma_(t, cu, nu_) + hu;
    q[26 - i] = fma_(half, fma_(e, ng - udg, rl3), fma_(fac[k], q[26 - i], S));
  }
}


// ------------------------------------------------------------------ pull streaming of one cell
// raw[i] = stored q_i = g_i / w_i - P_ref from r - c_i, or the opposite population of the cell itself
// on bounce-back links; rho_p, rho_m: density at r + e_a, r - e_a (the cell's own where the link there
// is not a plain pull). Offsets fit in 32 bits (checked at init). Per-axis offsets to the minus /
// plus neighbour wrap on periodic faces (a plain pull across a non-periodic face never happens: those
// links are bounce-back, inlet or outlet links). All loads are issued before any is converted.
template <int D, typename S, typename R, bool THERMAL>
__device__ __forceinline__ void pull_cell(const LBArgs<R>& a, int r, int x, int y, int z, uint32_t lw, S* raw,
                                          R* rho_p, R* rho_m) {
  constexpr int Q = Lat<D>::Q;
  const int nx = a.geo.nx, ny = a.geo.ny, nz = a.geo.nz, Ni = a.geo.N;
  const S* __restrict__ gin = (const S*)a.g_in;
  const int sy_ = nx, sz_ = nx * ny;
  const int oxm = x > 0 ? -1 : nx - 1, oxp = x < nx - 1 ? 1 : 1 - nx;
  const int oym = y > 0 ? -sy_ : (ny - 1) * sy_, oyp = y < ny - 1 ? sy_ : (1 - ny) * sy_;
  const int ozm = z > 0 ? -sz_ : (nz - 1) * sz_, ozp = z < nz - 1 ? sz_ : (1 - nz) * sz_;
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const int ci = cx(i), cj = cy(i), ck = (D == 3) ? cz(i) : 0;
    // source r - c_i
    const int s = r + (ci == 1 ? oxm : (ci == -1 ? oxp : 0)) + (cj == 1 ? oym : (cj == -1 ? oyp : 0)) +
                  (ck == 1 ? ozm : (ck == -1 ? ozp : 0));
    const bool link = (lw >> i) & 1u;
    raw[i] = ld_raw<S>(gin + (link ? (Q - 1 - i) * Ni + r : i * Ni + s));
    if constexpr (THERMAL) {
      if (ci * ci + cj * cj + ck * ck == 1 && !link) {
        // direction -e_a pulls from r + e_a; +e_a pulls from r - e_a
        const R rs = ldg(a.rho + s);
        if (ci == -1) rho_p[0] = rs;
        if (ci == 1) rho_m[0] = rs;
        if (cj == -1) rho_p[1] = rs;
        if (cj == 1) rho_m[1] = rs;
        if (D == 3 && ck == -1) rho_p[2] = rs;
        if (D == 3 && ck == 1) rho_m[2] = rs;
      }
    }
  }
}

// Inlet and outlet rules of one cell on its pulled populations q.
template <int D, typename R>
__device__ __forceinline__ void face_rules(const LBArgs<R>& a, int r, int x, int y, int z, uint32_t lw, R rho, R* q) {
  constexpr int Q = Lat<D>::Q;
  const int nx = a.geo.nx, ny = a.geo.ny, nz = a.geo.nz;
  // moving-wall term of the low-x inlet: g_i += 2 w_i rho (c_i . u_w)
  if (x == 0 && a.geo.bc_lo[0] == BC_INLET) {
    const int f = y + ny * z;
    const int nf = ny * nz;
    const R uw0 = ldg(a.inlet_u + f), uw1 = ldg(a.inlet_u + nf + f);
    const R uw2 = (D == 3) ? ldg(a.inlet_u + 2 * nf + f) : R(0);
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      if (cx(i) == 1) {
        if ((lw >> i) & 1u) {
          const R cu = uw0 + (R)cy(i) * uw1 + ((D == 3) ? (R)cz(i) * uw2 : R(0));
          q[i] += R(2) * rho * cu;
        }
      }
    }
  }
  // pressure outlet (anti-bounce-back at the half-way face, P_h = P_ref):
  // g_i = -g*_opp + 2 w_i (P_ref + rho (1.5 (c_i.u)^2 - 0.5 u^2)), u of the previous step
  if (x == nx - 1 && a.geo.bc_hi[0] == BC_OUTLET) {
    const size_t N = (size_t)a.geo.N;
    const R vx = a.u_in[r], vy = a.u_in[N + r], vz = (D == 3) ? a.u_in[2 * N + r] : R(0);
    const R vv = vx * vx + vy * vy + vz * vz;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      if (cx(i) == -1) {
        if ((lw >> i) & 1u) {
          const R cu = -vx + (R)cy(i) * vy + ((D == 3) ? (R)cz(i) * vz : R(0));
          q[i] = -q[i] + rho * (R(3) * cu * cu - vv);
        }
      }
    }
  }
}

// Update of the cell r = (x, y, z) by one thread.
// WALLS = false: a fluid cell, unless flagged LINK_WALL.
// WALLS = true: a flagged cell, row wrow of the wall table, with the interpolated bounce-back fix-up compiled
// in (so that it costs the other cells no registers). The arguments come by value, as a kernel's do: by
// reference nvcc fused other products of the inlet and outlet rules (a last place in a few cells).
template <int D, typename S, typename R, bool THERMAL, int COLL, bool WALLS>
__device__ __forceinline__ void lb_cell(const LBArgs<R> a, const int x, const int y, const int z, const int r,
                                        const int wrow) {
  constexpr int Q = Lat<D>::Q;
  const int nx = a.geo.nx, ny = a.geo.ny, nz = a.geo.nz;
  // the cell's rho, Lambda and T are loaded together with its link word (every cell has them)
  R rho = R(1), lam = R(0), T_early = R(0);
  if constexpr (THERMAL) {
    rho = ldg(a.rho + r);
    lam = ldg(a.lam + r);
    T_early = ldg(a.T + r);
  }
  const uint32_t lw = __ldg(a.links + r);
  if (!(lw >> 31)) return;
  if (!WALLS && (lw & LINK_WALL)) return;  // done by the blocks of the wall list
  const size_t N = (size_t)a.geo.N;
  const S* __restrict__ gin = (const S*)a.g_in;
  const R third = R(1) / R(3);
  R rho_p[3] = {rho, rho, rho}, rho_m[3] = {rho, rho, rho};  // rho at r + e_a, r - e_a

  // ---------------------------------------------------------------- pull streaming
  // q_i = g_i / w_i - P_ref (the stored shifted form). Offsets fit in 32 bits (checked at init).
  // Per-axis offsets to the minus / plus neighbour, wrapped on periodic faces (a plain pull across
  // a non-periodic face never happens: those links are bounce-back, inlet or outlet links).
  // phase 1 issues every load into raw[] (storage type), phase 2 converts: all loads of a cell
  // are in flight together whatever the storage type
  S raw[Q];
  const int sy_ = nx, sz_ = nx * ny;
  const int Ni = a.geo.N;
  const int oxm = x > 0 ? -1 : nx - 1, oxp = x < nx - 1 ? 1 : 1 - nx;
  const int oym = y > 0 ? -sy_ : (ny - 1) * sy_, oyp = y < ny - 1 ? sy_ : (1 - ny) * sy_;
  const int ozm = z > 0 ? -sz_ : (nz - 1) * sz_, ozp = z < nz - 1 ? sz_ : (1 - nz) * sz_;
  const bool outlet_cell = x == nx - 1 && a.geo.bc_hi[0] == BC_OUTLET;
  // interior warp: no lane has a bounce-back, inlet or outlet link or sits on a periodic face, so
  // every pull is a plain offset (same loads as below, without the per-direction link tests)
  const bool interior = !WALLS && (lw & ((1u << Q) - 1u)) == 0u && x > 0 && x < nx - 1 && y > 0 &&
                        y < ny - 1 && (D == 2 || (z > 0 && z < nz - 1));
  if (!WALLS && __all_sync(__activemask(), interior)) {
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      const int ci = cx(i), cj = cy(i), ck = (D == 3) ? cz(i) : 0;
      raw[i] = ld_raw<S>(gin + i * Ni + r - ci - cj * sy_ - ck * sz_);
    }
    if constexpr (THERMAL) {
      rho_p[0] = ldg(a.rho + r + 1);
      rho_m[0] = ldg(a.rho + r - 1);
      rho_p[1] = ldg(a.rho + r + sy_);
      rho_m[1] = ldg(a.rho + r - sy_);
      if (D == 3) {
        rho_p[2] = ldg(a.rho + r + sz_);
        rho_m[2] = ldg(a.rho + r - sz_);
      }
    }
  } else {
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const int ci = cx(i), cj = cy(i), ck = (D == 3) ? cz(i) : 0;
    if ((lw >> i) & 1u) {
      raw[i] = ld_raw<S>(gin + (Q - 1 - i) * Ni + r);
    } else {
      // source r - c_i
      const int s = r + (ci == 1 ? oxm : (ci == -1 ? oxp : 0)) + (cj == 1 ? oym : (cj == -1 ? oyp : 0)) +
                    (ck == 1 ? ozm : (ck == -1 ? ozp : 0));
      raw[i] = ld_raw<S>(gin + i * Ni + s);
      if constexpr (THERMAL) {
        if (ci * ci + cj * cj + ck * ck == 1) {
          // direction -e_a pulls from r + e_a; +e_a pulls from r - e_a
          const R rs = ldg(a.rho + s);
          if (ci == -1) rho_p[0] = rs;
          if (ci == 1) rho_m[0] = rs;
          if (cj == -1) rho_p[1] = rs;
          if (cj == 1) rho_m[1] = rs;
          if (D == 3 && ck == -1) rho_p[2] = rs;
          if (D == 3 && ck == 1) rho_m[2] = rs;
        }
      }
    }
  }
  }
  // the thermodynamic-pressure state of this step: after the kernel that updates it (launched just
  // before this one; the loads above read only what earlier kernels wrote)
  pdl_wait();
  if constexpr (THERMAL) {
    if constexpr (sizeof(R) == 8) lam += (R)a.pth->lb_lam_d;
    else lam += (R)a.pth->lb_lam;
  }
  R q[Q];
#pragma unroll
  for (int i = 0; i < Q; ++i) q[i] = cvt_pop<S, R>(raw[i]);
  // interpolated bounce-back (curved or offset walls) on flagged cells: for a link whose wall
  // lies at the fraction f of r -> r - c_i, with o the opposite direction and q_i = g*_o(r) above,
  //   f <  1/2:  g_i = 2 f g*_o(r) + (1 - 2 f) g*_o(r + c_i) = g*_o(r + c_i) + 2 f (g*_o(r) - g*_o(r + c_i))
  //   f >= 1/2:  g_i = g*_o(r) / (2 f) + (2 f - 1) / (2 f) g*_i(r) = g*_i(r) + (g*_o(r) - g*_i(r)) / (2 f)
  // (affine with weights summing to 1, so it holds for the shifted stored form as well; the
  // right-hand forms round once, on a difference of neighbouring populations)
  if constexpr (WALLS) {
    const R* __restrict__ wq = a.wall_q + (size_t)wrow * Q;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      if ((lw >> i) & 1u) {
        const R f = wq[i];
        if (f != R(0.5)) {
          const int ci = cx(i), cj = cy(i), ck = (D == 3) ? cz(i) : 0;
          if (f < R(0.5)) {
            // r + c_i: the pull source of the opposite direction (a fluid node, checked at set-up)
            const int s = r + (ci == -1 ? oxm : (ci == 1 ? oxp : 0)) + (cj == -1 ? oym : (cj == 1 ? oyp : 0)) +
                          (ck == -1 ? ozm : (ck == 1 ? ozp : 0));
            const R far_o = cvt_pop<S, R>(ld_raw<S>(gin + (Q - 1 - i) * Ni + s));
            q[i] = far_o + R(2) * f * (q[i] - far_o);  // one rounding on a small difference
          } else {
            const R own_i = cvt_pop<S, R>(ld_raw<S>(gin + i * Ni + r));
            q[i] = own_i + (q[i] - own_i) / (R(2) * f);
          }
        }
      }
    }
  }
  // moving-wall term of the low-x inlet: g_i += 2 w_i rho (c_i . u_w)
  if (x == 0 && a.geo.bc_lo[0] == BC_INLET) {
    const int f = y + ny * z;
    const int nf = ny * nz;
    const R uw0 = ldg(a.inlet_u + f), uw1 = ldg(a.inlet_u + nf + f);
    const R uw2 = (D == 3) ? ldg(a.inlet_u + 2 * nf + f) : R(0);
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      if (cx(i) == 1) {
        if ((lw >> i) & 1u) {
          const R cu = uw0 + (R)cy(i) * uw1 + ((D == 3) ? (R)cz(i) * uw2 : R(0));
          q[i] += R(2) * rho * cu;
        }
      }
    }
  }
  // pressure outlet (anti-bounce-back at the half-way face, P_h = P_ref):
  // g_i = -g*_opp + 2 w_i (P_ref + rho (1.5 (c_i.u)^2 - 0.5 u^2)), u of the previous step
  if (outlet_cell) {
    const R vx = a.u_in[r], vy = a.u_in[N + r], vz = (D == 3) ? a.u_in[2 * N + r] : R(0);
    const R vv = vx * vx + vy * vy + vz * vz;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      if (cx(i) == -1) {
        if ((lw >> i) & 1u) {
          const R cu = -vx + (R)cy(i) * vy + ((D == 3) ? (R)cz(i) * vz : R(0));
          q[i] = -q[i] + rho * (R(3) * cu * cu - vv);
        }
      }
    }
  }

  if constexpr (COLL == COLL_CUMULANT_FULL && sizeof(R) == 8) {
    LBCell<D, R, THERMAL> c;
    c.rho = rho;
    c.lam = lam;
    if constexpr (THERMAL) {
      c.gx = R(0.5) * (rho_p[0] - rho_m[0]);
      c.gy = R(0.5) * (rho_p[1] - rho_m[1]);
      c.gz = (D == 3) ? R(0.5) * (rho_p[2] - rho_m[2]) : R(0);
    }
    collide_full<D, R, THERMAL, R>(q, c, R(3) * a.nu_lat * (THERMAL ? pw<R>(T_early * a.T_ref_inv, a.mu_exp) : R(1)), a);
    S* __restrict__ gout = (S*)a.g_out;
#pragma unroll
    for (int i = 0; i < Q; ++i) st_pop<S, R>(gout + i * Ni + r, q[i]);
    if (a.write_u || outlet_cell) {
      a.u[r] = c.u[0];
      a.u[N + r] = c.u[1];
      if (D == 3) a.u[2 * N + r] = c.u[2];
    }
    if (a.ph_out) a.ph_out[r] = a.P_ref + c.psum + R(0.5) * c.rl3;
    if (!isfinite(c.usq)) atomicOr(a.flag, 1);
    return;
  }

  // ---------------------------------------------------------------- moments (Eq. 7)
  R psum = R(0), mx = R(0), my = R(0), mz = R(0);
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const R wq = (R)wgt<D>(i) * q[i];
    psum += wq;
    if (cx(i) == 1) mx += wq;
    if (cx(i) == -1) mx -= wq;
    if (cy(i) == 1) my += wq;
    if (cy(i) == -1) my -= wq;
    if (D == 3) {
      if (cz(i) == 1) mz += wq;
      if (cz(i) == -1) mz -= wq;
    }
  }
  const R inv_rho = R(1) / rho;
  const R ux = R(3) * mx * inv_rho, uy = R(3) * my * inv_rho, uz = (D == 3) ? R(3) * mz * inv_rho : R(0);
  const R usq = ux * ux + uy * uy + uz * uz;
  R gx = R(0), gy = R(0), gz = R(0), udg = R(0);
  if constexpr (THERMAL) {
    gx = R(0.5) * (rho_p[0] - rho_m[0]);
    gy = R(0.5) * (rho_p[1] - rho_m[1]);
    if (D == 3) gz = R(0.5) * (rho_p[2] - rho_m[2]);
    udg = ux * gx + uy * gy + uz * gz;
  }
  const R rl3 = rho * lam * third;  // rho cs2 Lambda

  // ------------------------------ source xi_i = Xi_i / w_i (Eq. 2) and pre-conditioning (Eq. 13)
  // s_i = q_i + xi_i / 2, S = sum w s; d_i = h_i / w_i - 1 = 3 (s_i - S) / rho.
  // With full relaxation of orders 3..6 the collision reads the source only through the central
  // moments of w xi of orders 0..2 (the higher ones are overwritten), which have closed forms on
  // the product-weight lattices: with L = rho cs2 Lambda and G = u . grad rho,
  //   k_0 = L + G/3, k_a = -u_a k_0, k_aa = L u_a^2 + L/3 + (G + 2 g_a u_a)/9,
  //   k_ab = L u_a u_b + (g_a u_b + g_b u_a)/9 (a != b);
  // they are added to the moments after the forward transform (SRC_MOM); otherwise the source is
  // added per direction here.
  constexpr bool SRC_MOM = THERMAL && COLL == COLL_CUMULANT_FULL;
  R Ssum = R(0);
  R k0 = R(0);
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    if constexpr (THERMAL && !SRC_MOM) {
      const R cu = (R)cx(i) * ux + (R)cy(i) * uy + ((D == 3) ? (R)cz(i) * uz : R(0));
      const R cg = (R)cx(i) * gx + (R)cy(i) * gy + ((D == 3) ? (R)cz(i) * gz : R(0));
      const R e = cu + R(1.5) * cu * cu - R(0.5) * usq;  // (f^eq/rho - w)/w * cs2
      q[i] += R(0.5) * (e * (cg - udg) + rl3);
    }
    Ssum += (R)wgt<D>(i) * q[i];
  }
  if constexpr (SRC_MOM) {
    k0 = rl3 + third * udg;
    Ssum += R(0.5) * k0;
  }
  const R three_over_rho = R(3) * inv_rho;
  // d_i = h_i / w_i - 1; the cumulant path works on w_i d_i (w_i folded into the factor)
#pragma unroll
  for (int i = 0; i < Q; ++i)
    q[i] = (COLL == COLL_BGK ? three_over_rho : three_over_rho * (R)wgt<D>(i)) * (q[i] - Ssum);

  // ---------------------------------------------------------------- relaxation time
  R tau0;
  if constexpr (THERMAL) {
    const R Tr = T_early;
    tau0 = R(3) * a.nu_lat * pw<R>(Tr * a.T_ref_inv, a.mu_exp) * inv_rho + R(0.5);
  } else {
    tau0 = R(3) * a.nu_lat + R(0.5);
  }

  if constexpr (COLL != COLL_BGK) {
    constexpr bool FULL = COLL == COLL_CUMULANT_FULL;
    // central moments of w d (d = h/w - 1) about u, minus those of h_eq - w, give the central
    // moments n of h - h_eq (h_eq: product-form equilibrium); see delta_eq
    const R dlx[3] = {R(0), -ux, ux * ux}, dly[3] = {R(0), -uy, uy * uy}, dlz[3] = {R(0), -uz, uz * uz};
#pragma unroll
    for (int j = 0; j < Q / 3; ++j) chim_fwd(q[3 * j], q[3 * j + 1], q[3 * j + 2], ux);
#pragma unroll
    for (int kz = 0; kz < Q / 9; ++kz)
#pragma unroll
      for (int ax = 0; ax < 3; ++ax) chim_fwd(q[ax + 9 * kz], q[ax + 3 + 9 * kz], q[ax + 6 + 9 * kz], uy);
    if constexpr (D == 3) {
#pragma unroll
      for (int j = 0; j < 9; ++j) chim_fwd(q[j], q[j + 9], q[j + 18], uz);
    }
    if constexpr (SRC_MOM) {
      // (3 / rho) (1/2) times the moments k of w xi listed above, orders 0..2
      const R h = R(1.5) * inv_rho, ninth = R(1) / R(9);
      const R u3[3] = {ux, uy, uz}, g3[3] = {gx, gy, gz};
      q[0] += h * k0;
#pragma unroll
      for (int a = 0; a < D; ++a) {
        const int ja = a == 0 ? 1 : (a == 1 ? 3 : 9);  // index of the first-order moment along a
        q[ja] += h * (-u3[a] * k0);
        q[2 * ja] += h * (rl3 * (u3[a] * u3[a] + third) + ninth * (udg + R(2) * g3[a] * u3[a]));
#pragma unroll
        for (int b = a + 1; b < D; ++b) {
          const int jb = b == 1 ? 3 : 9;
          q[ja + jb] += h * (rl3 * u3[a] * u3[b] + ninth * (g3[a] * u3[b] + g3[b] * u3[a]));
        }
      }
    }
    // full relaxation of orders 3..6 reads only the second-order moments, and orders 0 and 1
    // pass through unchanged: there the deviation is removed and restored for order 2 and
    // restored for orders >= 2 only (the skipped terms cancel exactly in real arithmetic)
    if constexpr (FULL) add_delta_eq<D, R, 0, 2, 2>(q, dlx, dly, dlz, R(-1));
    else add_delta_eq<D, R, 0>(q, dlx, dly, dlz, R(-1));
    // Smagorinsky: deviatoric part of the second central moments (equilibrium is isotropic)
    R tau = tau0;
    if (a.smag_k > R(0)) {
      R n2;
      if constexpr (D == 2) {
        const R tr = R(0.5) * (q[2] + q[6]);
        const R d0 = q[2] - tr, d1 = q[6] - tr;
        n2 = d0 * d0 + d1 * d1 + R(2) * q[4] * q[4];
      } else {
        const R tr = third * (q[2] + q[6] + q[18]);
        const R d0 = q[2] - tr, d1 = q[6] - tr, d2 = q[18] - tr;
        n2 = d0 * d0 + d1 * d1 + d2 * d2 + R(2) * (q[4] * q[4] + q[10] * q[10] + q[12] * q[12]);
      }
      tau = R(0.5) * (tau0 + sqrt(tau0 * tau0 + a.smag_k * sqrt(n2)));
    }
    const R om = R(1) / tau;
    if constexpr (D == 2) cumulant_relax2<FULL, R>(q, om, a.omega_b, a.om3, a.om4);
    else cumulant_relax3<FULL, R>(q, om, a.omega_b, a.om3, a.om4, a.om5, a.om6);
    if constexpr (FULL) add_delta_eq<D, R, 0, 2, 6>(q, dlx, dly, dlz, R(1));
    else add_delta_eq<D, R, 0>(q, dlx, dly, dlz, R(1));
    if constexpr (D == 3) {
#pragma unroll
      for (int j = 0; j < 9; ++j) chim_bwd(q[j], q[j + 9], q[j + 18], uz);
    }
#pragma unroll
    for (int kz = 0; kz < Q / 9; ++kz)
#pragma unroll
      for (int ax = 0; ax < 3; ++ax) chim_bwd(q[ax + 9 * kz], q[ax + 3 + 9 * kz], q[ax + 6 + 9 * kz], uy);
#pragma unroll
    for (int j = 0; j < Q / 3; ++j) chim_bwd(q[3 * j], q[3 * j + 1], q[3 * j + 2], ux);
    // q now holds w_i d*_i; the 1 / w_i is folded into the store below
  } else {
    // single rate towards the polynomial equilibrium f^eq(1, u) of Eq. 4: E_i = f^eq_i / w_i - 1
    R tau = tau0;
    if (a.smag_k > R(0)) {
      R pxx = R(0), pyy = R(0), pzz = R(0), pxy = R(0), pxz = R(0), pyz = R(0);
#pragma unroll
      for (int i = 0; i < Q; ++i) {
        const R cu = (R)cx(i) * ux + (R)cy(i) * uy + ((D == 3) ? (R)cz(i) * uz : R(0));
        const R ne = (R)wgt<D>(i) * (q[i] - (R(3) * cu + R(4.5) * cu * cu - R(1.5) * usq));
        const R c0 = (R)cx(i), c1 = (R)cy(i), c2 = (D == 3) ? (R)cz(i) : R(0);
        pxx += c0 * c0 * ne; pyy += c1 * c1 * ne; pxy += c0 * c1 * ne;
        if (D == 3) { pzz += c2 * c2 * ne; pxz += c0 * c2 * ne; pyz += c1 * c2 * ne; }
      }
      R n2;
      if (D == 2) {
        const R tr = R(0.5) * (pxx + pyy);
        n2 = (pxx - tr) * (pxx - tr) + (pyy - tr) * (pyy - tr) + R(2) * pxy * pxy;
      } else {
        const R tr = third * (pxx + pyy + pzz);
        n2 = (pxx - tr) * (pxx - tr) + (pyy - tr) * (pyy - tr) + (pzz - tr) * (pzz - tr) +
             R(2) * (pxy * pxy + pxz * pxz + pyz * pyz);
      }
      tau = R(0.5) * (tau0 + sqrt(tau0 * tau0 + a.smag_k * sqrt(n2)));
    }
    const R om = R(1) / tau;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      const R cu = (R)cx(i) * ux + (R)cy(i) * uy + ((D == 3) ? (R)cz(i) * uz : R(0));
      const R E = R(3) * cu + R(4.5) * cu * cu - R(1.5) * usq;
      q[i] -= om * (q[i] - E);
    }
  }

  // ------------------------------------------------- post-collision (Eq. 8), stored shifted
  // g*_i / w_i - P_ref = rho/3 (h*_i / w_i - 1) + S + xi_i / 2
  S* __restrict__ gout = (S*)a.g_out;
  const R rho3 = rho * third;
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    R half_xi = R(0);
    if constexpr (THERMAL) {
      const R cu = (R)cx(i) * ux + (R)cy(i) * uy + ((D == 3) ? (R)cz(i) * uz : R(0));
      const R cg = (R)cx(i) * gx + (R)cy(i) * gy + ((D == 3) ? (R)cz(i) * gz : R(0));
      const R e = cu + R(1.5) * cu * cu - R(0.5) * usq;
      half_xi = R(0.5) * (e * (cg - udg) + rl3);
    }
    const R fac = COLL == COLL_BGK ? rho3 : rho3 * (R)(1.0 / wgt<D>(i));
    st_pop<S, R>(gout + i * Ni + r, fac * q[i] + Ssum + half_xi);
  }
  if (a.write_u || outlet_cell) {
    a.u[r] = ux;
    a.u[N + r] = uy;
    if (D == 3) a.u[2 * N + r] = uz;
  }
  if (a.ph_out) a.ph_out[r] = a.P_ref + psum + R(0.5) * rl3;
  if (!isfinite(usq)) atomicOr(a.flag, 1);
}

// Cell i of the wall list, one thread each.
template <int D, typename S, typename R, bool THERMAL, int COLL>
__device__ __forceinline__ void lb_wall_cell(const LBArgs<R>& a, const int i) {
  if (i >= a.n_wall) return;
  const int nx = a.geo.nx, ny = a.geo.ny, r = __ldg(a.wall_cells + i);
  lb_cell<D, S, R, THERMAL, COLL, true>(a, r % nx, (r / nx) % ny, r / (nx * ny), r, i);
}

// One thread per cell, one block row of cells along x; y and z come from the grid (no integer division).
// LIST: the first planes of blocks (wall_planes) take the wall list, the others the cells that are not on
// it. In one launch the list's few cells, a chain of latencies, run beside the others and need no wait of
// their own (see launch_lb).
template <int D, typename S, typename R, bool THERMAL, int COLL, bool LIST>
__global__ void __launch_bounds__(LB_BLOCK, LB_MIN_BLOCKS) lb_step_kernel(const LBArgs<R> a) {
  int z = blockIdx.z;
  if constexpr (LIST) {
    if (z < a.wall_planes) {
      lb_wall_cell<D, S, R, THERMAL, COLL>(
          a, (blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * z)) * blockDim.x + threadIdx.x);
      return;
    }
    z -= a.wall_planes;
  }
  const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
  if (x >= a.geo.nx) return;
  lb_cell<D, S, R, THERMAL, COLL, false>(a, x, y, z, x + a.geo.nx * (y + a.geo.ny * z), 0);
}

// ------------------------------------------------------------------ two cells per thread
// Stream-collide of FP32 arithmetic with full relaxation of the orders 3..6 (the default rates): a
// thread owns the cells r, r + 1 (r even) of the linear index and runs them through packed
// instructions (packed.cuh). The one-cell kernel waited on instruction issue (70% of the slots, 44%
// of DRAM peak); here each arithmetic instruction serves two cells, the populations of c_x = 0 and
// all stores move 64 bits (VEC), and address arithmetic is shared: 86.5 M -> 44.9 M warp
// instructions on the reactive 192x96x96 case (30.3 M with collide_full). Rows of any length fill every warp, since the threads follow the linear
// index (with one block row per grid row, 135 cells took 256 threads).
// Before -> after per launch, FP32 / FP16 populations: cold swirl 256x128x128 180 -> 138 / 175 -> 104 us
// and periodic box 161x129x97 112 -> 72 us (90% of the copy peak by its 217 B per cell; bound by DRAM
// and its latency: 35% issue); reactive swirl 384x192x192 (collide_central) 655 -> 577 / 672 -> 554 us,
// bound by the FP32 pipe (57% busy) and load latency at 14 warps per SM. L2 prefetch hints of 64 to 256
// bytes, none, and streaming stores on FP32 differ by less than 2%; loads that do not allocate in L1
// cost 14-25% (the x-shifted pulls of a pair share lines there).
// VEC: nx even and every array aligned to two elements, else each element is loaded and stored by
// itself. Cells with boundary links or on periodic faces pull one by one (pull_cell) in the warps
// that hold such cells; the others take the plain offsets. (Taking plain loads there for each
// direction without links in the warp, behind 27 uniform branches, was level in FP32 and 10% slower
// in FP16: the branches keep the loads of a cell from being in flight together. Prefetching the
// populations of a later block into L2 was 2-30% slower.)
constexpr int LP_BLOCK = 64;
// resident blocks the registers are sized for: 128 registers thermal (102 registers spill, 13% slower),
// 96 isothermal (cold swirl 256x128x128 FP16 111 -> 104 us per step against 128 registers). Blocks of 64
// against 128 threads are 1% faster.
constexpr int LP_MIN_THERMAL = 8, LP_MIN_ISOTHERMAL = 10;

template <typename S> __device__ __forceinline__ void ld_raw2(const S* p, S& a, S& b);
template <> __device__ __forceinline__ void ld_raw2<float>(const float* p, float& a, float& b) {
  asm("ld.global.nc.L2::256B.v2.f32 {%0, %1}, [%2];" : "=f"(a), "=f"(b) : "l"(p));
}
template <> __device__ __forceinline__ void ld_raw2<__half>(const __half* p, __half& a, __half& b) {
  unsigned short u, v;
  asm("ld.global.nc.L2::256B.v2.u16 {%0, %1}, [%2];" : "=h"(u), "=h"(v) : "l"(p));
  a = __ushort_as_half(u);
  b = __ushort_as_half(v);
}
__device__ __forceinline__ void st2(float* p, F2 v) { *reinterpret_cast<float2*>(p) = make_float2(lo(v), hi(v)); }
__device__ __forceinline__ void st_pop2(float* p, F2 v) { st2(p, v); }
__device__ __forceinline__ void st_pop2(__half* p, F2 v) {
  const __half2 h = __floats2half2_rn(lo(v), hi(v));
  __stcs(reinterpret_cast<unsigned int*>(p), *reinterpret_cast<const unsigned int*>(&h));
}
template <bool VEC> __device__ __forceinline__ F2 ld_pair(const float* p, bool two) {
  if constexpr (VEC) {
    const float2 v = __ldg(reinterpret_cast<const float2*>(p));
    return pack2(v.x, v.y);
  }
  return pack2(__ldg(p), __ldg(p + (two ? 1 : 0)));
}

// LIST: the first blocks (wall_planes of them) take the wall list, one cell per thread, as in lb_step_kernel.
// a.pdl: a wait that every launch executes costs the others 1% (cold swirl 256x128x128 2875 against 2844 us
// per 20 steps, vessel 135x101x77 1568 against 1560 per 10).
template <int D, typename S, bool THERMAL, bool VEC, bool LIST>
__global__ void __launch_bounds__(LP_BLOCK, THERMAL ? LP_MIN_THERMAL : LP_MIN_ISOTHERMAL) lb_pair_kernel(const LBArgs<float> a) {
  constexpr int Q = Lat<D>::Q;
  constexpr uint32_t LINKS = (1u << Q) - 1u;
  const int nx = a.geo.nx, ny = a.geo.ny, nz = a.geo.nz, N = a.geo.N;
  int block = blockIdx.x;
  if constexpr (LIST) {
    if (block < a.wall_planes) {
      lb_wall_cell<D, S, float, THERMAL, COLL_CUMULANT_FULL>(a, block * LP_BLOCK + threadIdx.x);
      return;
    }
    block -= a.wall_planes;
  }
  const int r = 2 * (block * LP_BLOCK + threadIdx.x);
  if (r >= N) return;
  const bool two = VEC || r + 1 < N;  // the last cell of an odd grid has no partner
  F2 rho = splat<F2>(1.0), lam = splat<F2>(0.0), T = splat<F2>(1.0);
  if constexpr (THERMAL) {
    rho = ld_pair<VEC>(a.rho + r, two);
    lam = ld_pair<VEC>(a.lam + r, two);
    T = ld_pair<VEC>(a.T + r, two);
  }
  const uint32_t lw0 = __ldg(a.links + r), lw1 = two ? __ldg(a.links + r + 1) : 0u;
  // cells this launch updates: fluid ones, except those of the interpolated-wall list
  const bool act0 = (lw0 >> 30) == 2u, act1 = (lw1 >> 30) == 2u;
  if (!act0 && !act1) {
    // an exit without it makes the thermal kernel slower (swirl 384x192x192: 575 us, so 563)
    if (THERMAL && a.pdl) pdl_wait();
    return;
  }
  const int row = a.div_nx.div(r), z0 = D == 3 ? a.div_ny.div(row) : 0;
  const int x0 = r - row * nx, y0 = D == 3 ? row - z0 * ny : row;
  const bool plain = act0 && act1 && ((lw0 | lw1) & LINKS) == 0u && x0 > 0 && x0 + 2 < nx && y0 > 0 && y0 < ny - 1 &&
                     (D == 2 || (z0 > 0 && z0 < nz - 1));
  S raw0[Q], raw1[Q];
  F2 gx = splat<F2>(0.0), gy = gx, gz = gx;
  F2 q[Q];
  bool out0 = false, out1 = false;  // outlet cells
  if (__all_sync(__activemask(), plain)) {
    const S* __restrict__ gin = (const S*)a.g_in;
    const int sy_ = nx, sz_ = nx * ny;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      const int ci = cx(i), cj = cy(i), ck = (D == 3) ? cz(i) : 0;
      const S* p = gin + (size_t)i * N + (unsigned)(r - cj * sy_ - ck * sz_) - ci;
      if (VEC && ci == 0) {
        ld_raw2<S>(p, raw0[i], raw1[i]);
      } else {
        raw0[i] = ld_raw<S>(p);
        raw1[i] = ld_raw<S>(p + 1);
      }
    }
    if constexpr (THERMAL) {
      const float left = ldg(a.rho + r - 1), right = ldg(a.rho + r + 2);
      const F2 yp = ld_pair<VEC>(a.rho + r + sy_, true), ym = ld_pair<VEC>(a.rho + r - sy_, true);
      gx = splat<F2>(0.5) * (pack2(hi(rho), right) - pack2(left, lo(rho)));
      gy = splat<F2>(0.5) * (yp - ym);
      if constexpr (D == 3) {
        const F2 zp = ld_pair<VEC>(a.rho + r + sz_, true), zm = ld_pair<VEC>(a.rho + r - sz_, true);
        gz = splat<F2>(0.5) * (zp - zm);
      }
    }
    if (THERMAL && a.pdl) pdl_wait();
#pragma unroll
    for (int i = 0; i < Q; ++i) q[i] = pack2(cvt_pop<S, float>(raw0[i]), cvt_pop<S, float>(raw1[i]));
  } else {
    // cells on walls, inlets, outlets, next to solids or on periodic faces are in this warp
    const bool wrap = x0 + 1 == nx;
    const int x1 = wrap ? 0 : x0 + 1, y1 = wrap ? (y0 + 1 == ny && D == 3 ? 0 : y0 + 1) : y0;
    const int z1 = (D == 3 && wrap && y0 + 1 == ny) ? z0 + 1 : z0, r1 = two ? r + 1 : r;
    float rp[3], rm[3], sp[3], sm[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      rp[d] = rm[d] = lo(rho);
      sp[d] = sm[d] = hi(rho);
    }
    // a cell that is not updated reads its own populations
    pull_cell<D, S, float, THERMAL>(a, r, x0, y0, z0, act0 ? lw0 : LINKS, raw0, rp, rm);
    pull_cell<D, S, float, THERMAL>(a, r1, x1, y1, z1, act1 ? lw1 : LINKS, raw1, sp, sm);
    if constexpr (THERMAL) {
      gx = splat<F2>(0.5) * (pack2(rp[0], sp[0]) - pack2(rm[0], sm[0]));
      gy = splat<F2>(0.5) * (pack2(rp[1], sp[1]) - pack2(rm[1], sm[1]));
      if constexpr (D == 3) gz = splat<F2>(0.5) * (pack2(rp[2], sp[2]) - pack2(rm[2], sm[2]));
    }
    if (THERMAL && a.pdl) pdl_wait();
    float p0[Q], p1[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      p0[i] = cvt_pop<S, float>(raw0[i]);
      p1[i] = cvt_pop<S, float>(raw1[i]);
    }
    if (act0) face_rules<D, float>(a, r, x0, y0, z0, lw0, lo(rho), p0);
    if (act1) face_rules<D, float>(a, r1, x1, y1, z1, lw1, hi(rho), p1);
    out0 = x0 == nx - 1 && a.geo.bc_hi[0] == BC_OUTLET;
    out1 = x1 == nx - 1 && a.geo.bc_hi[0] == BC_OUTLET;
#pragma unroll
    for (int i = 0; i < Q; ++i) q[i] = pack2(p0[i], p1[i]);
  }
  LBCell<D, F2, THERMAL> c;
  c.rho = rho;
  c.lam = lam;
  F2 nu3 = splat<F2>(3.0f * a.nu_lat);
  if constexpr (THERMAL) {
    c.lam = lam + splat<F2>(a.pth->lb_lam);
    c.gx = gx;
    c.gy = gy;
    c.gz = gz;
    const F2 t = T * splat<F2>(a.T_ref_inv);
    nu3 = nu3 * pack2(pw<float>(lo(t), a.mu_exp), pw<float>(hi(t), a.mu_exp));
  }
  if constexpr (D == 3 && THERMAL) collide_central(q, c, nu3, a);
  else collide_full<D, F2, THERMAL, float>(q, c, nu3, a);

  S* __restrict__ gout = (S*)a.g_out;
  const bool both = act0 && act1;
  if (VEC && both) {
#pragma unroll
    for (int i = 0; i < Q; ++i) st_pop2(gout + (size_t)i * N + (unsigned)r, q[i]);
    if (a.write_u) {
#pragma unroll
      for (int d = 0; d < D; ++d) st2(a.u + (size_t)d * N + (unsigned)r, c.u[d]);
    }
  } else {
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      S* p = gout + (size_t)i * N + (unsigned)r;
      if (act0) st_pop<S, float>(p, lo(q[i]));
      if (act1) st_pop<S, float>(p + 1, hi(q[i]));
    }
    if (a.write_u) {
#pragma unroll
      for (int d = 0; d < D; ++d) {
        float* p = a.u + (size_t)d * N + (unsigned)r;
        if (act0) p[0] = lo(c.u[d]);
        if (act1) p[1] = hi(c.u[d]);
      }
    }
  }
  if (!a.write_u) {  // the outlet rule of the next step reads u
    if (out0 && act0)
      for (int d = 0; d < D; ++d) a.u[(size_t)d * N + r] = lo(c.u[d]);
    if (out1 && act1)
      for (int d = 0; d < D; ++d) a.u[(size_t)d * N + r + 1] = hi(c.u[d]);
  }
  if (a.ph_out) {
    const F2 p = fma_(splat<F2>(0.5), c.rl3, splat<F2>(a.P_ref) + c.psum);
    if (act0) a.ph_out[r] = lo(p);
    if (act1) a.ph_out[r + 1] = hi(p);
  }
  if ((act0 && !isfinite(lo(c.usq))) || (act1 && !isfinite(hi(c.usq)))) atomicOr(a.flag, 1);
}

// Whether every array of a pair launch may be accessed two elements at a time.
template <typename S> bool pair_aligned(const LBArgs<float>& a, bool thermal) {
  uintptr_t f = (uintptr_t)a.u | (uintptr_t)a.ph_out;
  if (thermal) f |= (uintptr_t)a.rho | (uintptr_t)a.lam | (uintptr_t)a.T;
  return a.geo.nx % 2 == 0 && f % 8 == 0 && ((uintptr_t)a.g_in | (uintptr_t)a.g_out) % (2 * sizeof(S)) == 0;
}

template <int D, typename S, bool THERMAL, bool LIST>
cudaError_t launch_pair(LBArgs<float> a, cudaStream_t st, bool pdl) {
  a.div_nx = FastDiv((uint32_t)a.geo.nx);
  a.div_ny = FastDiv((uint32_t)a.geo.ny);
  a.wall_planes = LIST ? (a.n_wall + LP_BLOCK - 1) / LP_BLOCK : 0;
  a.pdl = pdl;
  const int pairs = (a.geo.N + 1) / 2;
  const dim3 grid(a.wall_planes + (pairs + LP_BLOCK - 1) / LP_BLOCK);
  if (pair_aligned<S>(a, THERMAL))
    return launch_ex<LBArgs<float>>(lb_pair_kernel<D, S, THERMAL, true, LIST>, grid, dim3(LP_BLOCK), st, pdl, a);
  return launch_ex<LBArgs<float>>(lb_pair_kernel<D, S, THERMAL, false, LIST>, grid, dim3(LP_BLOCK), st, pdl, a);
}

// Small FP64 grids run blocks of one warp where the most loaded SM then holds fewer of the warps with cells:
// an FP64 instruction holds its sub-partition for 32 clocks, so the step lasts as long as the SM with the most
// warps. Blocks of 128 / of 32: planar flame 256x8 34.4 / 33.8 us per step, 2-D boxes 200x80 10.3 / 7.2,
// 129x240 17.4 / 10.3, level at 33x400 (8.2) and 97x300 (10.3; BGK 13.7 / 14.4, which the rule leaves at 128),
// 3-D 129x14x14 38.9 / 25.6. In 3-D only where a row takes several blocks of 128: with shorter rows the one-warp
// blocks of a row's full and last warps fall on the sub-partitions unevenly (33x28x28 27.4 / 36.7, 36x29x29
// 33.8 / 39.0). FP32 is bound by latency and gains nothing (2-D box 33x900 4.1 / 5.1).
constexpr int LB_ONE_WARP_MAX = 32768, LB_SMS = 152;
template <int D, typename R> bool one_warp_blocks(const Geo& g) {
  if (sizeof(R) == 4 || g.N >= LB_ONE_WARP_MAX || (D == 3 && g.nx <= LB_BLOCK)) return false;
  const long long rows = (long long)g.ny * g.nz, blocks = rows * ((g.nx + LB_BLOCK - 1) / LB_BLOCK);
  const long long warps = rows * ((g.nx + 31) / 32);
  // warps per SM: ceil(warps / SMs) against ceil(blocks / SMs) of warps / blocks each
  return (warps + LB_SMS - 1) / LB_SMS * blocks < (blocks + LB_SMS - 1) / LB_SMS * warps;
}

// FP32 arithmetic at the default rates: two cells per thread in 3-D, and in 2-D from PAIR_MIN_2D cells on; below that the grid does not fill the GPU
// with pairs and the longer threads cost what the fewer instructions save (chamber step, one cell / two:
// 256x64 13.47 / 13.53 us, 512x128 14.48 / 14.48, 600x200 17.58 / 16.59, 1024x256 27.20 / 25.07; 3-D
// gains at every size, e.g. periodic box of 82,615 cells 10.35 / 5.47 us). Otherwise one cell per thread.
constexpr int PAIR_MIN_2D = 100000;
template <int D, typename S, typename R, bool THERMAL, int COLL, bool LIST>
cudaError_t launch_cells(LBArgs<R> a, cudaStream_t st, bool pdl) {
  constexpr bool PAIR = COLL == COLL_CUMULANT_FULL && sizeof(R) == 4;
  if constexpr (PAIR) {
    if (D == 3 || a.geo.N >= PAIR_MIN_2D) return launch_pair<D, S, THERMAL, LIST>(a, st, pdl);
  }
  if constexpr (!PAIR || D == 2) {
    const int block = one_warp_blocks<D, R>(a.geo) ? 32 : LB_BLOCK;
    dim3 grid((a.geo.nx + block - 1) / block, a.geo.ny, a.geo.nz);
    const auto kernel = lb_step_kernel<D, S, R, THERMAL, COLL, LIST>;
    a.wall_planes = 0;
    if constexpr (LIST) {
      const size_t plane = (size_t)block * grid.x * grid.y;
      a.wall_planes = (int)((a.n_wall + plane - 1) / plane);
      if (grid.z + a.wall_planes > 65535u) {  // no planes left for the list: a launch of its own
        a.wall_planes = 1;
        const cudaError_t e = launch_ex<LBArgs<R>>(kernel, dim3((a.n_wall + block - 1) / block), dim3(block), st, pdl, a);
        if (e != cudaSuccess) return e;
        a.wall_planes = 0;
        pdl = false;
      }
      grid.z += a.wall_planes;
    }
    return launch_ex<LBArgs<R>>(kernel, grid, dim3(block), st, pdl, a);
  }
}

// pdl: the kernel may start while the one before it in the stream (the thermodynamic-pressure
// update) runs; it reads that kernel's state after pdl_wait. The cells of a wall list, a chain of latencies,
// take the first blocks of the same launch. As a launch of their own just before, that the other cells'
// started beside, the two needed a wait for each other; on a second stream, forked and joined by events, a
// graph ran them one after the other. Step of the swirl burner with curved walls, launch of its own beside /
// second stream / same launch: 96x48x48 62.4 / 64.1 / 53.0 us, 192x96x96 250 / 263 / 248; cold 128x64x64 FP32
// 53.0 / 48.5 / 45.4, FP16 27.9 / 33.7 / 22.8.
template <int D, typename S, typename R>
cudaError_t launch_lb(const LBArgs<R>& a, int thermal, int coll, cudaStream_t st, bool pdl) {
#define LB_LAUNCH(TH, CO) \
  return a.n_wall > 0 ? launch_cells<D, S, R, TH, CO, true>(a, st, pdl) : launch_cells<D, S, R, TH, CO, false>(a, st, pdl)
  if (thermal) {
    if (coll == COLL_CUMULANT_FULL) LB_LAUNCH(true, COLL_CUMULANT_FULL);
    else if (coll == COLL_CUMULANT) LB_LAUNCH(true, COLL_CUMULANT);
    else LB_LAUNCH(true, COLL_BGK);
  } else {
    if (coll == COLL_CUMULANT_FULL) LB_LAUNCH(false, COLL_CUMULANT_FULL);
    else if (coll == COLL_CUMULANT) LB_LAUNCH(false, COLL_CUMULANT);
    else LB_LAUNCH(false, COLL_BGK);
  }
#undef LB_LAUNCH
}

}  // namespace hlbm
