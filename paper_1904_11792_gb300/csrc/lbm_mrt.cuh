// Multiple-relaxation-time collision arithmetic of one node (used by the
// collide-stream bodies of lbm_node.cuh when the lattice selects it).
#pragma once

#include <utility>

#include "lbm_internal.h"

namespace lbm {

// ---------------------------------------------------------------------------
// Multiple-relaxation-time collision (the operator the conclusions name as
// the next step; not specified in the paper).  D3Q19 moments of d'Humieres,
// Ginzburg, Krafczyk, Lallemand and Luo (2002), rows as polynomials of the
// velocity c, and the forcing of Guo, Zheng and Shi (2002) in moment space:
//   m* = m - S (m - m_eq(rho, u)) + (I - S/2) M F_guo,  u = (j + F/2)/rho,
//   f* = M^-1 m* = M^T diag(1/|row|^2) m*.
// m_eq and M F_guo are the moments of Eq. 2's equilibrium and of Guo's
// forcing populations, in closed form.
// ---------------------------------------------------------------------------
__host__ __device__ constexpr int mrt_coef(int k, int a) {
  const int x = cx(a), y = cy(a), z = cz(a), c2 = x * x + y * y + z * z;
  switch (k) {
    case 0: return 1;
    case 1: return 19 * c2 - 30;
    case 2: return (21 * c2 * c2 - 53 * c2 + 24) / 2;
    case 3: return x;
    case 4: return (5 * c2 - 9) * x;
    case 5: return y;
    case 6: return (5 * c2 - 9) * y;
    case 7: return z;
    case 8: return (5 * c2 - 9) * z;
    case 9: return 3 * x * x - c2;
    case 10: return (3 * c2 - 5) * (3 * x * x - c2);
    case 11: return y * y - z * z;
    case 12: return (3 * c2 - 5) * (y * y - z * z);
    case 13: return x * y;
    case 14: return y * z;
    case 15: return x * z;
    case 16: return (y * y - z * z) * x;
    case 17: return (z * z - x * x) * y;
    default: return (x * x - y * y) * z;
  }
}
__host__ __device__ constexpr int mrt_norm(int k) {
  int n = 0;
  for (int a = 0; a < Q; ++a) n += mrt_coef(k, a) * mrt_coef(k, a);
  return n;
}

// v (+)= c * x with c a compile-time integer (0, +-1 and other values).
template <int Cf, typename C>
__device__ __forceinline__ void mrt_fma(C& v, C x) {
  if constexpr (Cf == 1) v = vadd(v, x);
  else if constexpr (Cf == -1) v = vsub(v, x);
  else if constexpr (Cf != 0) v = xfma(splat<C>((typename Lane<C>::S)Cf), x, v);
}
// m[K] = sum_a M[K][a] f[a] and f[A] = sum_k M[k][A] w[k], expanded at compile
// time so that only the non-zero integer coefficients cost instructions.
template <typename C, int K, int... A>
__device__ __forceinline__ C mrt_row(const C* f, std::integer_sequence<int, A...>) {
  C v = splat<C>((typename Lane<C>::S)0);
  (mrt_fma<mrt_coef(K, A)>(v, f[A]), ...);
  return v;
}
template <typename C, int A, int... K>
__device__ __forceinline__ C mrt_col(const C* w, std::integer_sequence<int, K...>) {
  C v = splat<C>((typename Lane<C>::S)0);
  (mrt_fma<mrt_coef(K, A)>(v, w[K]), ...);
  return v;
}
template <typename C, int... K>
__device__ __forceinline__ void mrt_forward(const C* f, C* m, std::integer_sequence<int, K...>) {
  ((m[K] = mrt_row<C, K>(f, std::make_integer_sequence<int, Q>{})), ...);
}
template <typename C, int... K>
__device__ __forceinline__ void mrt_scale(C* m, std::integer_sequence<int, K...>) {
  ((m[K] = xmul(m[K], splat<C>((typename Lane<C>::S)(1.0 / (double)mrt_norm(K))))), ...);
}
template <typename C, int... A>
__device__ __forceinline__ void mrt_backward(const C* w, C* fs, std::integer_sequence<int, A...>) {
  ((fs[A + 1] = mrt_col<C, A + 1>(w, std::make_integer_sequence<int, Q>{})), ...);
}

// Post-collision populations of a node with density rho, momentum (jx, jy,
// jz), psi pc and link sums as collide_math_ls.  C = float2 computes two nodes
// in paired FP32 instructions, lane by lane with the bits of C = float; the
// rates come from the host in FP32 (converted here they cost FP64-pipe
// operations).  256x128x128 FP32, 20 diagnosed steps: 2630 us one node at a
// time, 2462 us.
template <typename C>
__device__ __forceinline__ void collide_math_mrt_ls(const Phys& ph, const C f[Q], C rho, C jx, C jy, C jz, C pc, C ax,
                                                    C ay, C az, C dx, C dy, C dz, C fs[Q]) {
  using S = typename Lane<C>::S;
  auto k = [](double v) { return splat<C>((S)v); };
  S G_s, s_e, s_eps, s_q, s_pi, s_m, s_nu, h_e, h_eps, h_q, h_pi, h_nu;   // rates and 1 - rate / 2
  if constexpr (sizeof(S) == 4) {
    G_s = ph.G_f;
    s_e = ph.mrt_sf[0], s_eps = ph.mrt_sf[1], s_q = ph.mrt_sf[2], s_pi = ph.mrt_sf[3], s_m = ph.mrt_sf[4];
    s_nu = ph.omega_f;
    h_e = ph.mrt_hf[0], h_eps = ph.mrt_hf[1], h_q = ph.mrt_hf[2], h_pi = ph.mrt_hf[3], h_nu = ph.mrt_hf[4];
  } else {
    G_s = ph.G;
    s_e = ph.s_e, s_eps = ph.s_eps, s_q = ph.s_q, s_pi = ph.s_pi, s_m = ph.s_m, s_nu = ph.omega;
    h_e = xfma(-0.5, s_e, 1.0), h_eps = xfma(-0.5, s_eps, 1.0), h_q = xfma(-0.5, s_q, 1.0);
    h_pi = xfma(-0.5, s_pi, 1.0), h_nu = xfma(-0.5, s_nu, 1.0);
  }
  const C w1 = k(1.0 / 18.0), w2 = k(1.0 / 36.0);
  // products and sums through the forms that are not contracted: the same
  // bits in every kernel (see collide_math_ls)
  const C gp = xmul(splat<C>(-G_s), pc);
  const C Fx = xmul(gp, xfma(w1, ax, xmul(w2, dx)));
  const C Fy = xmul(gp, xfma(w1, ay, xmul(w2, dy)));
  const C Fz = xmul(gp, xfma(w1, az, xmul(w2, dz)));
  // Guo's velocity
  const C half = k(0.5), inv_rho = rcp_node(rho);
  const C ux = xmul(xfma(half, Fx, jx), inv_rho);
  const C uy = xmul(xfma(half, Fy, jy), inv_rho);
  const C uz = xmul(xfma(half, Fz, jz), inv_rho);
  // moments m = M f
  C m[Q];
  mrt_forward<C>(f, m, std::make_integer_sequence<int, Q>{});
  // equilibrium and forcing moments
  const C two = k(2.0);
  const C ux2 = xmul(ux, ux), uy2 = xmul(uy, uy), uz2 = xmul(uz, uz);
  const C uu = vadd(vadd(ux2, uy2), uz2);
  const C uF = xfma(uz, Fz, xfma(uy, Fy, xmul(ux, Fx)));
  const C pxx = vsub(vsub(xmul(two, ux2), uy2), uz2), pww = vsub(uy2, uz2);   // 2 ux2 is exact
  const C fyy = xmul(Fy, uy), fzz = xmul(Fz, uz);
  const C fxx = xmul(two, vsub(vsub(xmul(two, xmul(Fx, ux)), fyy), fzz)), fww = xmul(two, vsub(fyy, fzz));
  auto relax = [&](C mk, C meq, S s, S h, C src) {
    return xfma(splat<C>(h), src, xfma(splat<C>(-s), vsub(mk, meq), mk));
  };
  C ms[Q];
  ms[0] = rho;
  ms[3] = vadd(jx, Fx);
  ms[5] = vadd(jy, Fy);
  ms[7] = vadd(jz, Fz);
  ms[1] = relax(m[1], xmul(rho, xfma(k(19.0), uu, k(-11.0))), s_e, h_e, xmul(k(38.0), uF));
  ms[2] = relax(m[2], xmul(rho, xfma(k(-5.5), uu, k(3.0))), s_eps, h_eps, xmul(k(-11.0), uF));
  const C mtwo3 = k(-2.0 / 3.0), mhalf = k(-0.5);
  const C mr = xmul(mtwo3, rho);
  ms[4] = relax(m[4], xmul(mr, ux), s_q, h_q, xmul(mtwo3, Fx));
  ms[6] = relax(m[6], xmul(mr, uy), s_q, h_q, xmul(mtwo3, Fy));
  ms[8] = relax(m[8], xmul(mr, uz), s_q, h_q, xmul(mtwo3, Fz));
  const C rpxx = xmul(rho, pxx), rpww = xmul(rho, pww);
  ms[9] = relax(m[9], rpxx, s_nu, h_nu, fxx);
  ms[10] = relax(m[10], xmul(mhalf, rpxx), s_pi, h_pi, xmul(mhalf, fxx));
  ms[11] = relax(m[11], rpww, s_nu, h_nu, fww);
  ms[12] = relax(m[12], xmul(mhalf, rpww), s_pi, h_pi, xmul(mhalf, fww));
  ms[13] = relax(m[13], xmul(xmul(rho, ux), uy), s_nu, h_nu, xfma(Fy, ux, xmul(Fx, uy)));
  ms[14] = relax(m[14], xmul(xmul(rho, uy), uz), s_nu, h_nu, xfma(Fz, uy, xmul(Fy, uz)));
  ms[15] = relax(m[15], xmul(xmul(rho, ux), uz), s_nu, h_nu, xfma(Fz, ux, xmul(Fx, uz)));
  const C nsm = splat<C>(-s_m);
  ms[16] = xfma(nsm, m[16], m[16]);
  ms[17] = xfma(nsm, m[17], m[17]);
  ms[18] = xfma(nsm, m[18], m[18]);
  // f* = M^T diag(1/|row|^2) m*; the rest population takes the remainder of
  // the density so that each collision conserves mass up to one rounding
  mrt_scale<C>(ms, std::make_integer_sequence<int, Q>{});
  mrt_backward<C>(ms, fs, std::make_integer_sequence<int, Q - 1>{});
  C rest = rho;
#pragma unroll
  for (int a = 1; a < Q; ++a) rest = vsub(rest, fs[a]);
  fs[0] = rest;
}

// The same from the neighbour values pn[a] = psi(x + c_a) (a = 1..18).
template <typename C>
__device__ __forceinline__ void collide_math_mrt(const Phys& ph, const C f[Q], C pc, const C pn[Q], C fs[Q]) {
  C jx, jy, jz, ax, ay, az, dx, dy, dz;
  link_sums<C>(pn, ax, ay, az, dx, dy, dz);
  mom_of<C>(f, jx, jy, jz);
  collide_math_mrt_ls<C>(ph, f, rho_of<C>(f), jx, jy, jz, pc, ax, ay, az, dx, dy, dz, fs);
}

}  // namespace lbm
