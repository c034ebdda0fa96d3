// Green operator of the homogeneous micropolar reference medium, per
// wavevector (sm_103a).
//
// For a non-zero, non-Nyquist wavevector xi the strain / curvature
// fluctuations (e^, gamma^) produced by the polarizations (tau^, mu^) are
// those of the periodic displacement and micro-rotation amplitudes (u, phi)
// that balance t = A0 e + tau, m = B0 gamma + mu in Fourier space (the
// balance laws eq. momemtum_balance with the kinematics of eq. strains):
//
//   [(mu+kap) k^2 I + (lam+mu-kap) xi xi^T] u - 2 i kap (xi x phi) = f,
//   [(gam k^2 + 4 kap) I + (alp+bet) xi xi^T] phi - 2 i kap (xi x u) = g,
//   f_l = i xi_k tau^_kl,   g_l = i xi_k mu^_kl + eps_lkm tau^_km.
//
// Splitting along xi / across xi gives the closed form
//   u   = xi (xi.f) / ((lam + 2 mu) k^4) + [b P f - c (xi x g)] / D,
//   phi = xi (xi.g) / (((alp+bet+gam) k^2 + 4 kap) k^2) + [a P g - c (xi x f)] / D,
// a = (mu+kap) k^2, b = gam k^2 + 4 kap, c = -2 i kap, D = k^2 ((mu+kap) gam k^2 + 4 kap mu),
// P = I - xi xi^T / k^2; then e^_kl = i xi_k u_l + eps_lkm phi_m,
// gamma^_kl = i xi_l phi_k.  Lambda^1,2 of the paper act only at xi = 0,
// where the fluctuation is zero (the averages are prescribed).
#pragma once

#include "mp_common.cuh"

namespace mp {

// In-place: v[0..8] = tau^ -> e^, v[9..17] = mu^ -> gamma^, times `scale`.
// v may point to shared memory: every input is read before the first output
// is written, and only the 12 reals of f, g and of u, phi are kept in
// registers, never the 36 of the point itself.
template <class R>
__device__ __forceinline__ void green_point(const RefDev<R>& A0, R x1, R x2, R x3, cpx<R>* v,
                                            R scale) {
  const R xi[3] = {x1, x2, x3};
  // f = i xi . tau  (f_l = i xi_k tau_kl), g = i xi . mu + eps : tau
  cpx<R> f[3], g[3];
#pragma unroll
  for (int l = 0; l < 3; ++l) {
    cpx<R> a = cmake<R>(R(0), R(0)), b = cmake<R>(R(0), R(0));
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      a = cfma(v[3 * k + l], xi[k], a);
      b = cfma(v[9 + 3 * k + l], xi[k], b);
    }
    f[l] = cmuli(a);
    g[l] = cmuli(b);
  }
  // (eps : tau)_1 = tau_23 - tau_32, _2 = tau_31 - tau_13, _3 = tau_12 - tau_21
  g[0] = cadd(g[0], csub(v[5], v[7]));
  g[1] = cadd(g[1], csub(v[6], v[2]));
  g[2] = cadd(g[2], csub(v[1], v[3]));

  const R k2 = x1 * x1 + x2 * x2 + x3 * x3;
  const R ik2 = R(1) / k2;
  const R a = (A0.mu + A0.kap) * k2;
  const R b = A0.gamma * k2 + R(4) * A0.kap;
  const R iD = R(1) / (k2 * ((A0.mu + A0.kap) * A0.gamma * k2 + R(4) * A0.kap * A0.mu));
  // u = f u_f + xi (xi.f) u_x + i c_i (xi x g): the projection's terms collected
  // (three roundings a component; P f, b P f and c (xi x g) in turn took five)
  const R u_f = b * iD, p_g = a * iD, c_i = R(2) * A0.kap * iD;
  const R u_x = fma(-u_f, ik2, ik2 * ik2 / (A0.lam + R(2) * A0.mu));
  const R p_x = fma(-p_g, ik2, ik2 / ((A0.alpha + A0.beta + A0.gamma) * k2 + R(4) * A0.kap));

  cpx<R> xf = cmake<R>(R(0), R(0)), xg = cmake<R>(R(0), R(0));
#pragma unroll
  for (int l = 0; l < 3; ++l) {
    xf = cfma(f[l], xi[l], xf);
    xg = cfma(g[l], xi[l], xg);
  }
  // cross products xi x g, xi x f
  cpx<R> cg[3], cf[3];
  cg[0] = cfma(g[1], -x3, cscale(g[2], x2));
  cg[1] = cfma(g[2], -x1, cscale(g[0], x3));
  cg[2] = cfma(g[0], -x2, cscale(g[1], x1));
  cf[0] = cfma(f[1], -x3, cscale(f[2], x2));
  cf[1] = cfma(f[2], -x1, cscale(f[0], x3));
  cf[2] = cfma(f[0], -x2, cscale(f[1], x1));

  cpx<R> u[3], ph[3];
#pragma unroll
  for (int l = 0; l < 3; ++l) {
    u[l] = cfma(f[l], u_f, cfma(xf, xi[l] * u_x, cmuli(cscale(cg[l], c_i))));
    ph[l] = cfma(g[l], p_g, cfma(xg, xi[l] * p_x, cmuli(cscale(cf[l], c_i))));
  }
  // e^_kl = i xi_k u_l + eps_lkm phi_m ; gamma^_kl = i phi_k xi_l, scaled, each
  // component written once.
  // eps_lkm phi_m: (1,2) -phi3, (2,1) +phi3, (1,3) +phi2, (3,1) -phi2, (2,3) -phi1, (3,2) +phi1
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    u[i] = cscale(u[i], scale);
    ph[i] = cscale(ph[i], scale);
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) {
#pragma unroll
    for (int l = 0; l < 3; ++l) {
      // eps_lkm phi_m, m = 3 - k - l: -phi_m for (k, l) cyclic, +phi_m else
      const cpx<R> iu = cmuli(u[l]);
      cpx<R> ev;
      if (k == l) ev = cscale(iu, xi[k]);
      else if (l == (k + 1) % 3) ev = cfma(iu, xi[k], cmake<R>(-ph[3 - k - l].x, -ph[3 - k - l].y));
      else ev = cfma(iu, xi[k], ph[3 - k - l]);
      v[3 * k + l] = ev;
      v[9 + 3 * k + l] = cmuli(cscale(ph[k], xi[l]));
    }
  }
}

// The same operator on the 12 reduced values of a point (mp_lines.cuh): in,
// for l = 0..2, v[4l..4l+3] = A_l, T_l, B_l, M_l with f_l = A_l + i x3 T_l and
// g_l = B_l + i x3 M_l; out u_l, e_3l = i x3 u_l + eps_l3m phi_m, phi_l,
// gamma_l3 = i x3 phi_l times `scale`.
// v points to shared memory, 16-byte aligned; it moves in 16-byte pieces.
template <class R>
__device__ __forceinline__ void green_point_reduced(const RefDev<R>& A0, R x1, R x2, R x3, cpx<R>* v, R scale) {
  struct __align__(16) Piece {
    R w[16 / sizeof(R)];
  };
  const R xi[3] = {x1, x2, x3};
  cpx<R> f[3], g[3];
#pragma unroll
  for (int l = 0; l < 3; ++l) {
    __align__(16) cpx<R> q[4];
#pragma unroll
    for (int i = 0; i < (int)sizeof(q) / 16; ++i)
      reinterpret_cast<Piece*>(q)[i] = reinterpret_cast<const Piece*>(v + 4 * l)[i];
    f[l] = cmake<R>(fma(-x3, q[1].y, q[0].x), fma(x3, q[1].x, q[0].y));
    g[l] = cmake<R>(fma(-x3, q[3].y, q[2].x), fma(x3, q[3].x, q[2].y));
  }
  const R k2 = x1 * x1 + x2 * x2 + x3 * x3;
  const R ik2 = R(1) / k2;
  const R a = (A0.mu + A0.kap) * k2;
  const R b = A0.gamma * k2 + R(4) * A0.kap;
  const R iD = scale / (k2 * ((A0.mu + A0.kap) * A0.gamma * k2 + R(4) * A0.kap * A0.mu));
  const R u_f = b * iD, p_g = a * iD, c_i = R(2) * A0.kap * iD;
  const R u_x = fma(-u_f, ik2, scale * ik2 * ik2 / (A0.lam + R(2) * A0.mu));
  const R p_x = fma(-p_g, ik2, scale * ik2 / ((A0.alpha + A0.beta + A0.gamma) * k2 + R(4) * A0.kap));
  cpx<R> xf = cmake<R>(R(0), R(0)), xg = cmake<R>(R(0), R(0));
#pragma unroll
  for (int l = 0; l < 3; ++l) {
    xf = cfma(f[l], xi[l], xf);
    xg = cfma(g[l], xi[l], xg);
  }
  cpx<R> cg[3], cf[3];  // xi x g, xi x f
  cg[0] = cfma(g[1], -x3, cscale(g[2], x2));
  cg[1] = cfma(g[2], -x1, cscale(g[0], x3));
  cg[2] = cfma(g[0], -x2, cscale(g[1], x1));
  cf[0] = cfma(f[1], -x3, cscale(f[2], x2));
  cf[1] = cfma(f[2], -x1, cscale(f[0], x3));
  cf[2] = cfma(f[0], -x2, cscale(f[1], x1));
  cpx<R> u[3], ph[3];
#pragma unroll
  for (int l = 0; l < 3; ++l) {
    u[l] = cfma(f[l], u_f, cfma(xf, xi[l] * u_x, cmuli(cscale(cg[l], c_i))));
    ph[l] = cfma(g[l], p_g, cfma(xg, xi[l] * p_x, cmuli(cscale(cf[l], c_i))));
  }
#pragma unroll
  for (int l = 0; l < 3; ++l) {
    __align__(16) cpx<R> q[4];
    q[0] = u[l];
    q[1] = l == 0   ? cfma(cmuli(u[0]), x3, cmake<R>(-ph[1].x, -ph[1].y))
           : l == 1 ? cfma(cmuli(u[1]), x3, ph[0])
                    : cscale(cmuli(u[2]), x3);
    q[2] = ph[l];
    q[3] = cscale(cmuli(ph[l]), x3);
#pragma unroll
    for (int i = 0; i < (int)sizeof(q) / 16; ++i)
      reinterpret_cast<Piece*>(v + 4 * l)[i] = reinterpret_cast<const Piece*>(q)[i];
  }
}

}  // namespace mp
