// Per-node device code of the two step kernels, shared by the single-lattice
// kernels (step_kernels.cu) and the batched multi-lattice kernels (batch.cu) so
// that both perform identical arithmetic.
//
// The GB300 FP64 pipe issues about 0.53e12 instructions/s, a 38th of the integer pipes, so
// the per-node arithmetic runs on the integer pipes in fixed point (fixsum.cuh, fixmul.cuh,
// eos_fixed.cuh, collide_fixed.cuh), bound by their issue rather than by HBM; the
// double-precision forms below run the nodes that the frames cannot hold, and the fields.
//  * K1 hands K2 the moments instead of the populations, so K2 never re-sums f.
//  * With Lambda = I or with only the shear rates relaxing, f* is rebuilt
//    directly as w_i [rho + 3 c.P + 4.5 (c c - I/3) : Pi] plus the sigma term of
//    the Li scheme, which M^-1 maps onto (-8, 1, ..., 1) z. This equals
//    M^-1 m* for the moment vector m* of Eq. LiFS / GFS.
//  * |F|^2 / psi^2 is (G^2/144) |g|^2 with g the weighted psi differences, so the
//    Li term needs no division by psi^2.
//  * The optional surface-tension control (template flag ST) adds Li & Luo's
//    source C to m*; in population space it joins the Li term's z and the rows
//    7, 8 terms, and costs nothing when the flag is off.
#pragma once

#include <cuda_runtime.h>

#include "eos_dev.cuh"
#include "fixsum.cuh"
#include "fp64.cuh"
#include "internal.h"

namespace pplbm {

// K1 body for node i in double precision: moments, EOS, psi (Eqs. Density, Momentum, CS,
// Sec. III.D, InteractionPotential); error word on a non-finite or non-positive density or
// psi^2. Runs for the nodes outside the fixed-point path's domain.
template <int KIND>
__device__ __forceinline__ void rho_psi_double(const StepArgs& a, const double* f, int i) {
  const int N = (int)a.n;  // 9 n < 2^31: plane offsets fit 32 bits
  const double f0 = f[i], f1 = f[N + i], f2 = f[2 * N + i], f3 = f[3 * N + i], f4 = f[4 * N + i];
  const double f5 = f[5 * N + i], f6 = f[6 * N + i], f7 = f[7 * N + i], f8 = f[8 * N + i];
  double rho, jx, jy, m7 = 0.0, m8 = 0.0;
  // When all nine populations are positive normal doubles (every bulk and interface
  // node of a physical state), the moments are exact integer sums in one fixed-point
  // frame, each rounded once (fixsum.cuh). Otherwise the same moments as IEEE sums.
  const double fv[9] = {f0, f1, f2, f3, f4, f5, f6, f7, f8};
  unsigned max_hi = 0;
  if (KIND != kFullMrt && fx::positive_normal_range(fv, &max_hi)) {
    fx::density_moments<KIND == kShearTau>(fv, fx::frame_top(max_hi), &rho, &jx, &jy, &m7, &m8);
  } else if (KIND == kShearTau) {
    // rows 7, 8 of Eq. MatrixMRT share their pair sums with rho
    const double a13 = f1 + f3, a24 = f2 + f4, a57 = f5 + f7, a68 = f6 + f8;
    rho = f0 + ((a13 + a24) + (a57 + a68));
    const double p = f5 - f7, q = f6 - f8;
    jx = (f1 - f3) + (p - q);
    jy = (f2 - f4) + (p + q);
    m7 = a13 - a24;
    m8 = a57 - a68;
  } else {
    const double sxp = f1 + f5 + f8;  // populations with c_x = +1
    const double sxm = f3 + f6 + f7;  // c_x = -1
    rho = (f0 + f2 + f4) + (sxp + sxm);
    jx = sxp - sxm;
    jy = (f2 + f5 + f6) - (f4 + f7 + f8);
  }
  const double psi2 = eos_psi2_dev(a.eos, rho);
  // 0 < rho < 1e300 and 0 < psi^2 < inf, tested on the bit patterns (integer pipe)
  const long long rb = dbits(rho), pb = dbits(psi2);
  if (!(rb > 0 && rb < 0x7E37E43C8800759CLL && pb > 0 && pb < 0x7FF0000000000000LL)) atomicOr(a.err, 1);
  a.psi[i] = fast_sqrt(psi2);
  double* __restrict__ m = a.mom;
  m[i] = rho;
  m[N + i] = jx;
  m[2 * N + i] = jy;
  if (KIND == kShearTau) {
    m[3 * N + i] = m7;  // row 7 of Eq. MatrixMRT
    m[4 * N + i] = m8;  // row 8
  } else if (KIND == kFullMrt) {
    const double ax = f1 + f2 + f3 + f4, dg = f5 + f6 + f7 + f8;
    m[3 * N + i] = -4.0 * f0 - ax + 2.0 * dg;                    // row 1 (e)
    m[4 * N + i] = 4.0 * f0 - 2.0 * ax + dg;                     // row 2 (varsigma)
    m[5 * N + i] = -2.0 * (f1 - f3) + ((f5 - f6) - (f7 - f8));   // row 4 (q_x)
    m[6 * N + i] = -2.0 * (f2 - f4) + ((f5 + f6) - (f7 + f8));   // row 6 (q_y)
    m[7 * N + i] = (f1 + f3) - (f2 + f4);                        // row 7
    m[8 * N + i] = (f5 + f7) - (f6 + f8);                        // row 8
  }
}

template <int KIND>
__device__ __noinline__ void rho_psi_general(const StepArgs& a, const double* f, int i) {
  rho_psi_double<KIND>(a, f, i);
}

// K1 body for node i, in fixed point: the moments as exact integer sums in one frame
// (density_moments; with six relaxation times also rows 1, 2, 4, 6, 7, 8), the EOS and psi
// from the unrounded density sum (eos_fixed.cuh); the FP64 pipe only converts the results.
// Nodes the frames cannot hold (a population at or below zero or not finite, a density or
// EOS branch outside eos_fixed.cuh's domain) run the double-precision body, which raises
// the error word. What bounds it: the integer ALU pipe (ncu on a 2048 x 1024 droplet whose
// warps take the C-S and an ellipse branch: 636 instructions per node, ALU 76 % busy, FP64
// 31 %, 58 us). With the EOS and the root on the FP64 pipe (15 to 26 FP64 instructions per
// node) that pipe was 85 % busy and the pass took 107 us; over a batch of 12.9 M nodes
// 0.444 ms before, 0.282 ms now. The rms error of psi is 0.30 ulp on every branch (0.58
// next to the vapour at T_r = 0.35), where double precision gave 0.4 to 1.0 (22).
// (f is a plain pointer: the kernels that run several steps write it themselves.)
template <int KIND>
__device__ __forceinline__ void rho_psi_node(const StepArgs& a, const double* f, int i) {
  using namespace fx;
  const int N = (int)a.n;
  u64 b[9];
#pragma unroll
  for (int k = 0; k < 9; ++k) b[k] = bits_of(f[k * N + i]);
  u32 mn = hi32(b[0]), mx = mn;
#pragma unroll
  for (int k = 1; k < 9; k += 2) {
    mn = min3(mn, hi32(b[k]), hi32(b[k + 1]));
    mx = max3(mx, hi32(b[k]), hi32(b[k + 1]));
  }
  // positive normal populations, the largest in [2^-767, 2^993)
  bool ok = a.efix.ok && mn >= 0x00100000u && mx - 0x10000000u < 0x6E000000u;
  const int eg = frame_top(mx);
  u64 t[9];
#pragma unroll
  for (int k = 0; k < 9; ++k) t[k] = shr_u(significand(b[k]), eg - (int)(hi32(b[k]) >> 20));
  const u64 sxp = t[1] + t[5] + t[8], sxm = t[3] + t[6] + t[7];  // c_x = +1, -1
  const u64 syp = t[2] + t[5] + t[6], sym = t[4] + t[7] + t[8];  // c_y = +1, -1
  const u64 S = t[0] + t[2] + t[4] + sxp + sxm;                  // in [2^59, 2^64)
  const int k0 = eg - 1086;
  const double rho = scale2(bits_of(__ull2double_rn(S)), k0);
  const int lz = clz32((u32)(S >> 32));
  i64 P;
  int ex;
  ok = ok && psi2_fixed(a.efix, a.eos, S << (lz & 31), eg - lz, (i64)bits_of(rho), &P, &ex);
  if (!ok) {
    rho_psi_general<KIND>(a, f, i);
    return;
  }
  a.psi[i] = sqrt_double(P, ex);
  double* __restrict__ m = a.mom;
  m[i] = rho;
  m[N + i] = frame_to_double((i64)(sxp - sxm), k0);
  m[2 * N + i] = frame_to_double((i64)(syp - sym), k0);
  if (KIND == kShearTau) {
    m[3 * N + i] = frame_to_double((i64)((t[1] + t[3]) - (t[2] + t[4])), k0);  // row 7 of Eq. MatrixMRT
    m[4 * N + i] = frame_to_double((i64)((t[5] + t[7]) - (t[6] + t[8])), k0);  // row 8
  } else if (KIND == kFullMrt) {
    // rows 1, 2, 4, 6, 7, 8, each below 2^63 in magnitude
    const u64 ax = t[1] + t[2] + t[3] + t[4], dg = t[5] + t[6] + t[7] + t[8];
    m[3 * N + i] = frame_to_double((i64)(2 * dg - ax - 4 * t[0]), k0);
    m[4 * N + i] = frame_to_double((i64)(4 * t[0] - 2 * ax + dg), k0);
    m[5 * N + i] = frame_to_double((i64)(2 * (t[3] - t[1]) + ((t[5] - t[6]) - (t[7] - t[8]))), k0);
    m[6 * N + i] = frame_to_double((i64)(2 * (t[4] - t[2]) + ((t[5] + t[6]) - (t[7] + t[8]))), k0);
    m[7 * N + i] = frame_to_double((i64)((t[1] + t[3]) - (t[2] + t[4])), k0);
    m[8 * N + i] = frame_to_double((i64)((t[5] + t[7]) - (t[6] + t[8])), k0);
  }
}

__device__ __forceinline__ int wrap_index(int v, int n) {
  v %= n;
  return v < 0 ? v + n : v;
}

struct Post {
  double f[9];
};

// Surface-tension control (the technique of the paper's Sec. V; Li & Luo 2013):
// Q_ab = kappa (G/2) psi(x) sum_i w(|c_i|^2) [psi(x + c_i) - psi(x)] c_ia c_ib, kept as
// raw stencil sums with the scale k = kappa_q psi(x) (kappa_q = kappa G / 24), so that
// each use is one FMA:
//   (Q_xx + Q_yy) / 24 = k t,  t = (pE + pW + pN + pS)/6 + (four diagonals)/12 - psi,
//   Q_xx - Q_yy = 4 k sd,     sd = (pE + pW) - (pN + pS),
//   Q_xy = k xd,              xd = (pNE + pSW) - (pNW + pSE)
// (12 sum_i w_i [psi_i - psi] c_x^2 = 4 (pE + pW) + diagonals - 12 psi, likewise in y).
struct SurfQ {
  double k, t, sd, xd;
};

__device__ __forceinline__ SurfQ surface_q(const StepArgs& a, double p0, double pE, double pW, double pN, double pS,
                                           double pNE, double pNW, double pSW, double pSE) {
  const double sA = pE + pW, sB = pN + pS;
  const double dP = pNE + pSW, dM = pNW + pSE;
  SurfQ q;
  q.k = a.kappa_q * p0;
  q.t = fma(1.0 / 6.0, sA + sB, fma(1.0 / 12.0, dP + dM, -p0));
  q.sd = sA - sB;
  q.xd = dP - dM;
  return q;
}

// Collision for Lambda = I (KIND kUnitTau) or shear-only relaxation (kShearTau).
//
// With h = F/2: J = j + h = rho u (Eq. Momentum), P = j + 2h (momentum after the
// step), and the post-collision second moments (Lambda = I)
//   Pi_xx = rho ux^2 + ux Fx = ux (P_x + h_x),  Pi_yy = uy (P_y + h_y),
//   Pi_xy = rho ux uy + (ux Fy + uy Fx)/2 = ux P_y + uy h_x.
// These are rows 1, 7, 8 of m* = m_eq + S/2 (Eqs. LiFS, GFS with tau = 1);
// kShearTau relaxes rows 7, 8 with omega = 1/tau(rho) instead (Eq. RelaxationTime).
// Then
//   f*_i = w_i [rho + 3 c_i.P + 4.5 (c_i c_i - I/3) : Pi] + z_i,
// z_i = zz (-8, 1, 1, 1, 1, 1, 1, 1, 1) being M^-1 applied to the Li sigma terms
// +-12 sigma |F|^2 / psi^2 of rows 1 and 2 (tau_e = tau_zeta = 1), zz = sigma |F|^2 / (3 psi^2).
// With ST, the surface-tension source's rows 1, 2 (+-1.5 tr Q) map onto the same
// shape with zz += tr Q / 24, and rows 7, 8 (-l_nu (Q_xx - Q_yy), -l_nu Q_xy) add to
// the post-collision m_7, m_8 (l_nu = 1, or omega for kShearTau).
template <int KIND, bool ST = false>
__device__ __forceinline__ void collide_reduced(const StepArgs& a, int64_t node, double rho, double jx, double jy,
                                                double psi0, double gx, double gy, const SurfQ& sq, Post& out,
                                                double* ux_o, double* uy_o) {
  // Additions run on the integer pipe (add_int, bitwise the FP64 add); the FP64 pipe, which
  // bounds this form, keeps the products and fused multiply-adds.
  const double cH = a.half_force * psi0;  // h = cH g, cH = -G psi / 24
  const double hx = cH * gx, hy = cH * gy;
  const double inv_rho = fast_rcp(rho);
  const double ux = add_int(jx, hx) * inv_rho, uy = add_int(jy, hy) * inv_rho;
  *ux_o = ux;
  *uy_o = uy;
  const double Px = fma(2.0, hx, jx), Py = fma(2.0, hy, jy);
  const double Pxx = ux * add_int(Px, hx), Pyy = uy * add_int(Py, hy);
  const double tr = add_int(Pxx, Pyy);
  const double Pxy_eq = fma(ux, Py, uy * hx);
  double zz = a.zz_scale * fma(gx, gx, gy * gy);
  if (ST) zz = fma(sq.k, sq.t, zz);  // + tr Q / 24
  const double B0 = fma(-1.5, tr, rho);
  const double Q = fma(B0, 1.0 / 9.0, zz);
  double axp, ayp, Pxy;
  if (KIND == kUnitTau) {
    axp = fma(0.5, Pxx, Q);
    ayp = fma(0.5, Pyy, Q);
    Pxy = Pxy_eq;
    if (ST) {
      axp = fma(-sq.k, sq.sd, axp);  // m_7* -= Q_xx - Q_yy, n_7 = m_7 / 4
      ayp = fma(sq.k, sq.sd, ayp);
      Pxy = fma(-sq.k, sq.xd, Pxy);  // m_8* -= Q_xy
    }
  } else {
    // rows 7, 8: m* = m - omega (m - m_eq) + (1 - omega/2) S. With m_eq + S/2 the
    // unit-tau values Pi_xx - Pi_yy and Pi_xy above, this is
    //   m* = (m_eq + S/2) + (1 - omega) (m + S - m_eq - S/2),
    // and the brackets reduce to m7 - ux (jx - hx) + uy (jy - hy) and m8 - ux jy + uy hx.
    const double om = fast_rcp(fma(a.tau_b, rho, a.tau_a));
    const double omc = sub_int(1.0, om);
    const double m7 = a.mom[3 * a.n + node], m8 = a.mom[4 * a.n + node];
    const double A7 = fma(-ux, sub_int(jx, hx), fma(uy, sub_int(jy, hy), m7));
    const double A8 = fma(-ux, jy, fma(uy, hx, m8));
    double m7s = fma(omc, A7, sub_int(Pxx, Pyy));
    Pxy = fma(omc, A8, Pxy_eq);
    if (ST) {
      const double ok = om * sq.k;
      m7s = fma(-4.0 * ok, sq.sd, m7s);  // -omega (Q_xx - Q_yy)
      Pxy = fma(-ok, sq.xd, Pxy);        // -omega Q_xy
    }
    const double T4 = fma(0.25, tr, Q);
    axp = fma(0.25, m7s, T4);  // Q + Pi_xx/2 with Pi_xx = (tr + m7*)/2
    ayp = fma(-0.25, m7s, T4);
  }
  out.f[0] = fma(4.0 / 9.0, B0, -8.0 * zz);
  out.f[1] = fma(Px, 1.0 / 3.0, axp);
  out.f[3] = fma(-Px, 1.0 / 3.0, axp);
  out.f[2] = fma(Py, 1.0 / 3.0, ayp);
  out.f[4] = fma(-Py, 1.0 / 3.0, ayp);
  const double Dq = fma(fma(3.0, tr, rho), 1.0 / 36.0, zz);
  const double dp = fma(0.25, Pxy, Dq), dm = fma(-0.25, Pxy, Dq);
  const double ps = add_int(Px, Py), pd = sub_int(Py, Px);
  out.f[5] = fma(ps, 1.0 / 12.0, dp);
  out.f[7] = fma(-ps, 1.0 / 12.0, dp);
  out.f[6] = fma(pd, 1.0 / 12.0, dm);
  out.f[8] = fma(-pd, 1.0 / 12.0, dm);
}

// The same collision (Lambda = I, or rows 7, 8 at omega = 1/tau(rho) for kShearTau),
// without the surface-tension source, for the nodes that leave the fixed-point path
// (collide_general), arranged so that the FP64 pipe does only the
// products, the reciprocals and the Li term (19 FP64 instructions per node for unit
// relaxation times, 32 for the two-phase set): the sums J = j + h, P = j + 2h,
// P + h (and j - h) come from one fixed-point frame, and the nine populations are
// exact small-integer combinations of the inputs scaled by 1/36 (fixsum.cuh), each
// rounded once, instead of chains of FP64 fused multiply-adds.
template <int KIND>
__device__ __forceinline__ void collide_reduced_fx(const StepArgs& a, int64_t node, double rho, double jx, double jy,
                                                   double psi0, double gx, double gy, Post& out) {
  constexpr bool kShear = KIND == kShearTau;
  const double cH = a.half_force * psi0;  // h = F/2 = cH g, cH = -G psi / 24
  const double hx = cH * gx, hy = cH * gy;
  double Jx, Px, Qx, Kx = 0.0, Jy, Py, Qy, Ky = 0.0;
  fx::j_h_combos<kShear>(jx, hx, &Jx, &Px, &Qx, &Kx);
  fx::j_h_combos<kShear>(jy, hy, &Jy, &Py, &Qy, &Ky);
  const double inv36 = fast_rcp(36.0 * rho);
  const double ux = Jx * inv36, uy = Jy * inv36;  // u / 36
  const double xx = ux * Qx, yy = uy * Qy;        // Pi_xx / 36 = u_x (P_x + h_x) / 36
  const double xy = fma(ux, Py, uy * hx);         // Pi_xy / 36
  const double zz = a.zz_scale * fma(gx, gx, gy * gy);
  constexpr double s36 = 1.0 / 36.0;
  double p7 = 0.0, p8 = 0.0;
  if (kShear) {
    // rows 7, 8: m* = m_eq + S/2 + (1 - omega)(m + S/2 - m_eq), the brackets
    // A7 = m7 - u_x (j_x - h_x) + u_y (j_y - h_y), A8 = m8 - u_x j_y + u_y h_x
    const double om = fast_rcp(fma(a.tau_b, rho, a.tau_a));
    const double omc = 1.0 - om;
    const double A7 = fma(-ux, Kx, fma(uy, Ky, a.mom[3 * a.n + node] * s36));
    const double A8 = fma(-ux, jy, fma(uy, hx, a.mom[4 * a.n + node] * s36));
    p7 = omc * A7;
    p8 = omc * A8;
  }
  fx::reduced_populations<kShear>(rho * s36, xx, yy, xy, Px * s36, Py * s36, zz, p7, p8, out.f);
}

// General MRT collision in moment space (six relaxation times). With ST the
// surface-tension source C_k = l_k D_k enters as the shift D of m_eq in rows 1, 2,
// 7, 8 (+1.5 tr Q, -1.5 tr Q, -(Q_xx - Q_yy), -Q_xy), since m - l (m - m_eq - D) =
// m - l (m - m_eq) + l D.
template <bool ST = false>
__device__ __forceinline__ void collide_full(const StepArgs& a, int64_t node, double psi0, double gx, double gy,
                                             const SurfQ& sq, Post& out, double* rho_o, double* ux_o,
                                             double* uy_o) {
  const int64_t N = a.n;
  double m[9];
  m[0] = a.mom[node];
  m[3] = a.mom[N + node];
  m[5] = a.mom[2 * N + node];
  m[1] = a.mom[3 * N + node];
  m[2] = a.mom[4 * N + node];
  m[4] = a.mom[5 * N + node];
  m[6] = a.mom[6 * N + node];
  m[7] = a.mom[7 * N + node];
  m[8] = a.mom[8 * N + node];
  const double rho = m[0];
  const double cF = 2.0 * a.half_force * psi0;
  const double Fx = cF * gx, Fy = cF * gy;
  const double Jx = fma(0.5, Fx, m[3]), Jy = fma(0.5, Fy, m[5]);
  const double inv_rho = fast_rcp(rho);
  const double ux = Jx * inv_rho, uy = Jy * inv_rho;
  *rho_o = rho;
  *ux_o = ux;
  *uy_o = uy;
  const double ru2 = fma(ux, Jx, uy * Jy);
  const double uF = fma(ux, Fx, uy * Fy);
  const double F2p = a.G * a.G * (1.0 / 144.0) * fma(gx, gx, gy * gy);  // |F|^2 / psi^2
  double meq[9], S[9];
  meq[0] = rho;                   S[0] = 0.0;
  meq[1] = fma(3.0, ru2, -2.0 * rho); S[1] = fma(6.0, uF, a.li_e * F2p);
  meq[2] = fma(-3.0, ru2, rho);   S[2] = -fma(6.0, uF, a.li_z * F2p);
  meq[3] = Jx;                    S[3] = Fx;
  meq[4] = -Jx;                   S[4] = -Fx;
  meq[5] = Jy;                    S[5] = Fy;
  meq[6] = -Jy;                   S[6] = -Fy;
  meq[7] = fma(ux, Jx, -uy * Jy); S[7] = 2.0 * fma(ux, Fx, -uy * Fy);
  meq[8] = ux * Jy;               S[8] = fma(ux, Fy, uy * Fx);
  if (ST) {
    const double k36 = 36.0 * sq.k;  // 1.5 tr Q = 36 k t
    meq[1] = fma(k36, sq.t, meq[1]);
    meq[2] = fma(-k36, sq.t, meq[2]);
    meq[7] = fma(-4.0 * sq.k, sq.sd, meq[7]);
    meq[8] = fma(-sq.k, sq.xd, meq[8]);
  }
  double n[9];
  const double inv_norm[9] = {1.0 / 9.0, 1.0 / 36.0, 1.0 / 36.0, 1.0 / 6.0, 1.0 / 12.0,
                              1.0 / 6.0, 1.0 / 12.0, 1.0 / 4.0,  1.0 / 4.0};
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    const double om = a.omega[k];
    const double ms = fma(fma(-0.5, om, 1.0), S[k], fma(-om, m[k] - meq[k], m[k]));
    n[k] = ms * inv_norm[k];
  }
  // f* = M^T n (M^-1 = M^T diag(1/|row|^2))
  out.f[0] = n[0] - 4.0 * n[1] + 4.0 * n[2];
  const double A = n[0] - n[1] - 2.0 * n[2];
  const double X = n[3] - 2.0 * n[4], Y = n[5] - 2.0 * n[6];
  out.f[1] = A + X + n[7];
  out.f[3] = A - X + n[7];
  out.f[2] = A + Y - n[7];
  out.f[4] = A - Y - n[7];
  const double B = n[0] + 2.0 * n[1] + n[2];
  const double Px = n[3] + n[4], Py = n[5] + n[6];
  const double bp = B + n[8], bm = B - n[8];
  out.f[5] = bp + (Px + Py);
  out.f[7] = bp - (Px + Py);
  out.f[6] = bm + (Py - Px);
  out.f[8] = bm - (Py - Px);
}

// Where node (x, y)'s neighbours lie: the columns east and west (periodic), the offsets
// of its row and of the rows north and south (periodic, or the node's own row where a
// wall lies beyond: up, down). 32-bit, since 9 nx ny < 2^31.
struct Place {
  int x, xe, xw, r, rn, rs;
  bool up, down;
};

__device__ __forceinline__ Place place_of(const StepArgs& a, int x, int y) {
  Place p;
  const int nx = a.nx, ny = a.ny;
  p.x = x;
  p.xe = x + 1 == nx ? 0 : x + 1;
  p.xw = (x == 0 ? nx : x) - 1;
  const bool top = y + 1 == ny, bottom = y == 0;
  p.up = a.walls && top;
  p.down = a.walls && bottom;
  p.r = y * nx;
  p.rn = p.up ? p.r : top ? 0 : p.r + nx;
  p.rs = p.down ? p.r : (bottom ? ny * nx : p.r) - nx;
  return p;
}

// psi at the node and its eight neighbours (C, E, W, N, S, NE, NW, SW, SE) by bit pattern,
// wall ghosts beyond the walls. Loaded from global memory through L1, which neighbouring
// nodes' stencils share: a shared-memory tile with its halo arithmetic and barrier cost 150
// instructions per node more than these loads.
__device__ __forceinline__ void load_psi(const StepArgs& a, const Place& p, fx::u64 (&v)[9]) {
  const unsigned long long* psi = reinterpret_cast<const unsigned long long*>(a.psi);
  v[0] = psi[p.r + p.x];
  v[1] = psi[p.r + p.xe];
  v[2] = psi[p.r + p.xw];
  v[3] = psi[p.rn + p.x];
  v[4] = psi[p.rs + p.x];
  v[5] = psi[p.rn + p.xe];
  v[6] = psi[p.rn + p.xw];
  v[7] = psi[p.rs + p.xw];
  v[8] = psi[p.rs + p.xe];
  if (p.up) v[3] = v[5] = v[6] = fx::bits_of(a.psi_ghost_top);
  if (p.down) v[4] = v[7] = v[8] = fx::bits_of(a.psi_ghost_bottom);
}

// The collision of a node outside the domain of the fixed-point path (collide_fixed.cuh):
// force sums, then the general forms above. Out of line: inlined it would set the kernels'
// register count. 2 to 3 % of a droplet's nodes take it, those on the steep side of the
// interface, where the Li term leaves its frame (192^2, T_r = 0.6: 20 % of the rows of 32 have
// one at every step; two-phase 128^2 at T_r = 0.35: 8 to 11 % and 45 to 49 %).
template <int KIND, bool ST>
__device__ __noinline__ void collide_general(const StepArgs& a, int x, int y, Post* out) {
  const Place pl = place_of(a, x, y);
  fx::u64 v[9];
  load_psi(a, pl, v);
  double p[9];
  for (int k = 0; k < 9; ++k) p[k] = fx::double_of(v[k]);
  double gx, gy;
  fx::shan_chen_stencil(p[1], p[2], p[3], p[4], p[5], p[6], p[7], p[8], &gx, &gy);
  const int64_t N = a.n, node = pl.r + x;
  const double rho = a.mom[node], jx = a.mom[N + node], jy = a.mom[2 * N + node];
  if (KIND == kFullMrt) {
    double r, ux, uy;
    SurfQ sq = {0.0, 0.0, 0.0, 0.0};
    if (ST) sq = surface_q(a, p[0], p[1], p[2], p[3], p[4], p[5], p[6], p[7], p[8]);
    collide_full<ST>(a, node, p[0], gx, gy, sq, *out, &r, &ux, &uy);
  } else if (ST) {
    double ux, uy;
    const SurfQ sq = surface_q(a, p[0], p[1], p[2], p[3], p[4], p[5], p[6], p[7], p[8]);
    collide_reduced<KIND, ST>(a, node, rho, jx, jy, p[0], gx, gy, sq, *out, &ux, &uy);
  } else {
    collide_reduced_fx<KIND>(a, node, rho, jx, jy, p[0], gx, gy, *out);
  }
}

// Populations of collide_fixed that are rounded to double by the FP64 pipe's conversion
// rather than in integer code: the two pipes work side by side. On 12.9 M nodes with unit
// relaxation times 4 take 0.389 ms, 6 0.383, 7 0.386, 8 0.387 and 9 0.389.
constexpr int kFp64Conversions = 6;

template <int KIND, bool ST>
__device__ __forceinline__ void collide_fast(const StepArgs& a, const Place& pl, int y, const fx::u64 (&psi)[9],
                                             Post& out) {
  const int N = (int)a.n, node = pl.r + pl.x;
  constexpr int kMore = KIND == kUnitTau ? 0 : KIND == kShearTau ? 2 : 6;  // planes beside rho and j
  double m[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
#pragma unroll
  for (int k = 0; k < kMore; ++k) m[k] = a.mom[(3 + k) * N + node];
  if (!fx::collide_fixed<KIND, ST, kFp64Conversions>(a.fix, psi, a.mom[node], a.mom[N + node], a.mom[2 * N + node], m,
                                                     out.f)) {
    Post g;
    collide_general<KIND, ST>(a, pl.x, y, &g);
    out = g;
  }
}
static_assert(kUnitTau == fx::kFixUnit && kShearTau == fx::kFixShear && kFullMrt == fx::kFixMrt, "collision forms");

// K2 body for node (x, y): force, collision (with the surface-tension source when ST),
// then push streaming (or the macroscopic fields when FIELDS, which the source does not
// change).
template <int KIND, bool FIELDS, bool ST = false>
__device__ __forceinline__ void collide_node(const StepArgs& a, int x, int y, double* rho_o, double* ux_o,
                                             double* uy_o, double* psi_o) {
  const Place pl = place_of(a, x, y);
  const int N = (int)a.n, node = pl.r + x;
  fx::u64 psi[9];
  load_psi(a, pl, psi);
  Post o;
  if (!FIELDS) {
    // (a kernel built with the source runs lattices without it, kappa = 0, in a batch:
    // they take the same arithmetic as in the kernel without the source)
    if (!ST || a.kappa_q == 0.0)
      collide_fast<KIND, false>(a, pl, y, psi, o);
    else
      collide_fast<KIND, ST>(a, pl, y, psi, o);
  } else {
    double p[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) p[k] = fx::double_of(psi[k]);
    // 12 * sum_i w(|c_i|^2) psi(x + c_i) c_i  (w = 1/3 axis, 1/12 diagonal): exact
    // integer sums in one fixed-point frame, rounded once (fixsum.cuh); psi > 0 is
    // normal and finite wherever the density pass left the error word clear
    double gx, gy;
    fx::shan_chen_stencil(p[1], p[2], p[3], p[4], p[5], p[6], p[7], p[8], &gx, &gy);
    double rho, ux, uy;
    const SurfQ sq = {0.0, 0.0, 0.0, 0.0};  // the fields do not depend on the source
    if (KIND == kFullMrt) {
      collide_full<false>(a, node, p[0], gx, gy, sq, o, &rho, &ux, &uy);
    } else {
      rho = a.mom[node];
      collide_reduced<KIND, false>(a, node, rho, a.mom[N + node], a.mom[2 * N + node], p[0], gx, gy, sq, o, &ux, &uy);
    }
    if (rho_o) rho_o[node] = rho;
    if (ux_o) ux_o[node] = ux;
    if (uy_o) uy_o[node] = uy;
    if (psi_o) psi_o[node] = p[0];
    return;
  }
  // push streaming: f_i(x + c_i, t + 1) = f*_i(x, t); bounce-back into the opposite
  // population of the same node when x + c_i lies in a wall
  double* __restrict__ out = a.f_out;
  out[node] = o.f[0];
  out[N + pl.r + pl.xe] = o.f[1];
  out[3 * N + pl.r + pl.xw] = o.f[3];
  if (pl.up) {
    out[4 * N + node] = o.f[2];
    out[7 * N + node] = o.f[5];
    out[8 * N + node] = o.f[6];
  } else {
    out[2 * N + pl.rn + x] = o.f[2];
    out[5 * N + pl.rn + pl.xe] = o.f[5];
    out[6 * N + pl.rn + pl.xw] = o.f[6];
  }
  if (pl.down) {
    out[2 * N + node] = o.f[4];
    out[5 * N + node] = o.f[7];
    out[6 * N + node] = o.f[8];
  } else {
    out[4 * N + pl.rs + x] = o.f[4];
    out[7 * N + pl.rs + pl.xw] = o.f[7];
    out[8 * N + pl.rs + pl.xe] = o.f[8];
  }
}

// ---- per-M-step guard (Sec. III.A convergence check, mass, stability) --------------

constexpr int kGuardQ = 4;  // mass, max |u|, bad-node count, sum |rho - rho'|

// psi at (x + dx, y + dy) for 0 <= x < nx, 0 <= y < ny, |dx|, |dy| <= 1
__device__ __forceinline__ double psi_near(const StepArgs& a, int x, int y, int dx, int dy) {
  const int gx = wrap_index(x + dx, a.nx);
  int gy = y + dy;
  if (a.walls) {
    if (gy < 0) return a.psi_ghost_bottom;
    if (gy >= a.ny) return a.psi_ghost_top;
  } else {
    gy = wrap_index(gy, a.ny);
  }
  return a.psi[(int64_t)gy * a.nx + gx];
}

// Guard terms of node i, read from the psi and moment planes a density pass has just
// written for the current state: adds rho to v[0], raises v[1] to |u| with
// u = (j + F/2)/rho the fluid velocity of Eq. Momentum (F of Eq. ShanChenForce, wall
// ghosts as in the collision pass), and, when snap_valid, adds |rho - rho'| to v[3]
// with rho' = snap[i] the density of the previous guard call (the numerator of the
// Sec. III.A criterion). A non-finite or non-positive density adds 1 to v[2] and
// nothing else. Refreshes snap[i] = rho. IEEE division and sqrt: not on the hot path.
__device__ __forceinline__ void guard_node(const StepArgs& a, int64_t i, double* snap, bool snap_valid,
                                           double v[kGuardQ]) {
  const int64_t n = a.n;
  const double rho = a.mom[i];
  if (!(rho > 0.0 && rho < 1e300)) {
    v[2] += 1.0;
  } else {
    const int y = (int)(i / a.nx), x = (int)(i - (int64_t)y * a.nx);
    // the collision pass's stencil sums, rounded here to doubles
    double gx, gy;
    fx::shan_chen_stencil(psi_near(a, x, y, 1, 0), psi_near(a, x, y, -1, 0), psi_near(a, x, y, 0, 1),
                          psi_near(a, x, y, 0, -1), psi_near(a, x, y, 1, 1), psi_near(a, x, y, -1, 1),
                          psi_near(a, x, y, -1, -1), psi_near(a, x, y, 1, -1), &gx, &gy);
    const double cH = a.half_force * a.psi[i];
    const double ux = (a.mom[n + i] + cH * gx) / rho, uy = (a.mom[2 * n + i] + cH * gy) / rho;
    v[0] += rho;
    v[1] = fmax(v[1], sqrt(ux * ux + uy * uy));
    if (snap_valid) v[3] += fabs(rho - snap[i]);
  }
  snap[i] = rho;
}

// Fixed-order tree reduction of the guard terms over a block of `nthreads` (a power
// of two); s[q][0] holds the block's result.
template <int kNThreads>
__device__ __forceinline__ void guard_block_reduce(const double v[kGuardQ], double (*s)[kNThreads]) {
  for (int q = 0; q < kGuardQ; ++q) s[q][threadIdx.x] = v[q];
  __syncthreads();
  for (int w = kNThreads / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) {
      s[0][threadIdx.x] += s[0][threadIdx.x + w];
      s[1][threadIdx.x] = fmax(s[1][threadIdx.x], s[1][threadIdx.x + w]);
      s[2][threadIdx.x] += s[2][threadIdx.x + w];
      s[3][threadIdx.x] += s[3][threadIdx.x + w];
    }
    __syncthreads();
  }
}

}  // namespace pplbm
