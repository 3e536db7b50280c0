// Reverse mode of the fixed-point collision (collide_fixed.cuh) for unit relaxation times
// and the two-phase set, on the integer pipes.
//
// The nine adjoints mu_i of the populations become integers in one frame (units of
// 2^(el - 1086), headroom 10: every sum below stays under 2^63 with velocities under
// 0.875) with two places more, so the adjoints U of the populations' inputs
// (reduced_populations_transpose) are exact up to mu's rounding and are rounded once. Scaled
// by rho every factor between them and the adjoints of rho, j and h is a velocity, kept as
// u 2^63: with s = 1/36,
//   36 J_b  = U3 p_y + U1 q_x, U3 h_x + U2 q_y      (p = P/rho, q = Q/rho, h = F/(2 rho))
//   36 j_b  = J_b + U4 + U1 u_x, J_b + U5 + U3 u_x + U2 u_y
//   36 rho_b = U0 - J_b . u,  36 h_b = J_b + 2 P_b + 3 Q_b (+ U3 u_y),
// and for the two-phase set, with w = 1 - omega, A7 = m7 - u_x K_x + u_y K_y, A8 = m8 -
// u_x j_y + u_y h_x (K = j - h): m7_b = w U7, m8_b = w U8 through A7, A8 and
// 36 rho_b += (U7 A7 + U8 A8)/rho (omega - tau_a omega^2), as -rho d omega/d rho = omega -
// tau_a omega^2.
// A product of U and a velocity keeps it in U's units to 2 places, 2^-54 of the largest
// mu; the stored lambda's own rounding is 2^-53. mu itself needs an unbiased rounding: over a
// long rollout lambda's c . j_b grows beyond rho_b, and mu cut off towards zero at 2^-53 of the
// largest shrank rho_b: the gradient of 400 steps in the initial density had an rms error of
// 2.9e-13 of its rms against extended precision (two-phase 2.4e-13), 1.4e-14 (1.1e-14) so, and
// 4.3e-14 with rounded double-precision stages; of 100 steps 1.4e-14, 3.0e-15 and 1.0e-14. It costs
// 4 % of a gradient's step on 1024^2.
// Reports a node outside the domain (that of the forward, |u|, |h|, |K| below rho, the largest
// mu between 2^-700 and 2^400 or all nine zero), for which the caller runs the double-precision
// form.
//
// Compiles for the host too.
#pragma once

#include "collide_fixed.cuh"
#include "eos_fixed.cuh"

namespace pplbm {
namespace fx {

struct ReverseOut {
  double rho_b, jx_b, jy_b, m7_b, m8_b, psi_b, gx_b, gy_b, zs_b;
  double u6, u7, u8, om;  // the adjoints of zz and of the rows 7, 8 terms times 36 (for the
                          // surface-tension source), and omega (SRC)
  double t6, sd, xd;      // 6 t, sd, xd of the source's stencil sums (surface_q; SRC)
};

// how far n can be shifted left and stay below 2^62 in magnitude, so that its product keeps its bits
PPLBM_FX int spare_bits(i64 n) {
  const u64 a = (u64)(n < 0 ? ~n : n);
  const int z = clz64(a) - 2;
  return z > 0 ? z : 0;
}

template <bool SHEAR, bool SRC>
PPLBM_FX bool collide_reverse_fixed(const CollideFix& k, const u64 (&psi)[9], double rho, double jx, double jy,
                                    double m7, double m8, const double (&mu)[9], ReverseOut* o) {
  // forward: stencil sums, h, J and the velocities, as in collide_fixed
  u32 mx = max3(hi32(psi[1]), hi32(psi[2]), hi32(psi[3]));
  mx = max3(mx, hi32(psi[4]), hi32(psi[5]));
  mx = max3(mx, hi32(psi[6]), max3(hi32(psi[7]), hi32(psi[8]), hi32(psi[0])));  // (psi[0]: the source's sums)
  const int eg = frame_top(mx);
  auto at = [&](int i, int up) { return shr_u(significand(psi[i]), eg - up - (int)(hi32(psi[i]) >> 20)); };
  const u64 tE = at(1, 2), tW = at(2, 2), tN = at(3, 2), tS = at(4, 2);
  const u64 tNE = at(5, 0), tNW = at(6, 0), tSW = at(7, 0), tSE = at(8, 0);
  const u64 d1 = tNE - tSW, d2 = tSE - tNW;
  const i64 Gx = (i64)((tE - tW) + d1 + d2), Gy = (i64)((tN - tS) + d1 - d2);
  const u64 br = bits_of(rho);
  const int er = (int)(br >> 52), e0 = (int)(psi[0] >> 52);
  // rho between 2^-300 and 2^300, psi above 2^-200, so that no product's leaves the doubles' range
  bool ok = (u32)(er - 723) < 600u && mx < (1323u << 20) && mx >= (823u << 20) && (u32)(e0 - 823) < 500u;
  const u64 L = significand(br);
  const Factor psi0 = factor((i64)(significand(psi[0]) >> 1));
  const i64 a0 = mulhi(factor(k.ch.m), psi0);
  const Factor A = factor(a0), fGx = factor(Gx), fGy = factor(Gy);
  const int dh = er + 953 - k.ch.e - e0 - eg;
  const i64 hx = to_frame<4>(mulhi(A, fGx), dh, 0x08000000u, &ok);
  const i64 hy = to_frame<4>(mulhi(A, fGy), dh, 0x08000000u, &ok);
  const i64 Jx = scaled_term(bits_of(jx), er, 0, &ok) + hx, Jy = scaled_term(bits_of(jy), er, 0, &ok) + hy;
  ok = ok && in_range(Jx, 0x2D800000u) && in_range(Jy, 0x2D800000u);
  const Factor inv = factor(reciprocal<9>(L));
  // velocities times 2^60 below 0.9, then 2^63
  const i64 ux = mulhi(factor(Jx), inv), uy = mulhi(factor(Jy), inv);
  const i64 vx = mulhi(factor(hx), inv), vy = mulhi(factor(hy), inv);  // h / rho
  const i64 qx = ux + 2 * vx, qy = uy + 2 * vy, kx = ux - 2 * vx, ky = uy - 2 * vy;
  constexpr u32 kV = 0x0E000000u;  // 0.875 2^28
  ok = ok && in_range(ux, kV) && in_range(uy, kV) && in_range(qx, kV) && in_range(qy, kV) && in_range(vx, kV) &&
       in_range(vy, kV) && in_range(kx, kV) && in_range(ky, kV);
  auto q63 = [](i64 v) { return factor((i64)((u64)v << 3)); };
  const Factor fux = q63(ux), fuy = q63(uy), fvx = q63(vx), fqx = q63(qx), fqy = q63(qy), fpy = q63(uy + vy);

  // the adjoints of the populations' inputs, exact in one frame
  u64 b[9];
#pragma unroll
  for (int i = 0; i < 9; ++i) b[i] = bits_of(mu[i]);
  u32 mm = mag_hi(b[0]);
#pragma unroll
  for (int i = 1; i < 9; i += 2) mm = max3(mm, mag_hi(b[i]), mag_hi(b[i + 1]));
  // below 2^-700, and where zs_b, the smallest of the results, would leave the doubles' range,
  // the double-precision form keeps what this frame would drop (subnormals under 2^-1042, whose
  // upper words are zero, count as zero). A loss of one node has such adjoints far from it: of 300
  // steps back on 1024^2 half of them are below 2^-300.
  ok = ok && mm < (1423u << 20) && mm - 1u >= (323u << 20) - 1u;
  const int el = ((int)(mm >> 20) > 323 ? (int)(mm >> 20) : 323) + 10;
  ok = ok && (mm == 0u || el + 2 * eg >= 2236);  // 2^(kl + 2 eg - 2164) >= 2^-1014
  // mu and the sums of them carry two places more (72 2^56 < 2^63); what joins products is
  // rounded to whole units. mu is rounded to nearest, ties to even: half of the ties are
  // exact halves of doubles a few octaves below the largest (rho_b beside a large j_b)
  i64 t[9];
#pragma unroll
  for (int i = 0; i < 9; ++i) {
    const u64 m = shr_u(significand(b[i]), el - 4 - (int)(mag_hi(b[i]) >> 20));
    t[i] = with_sign((m + 1 + ((m >> 2) & 1ull)) >> 2, b[i]);
  }
  auto whole = [](i64 n) { return (n + 2) >> 2; };
  const i64 a13 = t[1] + t[3], a24 = t[2] + t[4], s57 = t[5] + t[7], s68 = t[6] + t[8];
  const i64 d57 = t[5] - t[7], d68 = t[6] - t[8], dg = s57 + s68;
  const i64 U0 = 16 * t[0] + 4 * (a13 + a24) + dg;  // with its two places
  const i64 U1 = whole(3 * dg - 24 * t[0] + 12 * a13 - 6 * a24), U2 = whole(3 * dg - 24 * t[0] - 6 * a13 + 12 * a24);
  const i64 U3 = whole(9 * (s57 - s68));
  const i64 U4 = whole(12 * (t[1] - t[3]) + 3 * (d57 - d68)), U5 = whole(12 * (t[2] - t[4]) + 3 * (d57 + d68));
  const i64 U6 = whole(a13 + a24 + dg - 8 * t[0]), U7 = whole(9 * (a13 - a24));
  // products with a velocity are in units of 2: doubled where they join whole ones
  const Factor f1 = factor(U1), f2 = factor(U2), f3 = factor(U3);
  i64 Jxb = 2 * (mulhi(f3, fpy) + mulhi(f1, fqx)), Jyb = 2 * (mulhi(f3, fvx) + mulhi(f2, fqy));
  const i64 Qxb = 2 * mulhi(f1, fux), Qyb = 2 * mulhi(f2, fuy);
  const i64 Pxb = U4, Pyb = U5 + 2 * mulhi(f3, fux);
  i64 hx0 = 2 * mulhi(f3, fuy), hy0 = 0, jy0 = 0, Kxb = 0, Kyb = 0, rb0 = 0;
  const int kl = el - 1086;
  // n / 36 in units of 2^(k - 4): times 16/36
  auto over36 = [&](i64 n, int k) { return frame_to_double(mulhi_k(factor((i64)kFourNinths), factor(n)), k - 4); };
  if (SHEAR) {
    const i64 w = one_minus_omega(k, L, er, &ok);
    ok = ok && in_range(w, 0x40000000u);
    const Factor fw = factor(w), f7 = factor(U7);
    // w U7, w U8 (w 2^62: the upper half is a quarter)
    const i64 B7 = mulhi(fw, f7) << 2, B8 = mulhi(fw, f3) << 2;
    const Factor g7 = factor(B7), g8 = factor(B8);
    // A7 / rho, A8 / rho times 2^60: m / rho from the scaled terms
    const i64 n7 = mulhi(factor(scaled_term(bits_of(m7), er, 0, &ok)), inv);
    const i64 n8 = mulhi(factor(scaled_term(bits_of(m8), er, 0, &ok)), inv);
    const Factor fkx = q63(kx), fky = q63(ky), fjy = q63(uy - vy);
    const i64 A7 = n7 - 2 * mulhi(fux, factor(kx)) + 2 * mulhi(fuy, factor(ky));
    const i64 A8 = n8 - 2 * mulhi(fux, factor(uy - vy)) + 2 * mulhi(fuy, factor(vx));
    ok = ok && in_range(A7, kV) && in_range(A8, kV);
    // rho d omega / d rho = -(omega - tau_a omega^2): omega 2^61, tau_a 2^58
    const i64 om = (1ll << 61) - (w >> 1);                       // omega 2^61, in (0, 2^62)
    const i64 ta = mulhi(factor(k.ta), factor(om)) << 3;          // tau_a omega 2^58
    ok = ok && in_range(ta, 0x10000000u);
    const i64 x = mulhi(factor(om), factor((1ll << 58) - ta)) << 3;  // (omega - tau_a omega^2) 2^58
    ok = ok && in_range(x, 0x08000000u);
    const i64 c = 2 * (mulhi(f7, q63(A7)) + mulhi(f3, q63(A8)));
    rb0 = mulhi(factor(x << 3), factor(c)) << 3;  // x 2^61
    Jxb -= 2 * (mulhi(g7, fkx) + mulhi(g8, fjy));
    Jyb += 2 * (mulhi(g7, fky) + mulhi(g8, fvx));
    Kxb = -2 * mulhi(g7, fux);
    Kyb = 2 * mulhi(g7, fuy);
    jy0 = -2 * mulhi(g8, fux);
    hx0 += 2 * mulhi(g8, fuy);
    o->m7_b = over36(B7, kl);
    o->m8_b = over36(B8, kl);
    if (SRC) o->om = frame_to_double(om, -61);
  }
  // 36 times the adjoints of rho, j, h
  const i64 Ru = rb0 - 2 * (mulhi(factor(Jxb), fux) + mulhi(factor(Jyb), fuy));
  ok = ok && in_range(Ru, 0x10000000u);  // with U0 < 36 2^56 below 2^63
  const i64 Xb = Jxb + Pxb + Qxb + Kxb, Yb = Jyb + Pyb + Qyb + Kyb + jy0;
  const i64 Hx = hx0 + Jxb + 2 * Pxb + 3 * Qxb - Kxb, Hy = hy0 + Jyb + 2 * Pyb + 3 * Qyb - Kyb;
  o->rho_b = over36(U0 + 4 * Ru, kl - 2);
  o->jx_b = over36(Xb, kl);
  o->jy_b = over36(Yb, kl);
  // through h = cH g: gx_b = cH/36 Hx + 2 zs U6 gx, psi_b = (hf/36) (Hx gx + Hy gy)
  const Factor fHx = factor(Hx), fHy = factor(Hy);
  const int n6 = spare_bits(U6);
  const Factor z6 = factor(mulhi(factor(k.zz.m), factor((i64)((u64)U6 << n6))));
  const int e1 = k.ch.e + e0 - 957, e2 = k.zz.e + eg - 957 - n6, em = e1 > e2 ? e1 : e2;
  // (k.zz.e is far below zero for zs = 0: its term is shifted out)
  o->gx_b = frame_to_double(shr_s(mulhi(fHx, A), em - e1) + shr_s(mulhi(z6, fGx), em - e2), kl + em);
  o->gy_b = frame_to_double(shr_s(mulhi(fHy, A), em - e1) + shr_s(mulhi(z6, fGy), em - e2), kl + em);
  const i64 hg = mulhi(fHx, fGx) + mulhi(fHy, fGy);
  const int nh = spare_bits(hg);
  o->psi_b = frame_to_double(mulhi(factor(k.ch.m), factor((i64)((u64)hg << nh))), kl + k.ch.e + eg - 958 - nh);
  const i64 g2 = mulhi(fGx, fGx) + mulhi(fGy, fGy);
  const int ng = spare_bits(g2);
  o->zs_b = frame_to_double(mulhi(factor((i64)((u64)U6 << n6)), factor((i64)((u64)g2 << ng))),
                            kl + 2 * eg - 2044 - n6 - ng);
  if (SRC) {
    const u64 sx = tE + tW, sy = tN + tS, dp = tNE + tSW, dm = tNW + tSE;  // sx, sy: 4 x the sums
    o->t6 = frame_to_double((i64)((sx >> 2) + (sy >> 2) + ((dp + dm) >> 1) - 6 * shr_u(significand(psi[0]), eg - e0)),
                            eg - 1086);
    o->sd = frame_to_double((i64)(sx - sy), eg - 1088);
    o->xd = frame_to_double((i64)(dp - dm), eg - 1086);
    o->u6 = frame_to_double(U6, kl);
    o->u7 = frame_to_double(U7, kl);
    o->u8 = frame_to_double(U3, kl);
  }
  return ok;
}

// d psi^2 / d rho on a C-S branch (psi2_fixed's psi^2 = rho x + k4) of the density with
// significand n and exponent er: with v = 1/(1 - eta), eta v^2 = v^2 - v, so
//   2^s (c1 (v^2 (3 v^2 - 2 v - 1) + 1/2) + 2 k2 rho + k3).
// Returns false outside eta < 1/2 (v <= 2: the polynomial stays below 32).
PPLBM_FX bool cs_slope_fixed(const EosFix& e, const CsFix& k, u64 n, int er, double* slope) {
  const int d = 1023 - er;
  if (!e.ok || d < 1 || d <= e.log2_b4) return false;
  const u64 rho63 = shr_u(n, d), eta = shr_u(n, d - e.log2_b4);
  const i64 v = reciprocal_q63((1ull << 63) - eta);  // v 2^61
  const i64 V = mulhi(factor(v), factor(v));         // v^2 2^58
  const i64 t = 3 * V - (v >> 2) - (1ll << 58);
  const i64 q = (mulhi(factor((i64)((u64)V << 2)), factor((i64)((u64)t << 2))) << 2) + (1ll << 57);  // 2^58
  const i64 D = mulhi(factor(k.c1), factor(q)) + mulhi(factor(k.k2), factor((i64)rho63)) + (e.k3_57 >> 1);
  *slope = frame_to_double(D, e.s - 56);
  return (eta >> 62) == 0;
}

// 1/(2 psi) of a positive normal psi
PPLBM_FX double half_reciprocal(u64 psi) {
  return frame_to_double(reciprocal<8>(significand(psi)), 960 - (int)(psi >> 52));
}

}  // namespace fx
}  // namespace pplbm
