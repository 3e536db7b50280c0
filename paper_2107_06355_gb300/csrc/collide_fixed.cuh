// The collision of one node in fixed point, for unit relaxation times, for the two-phase
// set (rows 7, 8 relaxing at omega = 1/tau(rho)) and for six relaxation times, with or
// without the surface-tension source: from the psi stencil and the node's moments to the
// nine post-collision populations, on the integer pipes.
//
// What bounds it: the integer ALU pipe and instruction issue (ncu on 2048 x 1024, unit
// relaxation times: 665 instructions per node, the ALU pipe 70 % and the multiply-add
// pipe 58 % busy, FP64 27 %). With its products on the FP64 pipe and each sum rounded to a
// double in integer code the collision took 19 FP64 and about 1,020 integer ALU
// instructions per node; here nothing is rounded before the populations, so the
// normalise-and-round steps are gone except the nine of the result, and a product costs
// three 32 x 32 multiply-adds instead of an FP64 instruction worth 32. Collision pass of
// a batch of 12.9 M nodes: 0.783 ms before, 0.388 ms now; two-phase 2048 x 1024: 154 and
// 75 us; a step with six relaxation times, 1300 x 810: 362 and 84 us. Against
// quad precision the populations' rms error is 0.34 ulp (0.41 two-phase), where the rounded
// stages gave 0.64 (0.67).
//
// Frames. With L the significand of rho (rho = L 2^(er - 1086), leading one at bit 63),
// every quantity of the output stage is scaled by 1/36 as in fx::reduced_populations
// and kept in units of 2^(er - 1086): r = rho/36 lies in [2^57.8, 2^58.9), so the
// smallest population keeps at least 5 bits below its last place. Momenta (j, h = F/2,
// J = j + h, P = j + 2 h, Q = j + 3 h) carry 4 bits more (units of 2^(er - 1090)), and
// velocities U = u 2^60, so that the upper half of U Q is in the output's units. With
// |J|, |Q| (and K = j - h) below 0.8 2^e (2^e <= rho), |zz| below 2^58 and the rows
// 7, 8 corrections below 2^57, every population's sum stays below 2^63 in magnitude:
// f1 is the largest, (8 + 18 0.64 + 12 0.8) 2^57.83 + 9 2^57 + 2^58 < 2^62.99. A node outside these
// bounds is reported, and the caller runs the general collision: nodes on the steep side of an
// interface, where the Li term's product, before its shift, is 2^56 or more (to_frame asks for
// six free places even where it then shifts right), and also |u| of order one, a density out
// of the range of the frames, a population at or below zero, a constant that is not finite.
#pragma once

#include "fixmul.cuh"

namespace pplbm {
namespace fx {

// the step's constants as fixed-point factors, set by set_collision_args
struct CollideFix {
  FixNum ch;  // half_force / 36: h / 36 = ch psi(x) g
  FixNum zz;  // the Li term's scale
  FixNum kq;  // kappa_q / 36
  FixNum tb;  // tau = ta + tb rho
  i64 ta;     // ta 2^58
  // six relaxation times: rates times 2^61 of rows 1, 2, (4, 6), (7, 8), and the Li term's
  // scales of rows 1 and 2 with G^2 / (144 36)
  i64 we, wz, wq, wn;
  FixNum le, lz;
};

// the collision's form: unit relaxation times, the two-phase set, six relaxation times
constexpr int kFixUnit = 0, kFixShear = 1, kFixMrt = 2;

// significand of rho/36 and of 16/36 x: 2^64/36 and 2^64 4/9
constexpr u64 kInv36 = 0x071C71C71C71C71Cull;
constexpr u64 kFourNinths = 0x71C71C71C71C71C7ull;

// in_range(x, b): |x| < b 2^32 (by its upper word)
PPLBM_FX bool in_range(i64 x, u32 b) { return (u32)(i32)(x >> 32) + b < 2 * b; }

// A double of either sign times 4/9 in units of 2^(er - 1090 + down): truncated in
// magnitude. ok is cleared when its exponent exceeds er + down.
PPLBM_FX i64 scaled_term(u64 b, int er, int down, bool* ok) {
  const int d = er - exponent(b);
  *ok = *ok && d + down >= 0;
  const u64 m = shr_u(mulhi_u(significand(b), kFourNinths), d + down);  // zero: exponent 0, shifted out
  return with_sign(m, b);
}

// Upper half of x y shifted to the frame: (x y 2^-64 2^up) >> (d + up), up making room
// for a frame finer than the product's; ok is cleared if the product is too large for
// that or d + up is negative. up places must be free above b.
template <int UP>
PPLBM_FX i64 to_frame(i64 x, int d, u32 b, bool* ok) {
  *ok = *ok && in_range(x, b) && d + UP >= 0;
  return shr_s((i64)((u64)x << UP), d + UP);
}

// (1 - omega) 2^62, omega = 1/tau(rho), of the density L 2^(er - 1086); ok is cleared
// outside 1/2 <= tau < 16
PPLBM_FX i64 one_minus_omega(const CollideFix& k, u64 L, int er, bool* ok) {
  const int d = 963 - k.tb.e - er;
  const i64 tau = k.ta + shr_s(mulhi(factor(k.tb.m), factor((i64)(L >> 1))), d);  // tau 2^58
  const u32 th = (u32)((u64)tau >> 32);
  *ok = *ok && d >= 0 && th - 0x02000000u < 0x3E000000u;
  const int lz = clz32(th);                                      // 6 for tau in [1/2, 1), ..., 2
  const u64 r = (u64)reciprocal<8>((u64)tau << (lz & 31));       // 2^62 / m, tau = m 2^(5 - lz)
  return (i64)((1ull << 62) - ((r << 1) >> ((6 - lz) & 31)));
}

// psi: the node and its eight neighbours as bit patterns (C, E, W, N, S, NE, NW, SW, SE);
// m the stress moments m7, m8 (kFixShear) or rows 1, 2, 4, 6, 7, 8 of Eq. MatrixMRT
// (kFixMrt). Returns false, with f undefined, for a node outside the fixed-point path's
// domain. NFP64 of the nine populations are converted on the FP64 pipe, the others in
// integer code.
template <int FORM, bool ST, int NFP64>
PPLBM_FX bool collide_fixed(const CollideFix& k, const u64 (&psi)[9], double rho, double jx, double jy,
                            const double (&mom)[6], double (&f)[9]) {
  constexpr bool SHEAR = FORM == kFixShear;
  // Shan-Chen stencil sums in one frame (see shan_chen_stencil)
  // (the source's sums take the node itself in too)
  u32 mx = max3(hi32(psi[1]), hi32(psi[2]), ST ? hi32(psi[0]) : 0u);
#pragma unroll
  for (int i = 3; i < 9; i += 2) mx = max3(mx, hi32(psi[i]), hi32(psi[i + 1]));
  const int eg = frame_top(mx);
  auto at = [&](int i, int up) { return shr_u(significand(psi[i]), eg - up - (int)(hi32(psi[i]) >> 20)); };
  const u64 tE = at(1, 2), tW = at(2, 2), tN = at(3, 2), tS = at(4, 2);
  const u64 tNE = at(5, 0), tNW = at(6, 0), tSW = at(7, 0), tSE = at(8, 0);
  const u64 d1 = tNE - tSW, d2 = tSE - tNW;
  const i64 Gx = (i64)((tE - tW) + d1 + d2), Gy = (i64)((tN - tS) + d1 - d2);

  const u64 br = bits_of(rho);
  const int er = (int)(br >> 52), e0 = (int)(psi[0] >> 52);  // signs: er, e0 above 2047 fail the tests
  bool ok = (u32)(er - 256) < 1664u && mx < kFrameMaxHi && e0 < 0x7EF;
  const u64 L = significand(br);

  // h = ch psi0 g and zz = zz_scale |g|^2
  const Factor psi0 = factor((i64)(significand(psi[0]) >> 1));
  const Factor A = factor(mulhi(factor(k.ch.m), psi0));
  const Factor fGx = factor(Gx), fGy = factor(Gy);
  const int dh = er + 953 - k.ch.e - e0 - eg;
  const i64 hx = to_frame<4>(mulhi(A, fGx), dh, 0x08000000u, &ok);
  const i64 hy = to_frame<4>(mulhi(A, fGy), dh, 0x08000000u, &ok);
  const i64 g2 = mulhi(fGx, fGx) + mulhi(fGy, fGy);
  auto li_term = [&](const FixNum& c) {
    return to_frame<6>(mulhi(factor(c.m), factor(g2)), er + 958 - c.e - 2 * eg, 0x01000000u, &ok);
  };

  const i64 jX = scaled_term(bits_of(jx), er, 0, &ok), jY = scaled_term(bits_of(jy), er, 0, &ok);
  const i64 Jx = jX + hx, Jy = jY + hy;
  const i64 Px = Jx + hx, Py = Jy + hy;
  const i64 Qx = Px + hx, Qy = Py + hy;
  constexpr u32 kBound = 0x2D800000u;  // 0.8 (4/9) 2^31, rounded down
  ok = ok && in_range(Jx, kBound) && in_range(Jy, kBound) && in_range(Qx, kBound) && in_range(Qy, kBound);

  // velocities U = u 2^60 and the unit-tau second moments / 36
  const Factor inv = factor(reciprocal<9>(L));
  const i64 Ux = mulhi(factor(Jx), inv), Uy = mulhi(factor(Jy), inv);
  const Factor fUx = factor(Ux), fUy = factor(Uy), fPy = factor(Py), fhx = factor(hx);
  const i64 r = (i64)mulhi_u(L, kInv36);
  i64 n[9];
  if (FORM == kFixMrt) {
    // m* = m + S + omega (m_eq - m - S/2) in the units of the output, by rows: 3, 5 give P
    // whatever omega_j; 4, 6: m_eq - S/2 = -j
    const i64 Jxx = mulhi(fUx, factor(Jx)), Jyy = mulhi(fUy, factor(Jy)), Jxy = mulhi(fUx, factor(Jy));
    const i64 Hxx = mulhi(fUx, fhx), Hyy = mulhi(fUy, factor(hy)), Hxy = mulhi2(fUx, factor(hy), fUy, fhx);
    const i64 ru2 = 3 * (Jxx + Jyy), uF = 12 * (Hxx + Hyy);
    const i64 le = li_term(k.le), lz = li_term(k.lz);
    const i64 S1 = uF + le, S2 = -uF - lz, S7 = 4 * (Hxx - Hyy), S8 = 2 * Hxy;
    i64 e1 = ru2 - 2 * r, e2 = r - ru2, e7 = Jxx - Jyy, e8 = Jxy;
    if (ST) {
      // m_eq shifts by 1.5 tr Q, -1.5 tr Q, -(Q_xx - Q_yy), -Q_xy (see below for t6, sd, xd)
      const u64 tC = shr_u(significand(psi[0]), eg - e0);
      const u64 sx = tE + tW, sy = tN + tS, dp = tNE + tSW, dm = tNW + tSE;
      const Factor K = factor(mulhi(factor(k.kq.m), psi0));
      const int ds = er + 957 - k.kq.e - e0 - eg;
      const i64 t6 = (i64)((sx >> 2) + (sy >> 2) + ((dp + dm) >> 1) - 6 * tC);
      const i64 kt = 6 * to_frame<4>(mulhi(K, factor(t6)), ds, 0x08000000u, &ok);
      ok = ok && in_range(kt, 0x08000000u);
      e1 += kt;
      e2 -= kt;
      e7 -= to_frame<4>(mulhi(K, factor((i64)(sx - sy))), ds, 0x08000000u, &ok);
      e8 -= to_frame<4>(mulhi(K, factor((i64)(dp - dm))), ds, 0x08000000u, &ok);
    }
    auto relax = [&](i64 m, i64 S, i64 w, i64 x) {  // |x| < 2^59
      ok = ok && in_range(x, 0x08000000u);
      return m + S + mulhi(factor(w), factor((i64)((u64)x << 3)));
    };
    i64 M[6];
#pragma unroll
    for (int i = 0; i < 6; ++i) M[i] = scaled_term(bits_of(mom[i]), er, 4, &ok);
    ok = ok && in_range(M[0], 0x20000000u) && in_range(M[1], 0x20000000u) && in_range(S1, 0x10000000u);
    const i64 m1 = relax(M[0], S1, k.we, e1 - M[0] - (S1 >> 1)), m2 = relax(M[1], S2, k.wz, e2 - M[1] - (S2 >> 1));
    const i64 px = (Px + 8) >> 4, py = (Py + 8) >> 4;
    const i64 m4 = relax(M[2], -(hx >> 3), k.wq, -(jX >> 4) - M[2]);
    const i64 m6 = relax(M[3], -(hy >> 3), k.wq, -(jY >> 4) - M[3]);
    const i64 m7 = relax(M[4], S7, k.wn, e7 - M[4] - (S7 >> 1)), m8 = relax(M[5], S8, k.wn, e8 - M[5] - (S8 >> 1));
    ok = ok && in_range(m1, 0x10000000u) && in_range(m2, 0x10000000u) && in_range(m4, 0x02000000u) &&
         in_range(m6, 0x02000000u) && in_range(m7, 0x02000000u) && in_range(m8, 0x02000000u);
    // f = M^-1 m*, times 36: see collide_full
    const i64 A = 4 * r - m1 - 2 * m2, B = 4 * r + 2 * m1 + m2;
    const i64 a1 = A + 9 * m7, a2 = A - 9 * m7, bp = B + 9 * m8, bm = B - 9 * m8;
    const i64 X = 6 * (px - m4), Y = 6 * (py - m6), C = 6 * px + 3 * m4, D = 6 * py + 3 * m6;
    n[0] = r - m1 + m2;  // f0 / 4
    n[1] = a1 + X;
    n[3] = a1 - X;
    n[2] = a2 + Y;
    n[4] = a2 - Y;
    n[5] = bp + C + D;
    n[7] = bp - C - D;
    n[6] = bm + D - C;
    n[8] = bm - D + C;
  } else {
    i64 zz = li_term(k.zz);
    const i64 xx = mulhi(fUx, factor(Qx)), yy = mulhi(fUy, factor(Qy));
    i64 xy = mulhi2(fUx, fPy, fUy, fhx);
    i64 p7 = 0, w = 0;
    if (SHEAR) {
      w = one_minus_omega(k, L, er, &ok);
      // rows 7, 8: p = (1 - omega) A / 36, A7 = m7 - u_x (j_x - h_x) + u_y (j_y - h_y),
      // A8 = m8 - u_x j_y + u_y h_x
      const i64 Kx = jX - hx, Ky = jY - hy;
      ok = ok && in_range(Kx, kBound) && in_range(Ky, kBound) && in_range(w, 0x40000000u);
      const Factor nUx = factor(-Ux), fw = factor(w);
      const i64 A7 = scaled_term(bits_of(mom[0]), er, 4, &ok) + mulhi2(nUx, factor(Kx), fUy, factor(Ky));
      const i64 A8 = scaled_term(bits_of(mom[1]), er, 4, &ok) + mulhi2(nUx, factor(jY), fUy, fhx);
      ok = ok && in_range(A7, 0x10000000u) && in_range(A8, 0x10000000u);
      p7 = mulhi(fw, factor((i64)((u64)A7 << 2)));
      const i64 p8 = mulhi(fw, factor((i64)((u64)A8 << 2)));
      ok = ok && in_range(p8, 0x02000000u);
      xy += p8;
    }
    if (ST) {
      // zz += 6 k t6, p7 -= 4 omega k sd, p8 -= omega k xd with k = kappa_q psi0 / 36,
      // t6 = (axis sum) + (diagonal sum) / 2 - 6 psi0 (6 psi0 < 2^63), sd, xd as in surface_q
      const u64 tC = shr_u(significand(psi[0]), eg - e0);
      const u64 sx = tE + tW, sy = tN + tS, dp = tNE + tSW, dm = tNW + tSE;  // sx, sy: 4 x the sums
      const i64 t6 = (i64)((sx >> 2) + (sy >> 2) + ((dp + dm) >> 1) - 6 * tC);
      const i64 sd = (i64)(sx - sy), xd = (i64)(dp - dm);  // 4 sd
      const Factor K = factor(mulhi(factor(k.kq.m), psi0));
      const int ds = er + 957 - k.kq.e - e0 - eg;
      zz += 6 * to_frame<4>(mulhi(K, factor(t6)), ds, 0x08000000u, &ok);
      i64 q7 = to_frame<4>(mulhi(K, factor(sd)), ds, 0x08000000u, &ok);
      i64 q8 = to_frame<4>(mulhi(K, factor(xd)), ds, 0x08000000u, &ok);
      if (SHEAR) {  // omega = 1 - w 2^-62
        ok = ok && in_range(q7, 0x10000000u) && in_range(q8, 0x10000000u);
        const Factor fw = factor(w);
        q7 -= mulhi(fw, factor((i64)((u64)q7 << 2)));
        q8 -= mulhi(fw, factor((i64)((u64)q8 << 2)));
      }
      p7 -= q7;
      ok = ok && in_range(q8, 0x01000000u);
      xy -= q8;
    }
    if (SHEAR || ST) ok = ok && in_range(p7, 0x02000000u);
    ok = ok && in_range(zz, 0x04000000u);

    // the populations as small-integer combinations (reduced_populations); n0 is f0 / 4
    const i64 T3 = 3 * (xx + yy);
    const i64 E = 4 * r + zz - 2 * T3;
    const i64 a1 = E + 18 * xx + ((SHEAR || ST) ? 9 * p7 : 0), a2 = E + 18 * yy - ((SHEAR || ST) ? 9 * p7 : 0);
    const i64 px = (Px + 8) >> 4, py = (Py + 8) >> 4;
    const i64 B = r + T3 + zz;
    const i64 bq = B + 9 * xy, bm = 2 * B - bq;
    n[0] = E - 3 * zz;
    n[1] = a1 + 12 * px;
    n[3] = 2 * a1 - n[1];
    n[2] = a2 + 12 * py;
    n[4] = 2 * a2 - n[2];
    n[5] = bq + 3 * (px + py);
    n[7] = 2 * bq - n[5];
    n[6] = bm + 3 * (py - px);
    n[8] = 2 * bm - n[6];
  }
  // all nine positive with a bit above 2^32, so that they can be rounded in integer code
  i32 lo = (i32)(n[0] >> 32);
#pragma unroll
  for (int i = 1; i < 9; i += 2) lo = min3s(lo, (i32)(n[i] >> 32), (i32)(n[i + 1] >> 32));
  ok = ok && lo > 0;
  const int sh = er - 1086;
#pragma unroll
  for (int i = 0; i < 9; ++i)
    f[i] = scale2(i < NFP64 ? to_double_fp64(n[i]) : to_double_int(n[i]), i == 0 ? sh + 2 : sh);
  return ok;
}

}  // namespace fx
}  // namespace pplbm
