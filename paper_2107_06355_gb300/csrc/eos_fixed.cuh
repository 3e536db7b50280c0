// psi(rho) of a node in fixed point (Sec. III.D shaped EOS, Eq. CS, Eq.
// InteractionPotential): the C-S branches, the ellipses and the cubic, and the square
// roots, on the integer pipes.
//
// Every branch gives psi^2 = P 2^ex with P a positive 64-bit integer, and one square root
// follows. With n the significand of rho (rho = n 2^(er - 1086), leading one at bit 63):
//  * C-S branches: psi^2 = rho x + k4 (eos_dev.cuh), x = c1 (v^3 - v + 1/2) + k2 rho + k3,
//    v = 1/(1 - eta). x is of order one, so it has an absolute frame (2^-57, scaled by a
//    power of two so that 1/2 <= k3 < 1), and rho x keeps rho's exponent: the vapour's
//    psi^2 has full relative precision. Domain: eta < 0.6 (v < 2.5).
//  * ellipses: psi^2 = k3 rho + A + B s, a s = sqrt((a - d)(a + d)), d = rho - rho0, and
//  * cubic: psi^2 = k3 rho + A + B t^2 (3 - 2 t), t = (rho - rho_max)/(rho_min - rho_max):
//    rho, rho0 and a in an absolute frame per branch (2^q), the sum in rho's own frame. The
//    error is a few units of 2^-59 rho and B 2^-58 / s; in double precision the latter is
//    B 2^-54 / s, tens of ulps of psi next to the vapour at T_r = 0.35, where B > rho.
// A branch or density outside these forms (the Peng loop inside, b that is not a power of
// two, eta >= 0.6, psi^2 not clearly positive) is reported and the caller evaluates
// eos_dev.cuh's forms on the FP64 pipe.
//
// What it measured is in step_device.cuh beside its use. Compiles for the host too.
#pragma once

#include "eos.cuh"
#include "fixmul.cuh"

namespace pplbm {

struct CsFix {
  fx::i64 c1;  // c1 2^(62 - s)
  fx::i64 k2;  // k2 2^(58 - s)
  fx::FixNum k4;  // k4 2^-s
};

struct LoopFix {
  fx::i64 rho0;     // rho0 2^q
  fx::i64 c;        // ellipses: a 2^q; cubic: 2^(126 - up - q) / (rho_min - rho_max)
  fx::FixNum A, B;  // A 2^-s, B 2^-s (ellipses: B/a 2^(62 - q - s))
  int q, up;
};

struct EosFix {
  int ok;        // 0: this EOS is evaluated on the FP64 pipe
  int s;         // psi^2 = 2^s (...): |k3| 2^-s in [1/2, 1)
  int log2_b4;   // eta = 2^log2_b4 rho
  int loop;      // 1: the shaped loop's branches are available (mode 1)
  fx::i64 k3_57, k3_60;  // k3 2^(57 - s), k3 2^(60 - s)
  CsFix cs[2];   // vapour, liquid
  LoopFix loops[3];  // ellipse 1, ellipse 3, cubic
};

namespace fx {

PPLBM_FX float rsqrt_seed32(float x) {
#ifdef __CUDA_ARCH__
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
#else
  return (float)(1.0 / std::sqrt((double)x));
#endif
}

PPLBM_FX float to_float(u32 x) {
#ifdef __CUDA_ARCH__
  return __uint2float_rn(x);
#else
  return (float)x;
#endif
}

PPLBM_FX float fma32(float a, float b, float c) {
#ifdef __CUDA_ARCH__
  return __fmaf_rn(a, b, c);
#else
  return (float)((double)a * b + c);
#endif
}

// 2^60 sqrt(N 2^-64), N in [2^62, 2^64): a 23-bit seed R 2^-22 of r = 1/sqrt(z) refined by
// the third-order step r (1 + e/2 + 3 e^2/8), e = 1 - z r^2 (|e| < 2^-20, first neglected
// term below 2^-62), then z r. Error below 3 units.
PPLBM_FX i64 sqrt60(u64 N) {
  const u32 nh = (u32)(N >> 32), nl = (u32)N;
  const float f = fma32(rsqrt_seed32(to_float(nh)), 65535.984375f, 2.0f);  // 2 + r (1 - 2^-22) < 4
  const u32 R = bits_of32(f) & 0x7FFFFFu;                                   // r 2^22
  const u64 R2 = mad_u(R, R, 0ull);
  const u32 rh = (u32)(R2 >> 32), rl = (u32)R2;
  // e 2^76 = 2^76 - (N R^2 2^-32) modulo 2^64
  const u64 q = mad_u(nh, rl, mad_u(nl, rh, mad_u(nl, rl, 0ull) >> 32)) + ((u64)(nh * rh) << 32);
  const i64 E = (i64)(0ull - q);
  const i32 eh = (i32)(E >> 32);
  const i64 C = (E >> 1) + (mad(eh, 3 * eh, 0) >> 15);
  const i64 c = mad((i32)R, (i32)(C >> 32), (i64)(mad_u(R, (u32)C, 0ull) >> 32)) >> 5;
  const i64 r1 = (i64)((u64)R << 39) + c;  // r 2^61
  return mulhi(factor((i64)(N >> 1)), factor(r1));
}

// The double nearest to sqrt(P 2^ex), P >= 2^32
PPLBM_FX double sqrt_double(i64 P, int ex) {
  const int lz = clz32((u32)((u64)P >> 32));  // >= 1
  const int sh = lz - ((lz + ex) & 1);        // ex - sh even
  const i64 s = sqrt60((u64)P << sh);         // [2^59, 2^60]
  const u64 m = ((u64)s + 0x3Full + (((u64)s >> 7) & 1ull)) >> 7;
  return double_of(m + ((u64)(((ex - sh) >> 1) + 1053) << 52));
}

// 1/om 2^61 for om = x 2^-63 in [0.4, 1]; relative error below 2^-59
PPLBM_FX i64 reciprocal_q63(u64 x) {
  // y + 8 as a float: its mantissa is y 2^20
  const float f = fma32(rcp_seed32(to_float((u32)(x >> 32))), 2147483648.0f, 8.0f);
  const u32 Y = bits_of32(f) & 0x7FFFFFu;
  // e 2^83 = 2^83 - x Y modulo 2^64 (|e| < 2^-20)
  const i64 E = (i64)(0ull - (mad_u((u32)x, Y, 0ull) + ((u64)((u32)(x >> 32) * Y) << 32)));
  const i32 eh = (i32)(E >> 32);
  const i64 T = E + (mad(eh, eh, 0) >> 19);
  const i64 c = mad((i32)Y, (i32)(T >> 32), (i64)(mad_u(Y, (u32)T, 0ull) >> 32)) >> 10;
  return (i64)((u64)Y << 41) + c;
}

}  // namespace fx

// psi^2 = P 2^ex of the density with significand n, exponent er and double rb (bits).
// Returns false outside the domain above.
PPLBM_FX bool psi2_fixed(const EosFix& e, const EosConst& c, fx::u64 n, int er, fx::i64 rb, fx::i64* P, int* ex) {
  using namespace fx;
  const bool vap = rb <= c.bits_rho_v, liq = rb >= c.bits_rho_l;
  if (c.mode == 0 || vap || liq) {
    const CsFix& k = e.cs[c.mode == 1 && vap ? 0 : 1];
    const int d = 1023 - er;
    const u64 rho63 = shr_u(n, d), eta = shr_u(n, d - e.log2_b4);
    bool ok = d >= 1 && d > e.log2_b4 && eta < 0x4CCCCCCC00000000ull;  // eta < 0.6
    const Factor v = factor(reciprocal_q63((1ull << 63) - eta));       // v 2^61
    const i64 w = (mulhi(v, v) - (1ll << 58)) << 2;                    // (v^2 - 1) 2^60
    const i64 q = (mulhi(v, factor(w)) + (1ll << 56)) << 2;            // (v (v^2 - 1) + 1/2) 2^59
    const i64 x = mulhi(factor(k.c1), factor(q)) + mulhi(factor(k.k2), factor((i64)rho63)) + e.k3_57;
    const int d4 = er - 1081 - k.k4.e;
    ok = ok && (x >> 59) == 0 && (k.k4.m == 0 || d4 >= 0);  // 0 <= x < 4
    *P = mulhi(factor((i64)(n >> 1)), factor((i64)((u64)x << 3))) + shr_s(k.k4.m, d4 < 0 ? 0 : d4);
    *ex = er - 1081 + e.s;
    return ok && (*P >> 32) > 0;
  }
  if (!e.loop) return false;
  const bool first = rb <= c.bits_rho_max, cubic = !first && rb < c.bits_rho_min;
  const LoopFix& L = e.loops[cubic ? 2 : first ? 0 : 1];
  const int dr = 1086 - er - L.q;
  const i64 rho = (i64)shr_u(n, dr);  // rho 2^q
  const i64 d = rho - L.rho0;
  const int dA = er - 1081 - L.A.e, dB = dA + L.A.e - L.B.e;
  bool ok = dr >= 1 && dA >= 0 && dB >= 0;
  i64 g;  // what B multiplies, times 2^60
  if (cubic) {
    const i64 t = (i64)((u64)mulhi(factor(d), factor(L.c)) << L.up);  // t 2^62
    const i64 t2 = mulhi(factor(t), factor(t));                       // t^2 2^60
    g = mulhi(factor((i64)((u64)t2 << 2)), factor(3 * (1ll << 60) - (t >> 1))) << 2;
  } else {
    const i64 w = mulhi(factor(L.c - d), factor(L.c + d));  // (a s)^2 2^(2 q - 64), at most 2^60
    ok = ok && (w >> 32) > 0;
    const int sh = clz32((u32)((u64)w >> 32)) & ~1;  // even, >= 2
    g = (i64)(((u64)sqrt60((u64)w << sh) << 1) >> ((sh >> 1) - 1));  // a s 2^(q - 2)
  }
  *P = mulhi(factor((i64)(n >> 1)), factor(e.k3_60)) + shr_s(L.A.m, dA) +
       shr_s((i64)((u64)mulhi(factor(L.B.m), factor(g)) << 4), dB);
  *ex = er - 1081 + e.s;
  return ok && (*P >> 32) > 0;
}

}  // namespace pplbm
