// Products, a reciprocal and the conversion back to double of 64-bit fixed-point
// numbers on the integer pipes, for the step's per-node arithmetic.
//
// GB300's SM issues 2 FP64 operations per clock, but 64 32-bit multiply-adds with a
// 64-bit sum (IMAD.WIDE) and beside them 64 integer ALU instructions. A product of two
// fixed-point numbers kept to its upper 64 bits is three IMAD.WIDE and two shifts, so
// it costs the time of a sixth of an FP64 instruction, and its error (below 3 units of
// the 64-bit result) is set by the frame it is in, not by 53 bits. Measured per SM and
// clock (dependent chains, 1,024 threads): fma.f64 2.0, mad.wide.u32 64, 64-bit shift
// 32, 64-bit add 43, clz 16, mul.hi.u64 8.
//
// A frame is a power of two that a set of integers share as their unit. Signed products
// drop the product of the two low halves; they are rounded so that their mean error is zero.
//
// The functions compile for the host as well, so that CPU tests can compare them with
// exact rational arithmetic.
#pragma once

#include "fixsum.cuh"

#ifdef __CUDACC__
#include <cuda_runtime.h>
#endif

namespace pplbm {
namespace fx {

typedef unsigned u32;
typedef int i32;

// x >> d for d >= 0, 0 (or the sign) from d = 64 on
PPLBM_FX u64 shr_u(u64 x, int d) {
#ifdef __CUDA_ARCH__
  u64 r;
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(d));
  return r;
#else
  return d > 63 ? 0ull : x >> d;
#endif
}

PPLBM_FX i64 shr_s(i64 x, int d) {
#ifdef __CUDA_ARCH__
  i64 r;
  asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(d));
  return r;
#else
  return x >> (d > 63 ? 63 : d);
#endif
}

PPLBM_FX int clz32(u32 v) {
#ifdef __CUDA_ARCH__
  return __clz((int)v);
#else
  return v ? __builtin_clz(v) : 32;
#endif
}

// three-operand extrema, one instruction each (with pairs of comparisons and selects the
// density pass of 12.9 M nodes took 0.300 ms, 0.282 so; the collision 0.400 and 0.389)
PPLBM_FX u32 max3(u32 a, u32 b, u32 c) {
#ifdef __CUDA_ARCH__
  return __vimax3_u32(a, b, c);
#else
  return a > b ? (a > c ? a : c) : (b > c ? b : c);
#endif
}

PPLBM_FX u32 min3(u32 a, u32 b, u32 c) {
#ifdef __CUDA_ARCH__
  return __vimin3_u32(a, b, c);
#else
  return a < b ? (a < c ? a : c) : (b < c ? b : c);
#endif
}

PPLBM_FX i32 min3s(i32 a, i32 b, i32 c) {
#ifdef __CUDA_ARCH__
  return __vimin3_s32(a, b, c);
#else
  return a < b ? (a < c ? a : c) : (b < c ? b : c);
#endif
}

// A signed factor of products, its low half shifted down by one so that all partial
// products are signed 32 x 32.
struct Factor {
  i32 hi, lo;  // x >> 32, (x & (2^32 - 1)) >> 1
};

PPLBM_FX Factor factor(i64 x) { return Factor{(i32)(x >> 32), (i32)((u32)x >> 1)}; }

// a b + c by one multiply-add. (Through the PTX instruction: a product of a sign- and a
// zero-extended half written in C++ becomes a 64 x 64 multiplication.)
PPLBM_FX i64 mad(i32 a, i32 b, i64 c) {
#ifdef __CUDA_ARCH__
  i64 r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
#else
  return (i64)a * b + c;
#endif
}

PPLBM_FX u64 mad_u(u32 a, u32 b, u64 c) {
#ifdef __CUDA_ARCH__
  u64 r;
  asm("mad.wide.u32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
#else
  return (u64)a * b + c;
#endif
}

// Upper 64 bits of x y; error below 2 units and 0 on average: the middle sum's addend, 0.75
// units, stands for half a unit of its shift and the dropped product of the low halves (1/4).
// Rounded down, every product was 3/4 unit low, the force in units of up to 2^-60 rho in both
// components: a droplet at rest gained a momentum of -6e-19 rho per step along (-1, -1), which
// after 10^6 steps would have moved it by 0.3 nodes; it is a random walk of 1e-18 now. The
// addend costs 1 to 2 % of a pass on large lattices. A factor of zero gives exactly zero.
PPLBM_FX i64 mulhi(Factor x, Factor y) {
  const i64 m = mad(x.hi, y.lo, mad(y.hi, x.lo, 0x60000000));
  return mad(x.hi, y.hi, m >> 31);
}

// Upper 64 bits of k x for a constant k: the product of the low halves has the mean lo/2 units of
// k's low half instead of 1/4, which would leave up to 1/4 unit in every result. (x's lowest
// bit, which a factor drops, counts for hi/4 on average where it is not empty; the
// finite-difference update's factors are shifted up or come from doubles.)
PPLBM_FX i64 mulhi_k(Factor k, Factor x) {
  const i64 m = mad(k.hi, x.lo, mad(x.hi, k.lo, (1 << 30) + (k.lo >> 1)));
  return mad(k.hi, x.hi, m >> 31);
}

// Upper 64 bits of x y + z w (the middle partial sums of both below 2^63 in magnitude:
// factors below 2^62); error below 4 units, on average none.
PPLBM_FX i64 mulhi2(Factor x, Factor y, Factor z, Factor w) {
  const i64 m = mad(x.hi, y.lo, mad(y.hi, x.lo, mad(z.hi, w.lo, mad(w.hi, z.lo, 0x7FFFFFFF))));
  return mad(x.hi, y.hi, mad(z.hi, w.hi, m >> 31));
}

// upper 64 bits of the unsigned product x y; error below 2 units
PPLBM_FX u64 mulhi_u(u64 x, u64 y) {
  const u32 xh = (u32)(x >> 32), xl = (u32)x, yh = (u32)(y >> 32), yl = (u32)y;
  const u64 m = (mad_u(xh, yl, 0ull) >> 32) + (mad_u(xl, yh, 0xFFFFFFFFull) >> 32);
  return mad_u(xh, yh, m);
}

// significand of a normal double with its leading one at bit 63: |x| = L 2^(e - 1086)
PPLBM_FX u64 significand(u64 b) { return (b << 11) | (1ull << 63); }

PPLBM_FX int exponent(u64 b) { return (int)((u32)(b >> 52) & 0x7FFu); }

PPLBM_FX i64 with_sign(u64 mag, u64 b) {
  const u64 neg = (u64)((i64)b >> 63);
  return (i64)((mag ^ neg) - neg);
}

// y0 ~ 1/x for x in [1, 2), about 23 correct bits
PPLBM_FX float rcp_seed32(float x) {
#ifdef __CUDA_ARCH__
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
#else
  return 1.0f / x;
#endif
}

PPLBM_FX float float_of(u32 b) {
#ifdef __CUDA_ARCH__
  return __uint_as_float(b);
#else
  float f;
  std::memcpy(&f, &b, 4);
  return f;
#endif
}

PPLBM_FX u32 bits_of32(float f) {
#ifdef __CUDA_ARCH__
  return __float_as_uint(f);
#else
  u32 b;
  std::memcpy(&b, &f, 4);
  return b;
#endif
}

// MUL 2^59 / m, MUL <= 9, for m = L 2^-63 in [1, 2) given by a significand L whose three
// lowest bits are zero (a double's eleven are): relative error below 2^-60. A 23-bit
// seed Y 2^-23 is refined by the third-order step 1/m = y (1 + e + e^2 + ...),
// e = 1 - m y, whose first neglected term is below 2^-62.
template <int MUL>
PPLBM_FX i64 reciprocal(u64 L) {
  const u32 lh = (u32)(L >> 32);
  const float m = float_of(((lh >> 8) & 0x7FFFFFu) | 0x3F800000u);  // truncated to 24 bits
  // y in (1/2, 1) as 1 + y (1 - 2^-22), whose float mantissa is y 2^23 (y = 1 stays below 1)
#ifdef __CUDA_ARCH__
  const float f = __fmaf_rn(rcp_seed32(m), 0x1.fffff8p-1f, 1.0f);
#else
  const float f = (float)((double)rcp_seed32(m) * 0x1.fffff8p-1 + 1.0);
#endif
  const u32 Y = bits_of32(f) & 0x7FFFFFu;
  const u64 X = L >> 3;  // m 2^60
  // e 2^83 = 2^83 - X Y, which fits 64 bits signed (|e| < 2^-20.9): the product modulo 2^64
  const i64 E = (i64)(0ull - (mad_u((u32)X, Y, 0ull) + ((u64)((u32)(X >> 32) * Y) << 32)));
  const i32 eh = (i32)(E >> 32);
  const i64 T = E + (mad(eh, eh, 0) >> 19);  // (e + e^2) 2^83
  const u32 M = MUL * Y;                     // below 2^27
  // M T 2^-47, the correction to M 2^36
  const i64 c = mad((i32)M, (i32)(T >> 32), (i64)(mad_u(M, (u32)T, 0ull) >> 32)) >> 15;
  return (i64)((u64)M << 36) + c;
}

// n as a double, rounded to nearest, ties to even. The integer version needs n >= 2^32
// and stays off the FP64 pipe (12 instructions against one of the FP64 pipe's 64-bit
// conversions, which takes the time of 32 integer instructions).
PPLBM_FX u64 to_double_int(i64 n) {
  const int s = clz32((u32)((u64)n >> 32)) - 1;  // 0 .. 30
  u64 v = (u64)n << s;                           // leading one at bit 62
  v += 0x1FFull + ((v >> 10) & 1ull);
  return (v >> 10) + ((u64)(1084 - s) << 52);
}

PPLBM_FX u64 to_double_fp64(i64 n) {
#ifdef __CUDA_ARCH__
  return bits_of(__ll2double_rn(n));
#else
  return bits_of((double)n);
#endif
}

// adds k to the exponent field of the double with bit pattern b
PPLBM_FX double scale2(u64 b, int k) { return double_of(b + ((u64)(u32)(k << 20) << 32)); }

// n 2^k as a double (normal or zero), on the FP64 pipe
PPLBM_FX double frame_to_double(i64 n, int k) {
  const u64 b = to_double_fp64(n);
  return scale2(b, hi32(b) ? k : 0);
}

// A constant of the step as a signed 63-bit factor: x = m 2^e, 2^62 <= |m| < 2^63 (0 for 0).
struct FixNum {
  i64 m;
  int e;
  int pad;
};

}  // namespace fx
}  // namespace pplbm
