// Finite-difference (MacCormack) solver of the macroscopic equations the method
// recovers (App. A), periodic grids, FP64.
//
//   d_t rho = -(rho d_g u_g + u_g d_g rho)
//   d_t u_a = -u_g d_g u_a - d_a p_EOS / rho - d_b p'_ab / rho + d_b sigma'_ab / rho
// with sigma' of Eq. StressTensor expanded as Eq. FDstressTensor (mu = rho/3
// (tau_nu - 1/2), mu_B = rho/3 (tau_e - tau_nu), Eq. DynamicViscosity; gradients
// via dmu/drho, Eq. FDviscosityDerivative) and d_b p'_ab of Eq. FDforce
//   -eps (G/4)(d_g psi)(d_a d_g psi) + (G/12)(d_a psi) lap psi + (G/6)(d_g psi)(d_a d_g psi)
//   + (G/4) psi d_a lap psi          (c = 1),
// plus, with the surface-tension control of Sec. V's technique (kappa), the
// divergence of its second-order pressure tensor (kappa G/6) psi (delta lap psi -
// d_a d_b psi): (kappa G/6) [(d_a psi) lap psi - (d_g psi)(d_a d_g psi)], which only
// changes the coefficients of the first and third terms above.
// Predictor: first derivatives of rho, u, p_EOS and rho in the viscous terms are
// forward differences; corrector: backward; second derivatives central; every
// derivative of psi central (the third derivative through lap psi at +-1).
// One MacCormack step = EOS pass (psi, p of U) + predictor pass (U* = U + dt R_f(U))
// + EOS pass (of U*) + corrector pass (U <- (U + U* + dt R_b(U*)) / 2, in place:
// the corrector reads U only at its own node).
// x is periodic; y is periodic or bounded by the wall layers of the grid-dependency
// appendix (Eqs. B1, B2): every plane then carries two ghost rows below and above
// the fluid rows, which a boundary pass fills after each EOS pass.
#include <cuda_runtime.h>

#include <cmath>
#include <cstring>
#include <initializer_list>
#include <new>
#include <string>

#include "../../include/pplbm.h"
#include "dependent_launch.cuh"
#include "eos_dev.cuh"
#include "eos_fixed.cuh"
#include "fixsum.cuh"
#include "fp64.cuh"
#include "internal.h"

namespace pplbm {
namespace {

struct FDArgs {
  const double* rho;  // source state of the RHS (U for the predictor, U* for the corrector)
  const double* ux;
  const double* uy;
  const double* psi;  // psi(rho), p_EOS(rho) of the source state
  const double* p;
  const double* rho0;  // corrector: U^n
  const double* ux0;
  const double* uy0;
  double* orho;  // output state
  double* oux;
  double* ouy;
  int nx, ny;
  int walls;  // 1: planes hold ghost rows (fluid row y at row y + 2), y not periodic
  // Every derivative is formed from raw stencil differences; the powers of
  // h = 1/dx, the time step and the force and viscosity coefficients are folded
  // into these constants on the host (mu = mu_c rho, mu_B = muB_c rho):
  double cA;              // dt h: advection, mass flux, pressure gradient
  double kS, kL, kD;      // dt (h^3/2) (G/6 - eps G/4), dt (h^3/2) G/12, dt (h^3/2) G/4
  double v1, v2, v3, v4;  // dt h^2 mu_c, dt h^2 muB_c, dt h^2 (2 mu_c + muB_c), dt h^2 (mu_c + muB_c)/4
  // tau_nu(rho) = ta + tb rho (Eq. RelaxationTime) in the VV kernels: mu = dt h^2 rho (g0 + g1 rho),
  // mu_B = dt h^2 rho (e0 - g1 rho), and d/drho of both (Eq. FDviscosityDerivative)
  double g0, g1, e0;
};

// The same constants as fixed-point factors, those of one sum in one frame
struct FDFix {
  int ok;              // 0: a constant lies outside the frames (k_fd_update_general runs)
  int eF, ev, eA;
  fx::i64 kS4, kL, kD;      // kS / 4, kL, kD: m 2^eF, below 2^62
  fx::i64 v1, v2, v3, v4;   // m 2^ev (constant viscosities)
  fx::i64 g0, e0;           // m 2^ev (VV)
  fx::FixNum g1;            // VV
  fx::i64 cA;               // m 2^eA
};

struct FDKernelArgs {
  FDArgs a;
  FDFix k;
};

__device__ __noinline__ void fd_eos_double(const EosConst& e, double r, double* psi, double* p) {
  const double pr = eos_pressure(e, r);
  *p = pr;
  const double psi2 = e.psi2_scale * (pr - r * (1.0 / 3.0));
  *psi = psi2 > 0.0 ? fast_sqrt(psi2) : sqrt(psi2);  // IEEE result at 0, below 0 and NaN
}

struct FDEosArgs {
  EosConst eos;
  EosFix fix;
  fx::i64 half;  // |G|/2 2^(63 + fix.s), in (2^61, 2^63): p = rho/3 - |G|/2 psi^2
};

// psi and p of one density: in fixed point on the integer pipes (eos_fixed.cuh), p from
// psi^2 before its root; a density outside that domain in double precision. In double
// precision throughout (25 FP64 instructions per point) the pass was bound by the FP64
// pipe. (Plain pointers: the blocks are resident while the previous launch still writes rho.)
__global__ void __launch_bounds__(128) k_fd_eos(const __grid_constant__ FDEosArgs a, const double* rho, double* psi,
                                                double* p, int64_t n) {
  using namespace fx;
  begin_dependent();
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double r = rho[i];
  const u64 b = bits_of(r), L = significand(b);
  const int er = (int)(b >> 52);
  i64 P;
  int ex;
  if (a.fix.ok && (u32)(er - 256) < 1664u && psi2_fixed(a.fix, a.eos, L, er, (i64)b, &P, &ex)) {
    psi[i] = sqrt_double(P, ex);
    // both terms in units of 2^(er - 1081): rho/3 and |G|/2 psi^2 (P < 2^61)
    const i64 third = mulhi(factor((i64)(L >> 1)), factor(0x0555555555555555ll));
    p[i] = frame_to_double(third - mulhi(factor(a.half), factor((i64)((u64)P << 1))), er - 1081);
    return;
  }
  double s, q;
  fd_eos_double(a.eos, r, &s, &q);
  psi[i] = s;
  p[i] = q;
}

// Wall layers (Eqs. B1, B2), one thread per column of a padded plane set: b1 (row
// 1) on the bottom wall, no slip, density and psi extrapolated from the first two
// fluid rows, p of that density; b2 (row 0) in the solid, psi_b2 = psi_b1 + 2 dy
// (psi_l - psi_b1); top rows mirror the last fluid rows with the velocity
// reversed (reflexive layers t1 = row ny + 2, t2 = row ny + 3).
__global__ void __launch_bounds__(64) k_fd_walls(const __grid_constant__ EosConst e, double* rho, double* ux, double* uy, double* psi, double* p, int nx,
                           int ny, double two_dy, double psi_l) {
  begin_dependent();
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  if (x >= nx) return;
  auto at = [&](int row) { return (int64_t)row * nx + x; };
  const double rb1 = 2.0 * rho[at(2)] - rho[at(3)];
  const double sb1 = 2.0 * psi[at(2)] - psi[at(3)];
  const double pb1 = eos_pressure(e, rb1);
  rho[at(1)] = rb1;
  psi[at(1)] = sb1;
  p[at(1)] = pb1;
  ux[at(1)] = 0.0;
  uy[at(1)] = 0.0;
  rho[at(0)] = rb1;
  psi[at(0)] = fma(two_dy, psi_l - sb1, sb1);
  p[at(0)] = pb1;
  ux[at(0)] = 0.0;
  uy[at(0)] = 0.0;
  const int t1 = ny + 2, t2 = ny + 3, f1 = ny + 1, f2 = ny;
  rho[at(t1)] = rho[at(f1)];
  psi[at(t1)] = psi[at(f1)];
  p[at(t1)] = p[at(f1)];
  ux[at(t1)] = -ux[at(f1)];
  uy[at(t1)] = -uy[at(f1)];
  rho[at(t2)] = rho[at(f2)];
  psi[at(t2)] = psi[at(f2)];
  p[at(t2)] = p[at(f2)];
  ux[at(t2)] = 0.0;
  uy[at(t2)] = 0.0;
}

// Stencil differences as exact integer combinations in one fixed-point frame per
// field (fixsum.cuh), each rounded once: integer-pipe work in place of chains of
// software IEEE additions and FP64 fused multiply-adds.
using fx::u64;

// psi's raw differences at a point from the 13 values of its 5 x 5 cross and
// diagonals: central first differences Pd, second differences Pxx, Pyy, the mixed
// one q = Dxy / 4, the Laplacian Lc = Pxx + Pyy and the differences DL of the
// 5-point Laplacians at +-1 (their coefficients sum to 14 at most: headroom 5 + sign).
// A value out of the frames' range (non-finite, or at or above 2^1008) makes them all
// NaN.
struct PsiDiffs {
  double Pd0, Pd1, Pxx, Pyy, q, Lc, DL0, DL1;
};

__device__ __forceinline__ PsiDiffs psi_diffs(double c, double e, double w, double n, double s, double ne, double nw,
                                              double sw, double se, double ee, double ww, double nn, double ss) {
  const double v[13] = {c, e, w, n, s, ne, nw, sw, se, ee, ww, nn, ss};
  u64 b[13];
  unsigned mx = 0;
#pragma unroll
  for (int k = 0; k < 13; ++k) {
    b[k] = fx::bits_of(v[k]);
    mx = max(mx, fx::mag_hi(b[k]));
  }
  const int eg = (int)(mx >> 20) + 6;
  u64 t[13];
#pragma unroll
  for (int k = 0; k < 13; ++k) t[k] = (u64)fx::sterm(b[k], eg);
  const u64 tC = t[0], tE = t[1], tW = t[2], tN = t[3], tS = t[4], tNE = t[5], tNW = t[6], tSW = t[7], tSE = t[8];
  const u64 pd0 = tE - tW, pd1 = tN - tS;
  const u64 pxx = tE + tW - 2 * tC, pyy = tN + tS - 2 * tC;
  const u64 dxy = (tNE - tSE) - (tNW - tSW);
  const u64 dl0 = (t[9] - t[10]) + (tNE + tSE) - (tNW + tSW) - 4 * pd0;  // L5(1, 0) - L5(-1, 0)
  const u64 dl1 = (t[11] - t[12]) + (tNE + tNW) - (tSE + tSW) - 4 * pd1;  // L5(0, 1) - L5(0, -1)
  const bool bad = mx >= fx::kFrameMaxHi;
  auto out = [&](u64 x, int shift) {
    return fx::double_of(bad ? fx::kNaN : fx::round_frame_s((fx::i64)x, eg + shift));
  };
  PsiDiffs r;
  r.Pd0 = out(pd0, 0);
  r.Pd1 = out(pd1, 0);
  r.Pxx = out(pxx, 0);
  r.Pyy = out(pyy, 0);
  r.q = out(dxy, -2);
  r.Lc = out(pxx + pyy, 0);
  r.DL0 = out(dl0, 0);
  r.DL1 = out(dl1, 0);
  return r;
}

// a velocity component's raw differences from its 3 x 3 neighbourhood: the one-sided
// first differences along x and y (forward in the predictor, backward in the
// corrector) and the central Dxx, Dyy, Dxy (coefficients sum to 4: headroom 3 + sign)
struct VelDiffs {
  double D0, D1, xx, yy, xy;
};

template <bool PRED>
__device__ __forceinline__ VelDiffs vel_diffs(double c, double e, double w, double n, double s, double ne, double nw,
                                              double sw, double se) {
  const double v[9] = {c, e, w, n, s, ne, nw, sw, se};
  u64 b[9];
  unsigned mx = 0;
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    b[k] = fx::bits_of(v[k]);
    mx = max(mx, fx::mag_hi(b[k]));
  }
  const int eg = (int)(mx >> 20) + 4;
  u64 t[9];
#pragma unroll
  for (int k = 0; k < 9; ++k) t[k] = (u64)fx::sterm(b[k], eg);
  const u64 tC = t[0], tE = t[1], tW = t[2], tN = t[3], tS = t[4];
  const bool bad = mx >= fx::kFrameMaxHi;
  auto out = [&](u64 x) { return fx::double_of(bad ? fx::kNaN : fx::round_frame_s((fx::i64)x, eg)); };
  VelDiffs r;
  r.D0 = out(PRED ? tE - tC : tC - tW);
  r.D1 = out(PRED ? tN - tC : tC - tS);
  r.xx = out(tE + tW - 2 * tC);
  r.yy = out(tN + tS - 2 * tC);
  r.xy = out((t[5] - t[8]) - (t[6] - t[7]));
  return r;
}

// The update of point (x, y) with its products in double precision: PRED: predictor
// (forward differences) or corrector (backward); VV: tau_nu(rho) viscosities. Runs for the
// points outside the fixed-point path's domain (fd_update_fixed).
template <bool PRED, bool VV>
__device__ __noinline__ void fd_update_general(const FDArgs& a, int x, int y) {
  const int nx = a.nx, ny = a.ny;
  // periodic columns and row offsets of the 5 x 5 neighbourhood, wrapped once
  // (offsets reach +-2, so a grid of width 1 or 2 wraps twice)
  auto wrap = [](int v, int n) {
    if (v < 0) v += n;
    if (v < 0) v += n;
    if (v >= n) v -= n;
    if (v >= n) v -= n;
    return v;
  };
  int cx[5];
  int64_t ry[5];
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    cx[k] = wrap(x + k - 2, nx);
    ry[k] = (int64_t)(a.walls ? y + k : wrap(y + k - 2, ny)) * nx;  // walls: padded rows, no wrap
  }
  auto at = [&](const double* f, int dx, int dy) { return f[ry[dy + 2] + cx[dx + 2]]; };
  // one-sided first difference along x (axis 0) or y (axis 1) of rho and p: forward in
  // the predictor, backward in the corrector; true derivative = h D (integer pipe,
  // add_int: bitwise the FP64 add)
  auto D1 = [&](const double* f, int axis) {
    const double c = at(f, 0, 0);
    if (PRED) return axis == 0 ? sub_int(at(f, 1, 0), c) : sub_int(at(f, 0, 1), c);
    return axis == 0 ? sub_int(c, at(f, -1, 0)) : sub_int(c, at(f, 0, -1));
  };
  auto vel = [&](const double* f) {
    return vel_diffs<PRED>(at(f, 0, 0), at(f, 1, 0), at(f, -1, 0), at(f, 0, 1), at(f, 0, -1), at(f, 1, 1),
                           at(f, -1, 1), at(f, -1, -1), at(f, 1, -1));
  };
  const double rho = at(a.rho, 0, 0), ux = at(a.ux, 0, 0), uy = at(a.uy, 0, 0);
  // velocity differences: Du_ab = d_a u_b (one-sided), second differences central
  // (d_xx = h^2 Dxx, d_xy = (h^2/4) Dxy)
  const VelDiffs vx = vel(a.ux), vy = vel(a.uy);
  const double Du00 = vx.D0, Du01 = vy.D0, Du10 = vx.D1, Du11 = vy.D1;
  // mass: d_t rho = -(rho div u + u . grad rho)
  const double Dr0 = D1(a.rho, 0), Dr1 = D1(a.rho, 1);
  const double Dv = add_int(Du00, Du11), Sh = add_int(Du01, Du10);
  const double drho = -a.cA * fma(rho, Dv, fma(ux, Dr0, uy * Dr1));
  // psi: dpsi = (h/2) Pd, d_ab psi from Pxx, Pyy, q = Dxy/4, lap = h^2 Lc, and the
  // derivative of lap psi = (h^3/2) DL from the 5-point sums at +-1
  const double* ps = a.psi;
  const double psi = at(ps, 0, 0);
  const PsiDiffs pd = psi_diffs(psi, at(ps, 1, 0), at(ps, -1, 0), at(ps, 0, 1), at(ps, 0, -1), at(ps, 1, 1),
                                at(ps, -1, 1), at(ps, -1, -1), at(ps, 1, -1), at(ps, 2, 0), at(ps, -2, 0),
                                at(ps, 0, 2), at(ps, 0, -2));
  const double Pd0 = pd.Pd0, Pd1 = pd.Pd1, Pxx = pd.Pxx, Pyy = pd.Pyy, q = pd.q, Lc = pd.Lc;
  const double DL0 = pd.DL0, DL1 = pd.DL1;
  // d_b p'_ab (Eq. FDforce) = (h^3/2) [(G/6 - eps G/4) S_a + (G/12) Pd_a Lc + (G/4) psi DL_a],
  // S_a = sum_g Pd_g (d_a d_g psi in the same units)
  const double S0 = fma(Pd0, Pxx, q * Pd1), S1 = fma(Pd1, Pyy, q * Pd0);
  const double kDpsi = a.kD * psi;
  const double F0 = fma(a.kS, S0, fma(a.kL * Pd0, Lc, kDpsi * DL0));
  const double F1 = fma(a.kS, S1, fma(a.kL * Pd1, Lc, kDpsi * DL1));
  // d_b sigma'_ab (Eqs. FDstressTensor, FDviscosityDerivative) with one-sided grad rho, grad u
  // and central second derivatives of u
  const double U0xx = vx.xx, U0yy = vx.yy, U1xx = vy.xx, U1yy = vy.yy;
  const double U0xy = vx.xy, U1xy = vy.xy;
  double V0, V1;
  if (!VV) {
    V0 = fma(a.v1, fma(2.0 * Dr0, Du00, Dr1 * Sh),
             fma(a.v2 * Dr0, Dv, rho * fma(a.v3, U0xx, fma(a.v4, U1xy, a.v1 * U0yy))));
    V1 = fma(a.v1, fma(2.0 * Dr1, Du11, Dr0 * Sh),
             fma(a.v2 * Dr1, Dv, rho * fma(a.v3, U1yy, fma(a.v4, U0xy, a.v1 * U1xx))));
  } else {
    const double mu = rho * fma(a.g1, rho, a.g0), muB = rho * fma(-a.g1, rho, a.e0);
    const double dmu = fma(2.0 * a.g1, rho, a.g0), dmuB = fma(-2.0 * a.g1, rho, a.e0);
    const double c2 = 2.0 * mu + muB, c4 = 0.25 * (mu + muB);
    V0 = fma(dmu, fma(2.0 * Dr0, Du00, Dr1 * Sh), fma(dmuB * Dr0, Dv, fma(c2, U0xx, fma(c4, U1xy, mu * U0yy))));
    V1 = fma(dmu, fma(2.0 * Dr1, Du11, Dr0 * Sh), fma(dmuB * Dr1, Dv, fma(c2, U1yy, fma(c4, U0xy, mu * U1xx))));
  }
  // dt d_t u_a = -dt u . grad u_a + (dt/rho)(d_b sigma'_ab - d_a p_EOS - d_b p'_ab)
  const double inv_rho = fast_rcp(rho);
  const double dux = fma(V0 - F0 - a.cA * D1(a.p, 0), inv_rho, -a.cA * fma(ux, Du00, uy * Du10));
  const double duy = fma(V1 - F1 - a.cA * D1(a.p, 1), inv_rho, -a.cA * fma(ux, Du01, uy * Du11));
  const int64_t i = (int64_t)(a.walls ? y + 2 : y) * nx + x;
  if (PRED) {
    a.orho[i] = rho + drho;
    a.oux[i] = ux + dux;
    a.ouy[i] = uy + duy;
  } else {
    a.orho[i] = 0.5 * (a.rho0[i] + (rho + drho));
    a.oux[i] = 0.5 * (a.ux0[i] + (ux + dux));
    a.ouy[i] = 0.5 * (a.uy0[i] + (uy + duy));
  }
}


// ---- the update in fixed point ------------------------------------------------------
//
// Every field's stencil values become integers in one frame (psi: 13 values, the two
// velocity components together: 18, unless their largest values are a factor of 2^7 or more
// apart; rho and p: 3 each), so differences are exact, and the
// products of differences are taken to 64 bits (fixmul.cuh) in frames that follow from
// the fields' and the constants'. With psi in units of 2^es (psi < 2^60), u of 2^eu (u <
// 2^59), rho of 2^er and p of 2^ep (below 2^61):
//   F (the psi terms)      in units of 2^(2 es + 125 + eF),
//   V (the viscous terms)  in units of 2^(er + eu + 127 + ev),
//   cA dp                  in units of 2^(ep + 64 + eA);
// V - F - cA dp is formed in units of 2^-60 of the largest of the three, divided by rho and
// joined with the advection. The units are below the rounding errors that the stored doubles
// bring into the differences (2^-53 psi, u, rho): F is kept to 2^-56 psi^2 of its coefficients,
// V to 2^-56 rho u, so the results' errors are those of the double-precision form. They must
// have no mean, which nothing takes back out of a velocity: with products rounded down and the
// three cut to the coarsest of their units, a 44 x 40 droplet gained 2e-18 per step in both
// components (rms error against extended precision after 400 steps 7.4e-16; 1.0e-16 so, and in
// double precision), with tau(rho) 5e-17 (2.3e-14; 1.0e-16, in double precision 7.7e-17), a
// shear flow of 1e-3 1.4e-18 (5.4e-16; 3e-19 and 2e-19). It costs 3 to 4 % of a step. A velocity
// component much smaller than the other (a shear of 1e-8 across a uniform drift of 0.1) would
// lose places in a common frame: 4e-16 after 400 steps; 3e-24 so, as in double precision, for
// another 2 to 3 % of a step.
// Conditions: psi, rho positive, all fields between 2^-320 and 2^100, velocities from 2^-900 on
// (smaller velocities and pressures count as zero: around a droplet in a fluid at rest they fall
// off to nothing over hundreds of points, and in double precision every one of them would
// take the time of three).
//
// What bounds it: instruction issue and the integer ALU pipe (1,470 to 1,500 instructions per
// point, 960 of them on that pipe). With its products on the FP64 pipe (54 to 60 instructions per
// point) and every difference rounded to a double in integer code (1,950) both pipes were 80
// to 90 % busy. Per step (two updates, two density passes): 1200 x 500 264 -> 115 us, 2048 x
// 1024 804 -> 314, 600 x 250 with tau(rho) 99 -> 55; 102, 310 and 40 with dependent launches,
// 111, 343 and 44 with results that have no mean error.
using fx::Factor;
using fx::factor;
using fx::i64;
using fx::mulhi;
using fx::mulhi2;
using fx::mulhi_k;
using fx::u32;

__device__ __forceinline__ u32 i32_of(i64 x) { return (u32)((u64)x >> 32); }

constexpr int kFDThreads = 128, kFDBlocks = 5;
constexpr int kLowest = -1000;  // of the results' units: exponents stay those of normal doubles

// a value of either sign in the frame with top exponent eg, truncated in magnitude
__device__ __forceinline__ i64 fd_term(u64 b, int eg) {
  return fx::with_sign(fx::shr_u(fx::significand(b), eg - (int)(fx::mag_hi(b) >> 20)), b);
}

__device__ __forceinline__ i64 up(i64 x, int k) { return (i64)((u64)x << k); }

// x 2^k for k of either sign, and |x| up to one
__device__ __forceinline__ i64 moved(i64 x, int k) { return k >= 0 ? up(x, k) : fx::shr_s(x, -k); }
__device__ __forceinline__ u64 mag(i64 x) { return (u64)(x ^ (x >> 63)); }

template <bool PRED, bool VV>
__device__ __forceinline__ bool fd_update_fixed(const FDArgs& a, const FDFix& k, const int (&cx)[5],
                                                const int (&ry)[5], double* drho, double* dux, double* duy) {
  auto at = [&](const double* f, int dx, int dy) { return fx::bits_of(f[ry[dy + 2] + cx[dx + 2]]); };
  constexpr u32 kTop = 1123u << 20;  // 2^100
  // psi: C, E, W, N, S, NE, NW, SW, SE, EE, WW, NN, SS
  const u64 sb[13] = {at(a.psi, 0, 0),  at(a.psi, 1, 0),   at(a.psi, -1, 0), at(a.psi, 0, 1),  at(a.psi, 0, -1),
                      at(a.psi, 1, 1),  at(a.psi, -1, 1),  at(a.psi, -1, -1), at(a.psi, 1, -1), at(a.psi, 2, 0),
                      at(a.psi, -2, 0), at(a.psi, 0, 2),   at(a.psi, 0, -2)};
  u32 mx = fx::hi32(sb[0]);
#pragma unroll
  for (int i = 1; i < 13; i += 2) mx = fx::max3(mx, fx::hi32(sb[i]), fx::hi32(sb[i + 1]));
  bool ok = mx < kTop && mx >= (703u << 20);
  const int egs = (int)(mx >> 20) + 4, es = egs - 1086;
  i64 t[13];
#pragma unroll
  for (int i = 0; i < 13; ++i)
    t[i] = (i64)fx::shr_u(fx::significand(sb[i]), egs - (int)(fx::hi32(sb[i]) >> 20));
  const i64 pd0 = t[1] - t[2], pd1 = t[3] - t[4];
  const i64 pxx = t[1] + t[2] - 2 * t[0], pyy = t[3] + t[4] - 2 * t[0];
  const i64 dxy = (t[5] - t[8]) - (t[6] - t[7]), Lc = pxx + pyy;
  const i64 dl0 = (t[9] - t[10]) + (t[5] + t[8]) - (t[6] + t[7]) - 4 * pd0;
  const i64 dl1 = (t[11] - t[12]) + (t[5] + t[6]) - (t[8] + t[7]) - 4 * pd1;
  i64 F0, F1;
  {
    const Factor q = factor(dxy), f0 = factor(pd0), f1 = factor(pd1), fl = factor(Lc), fc = factor(4 * t[0]);
    const Factor kS = factor(k.kS4), kL = factor(k.kL), kD = factor(k.kD);
    // 4 S_a, S_0 = Pd_0 Pxx + Pd_1 Dxy / 4
    const i64 s0 = mulhi2(factor(4 * pd0), factor(pxx), q, f1), s1 = mulhi2(factor(4 * pd1), factor(pyy), q, f0);
    F0 = mulhi_k(kS, factor(up(s0, 3))) + mulhi_k(kL, factor(up(mulhi(f0, fl), 3))) +
         mulhi_k(kD, factor(up(mulhi(fc, factor(dl0)), 1)));
    F1 = mulhi_k(kS, factor(up(s1, 3))) + mulhi_k(kL, factor(up(mulhi(f1, fl), 3))) +
         mulhi_k(kD, factor(up(mulhi(fc, factor(dl1)), 1)));
  }
  // velocities (9 values each: C, E, W, N, S, NE, NW, SW, SE), in one frame, or each in its own
  // where the smaller one would lose places that the stored doubles have (see far)
  u64 ub[2][9];
  int eu[2];  // units 2^eu
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    const double* f = c == 0 ? a.ux : a.uy;
    const u64 v[9] = {at(f, 0, 0), at(f, 1, 0), at(f, -1, 0), at(f, 0, 1),  at(f, 0, -1),
                      at(f, 1, 1), at(f, -1, 1), at(f, -1, -1), at(f, 1, -1)};
#pragma unroll
    for (int i = 0; i < 9; ++i) ub[c][i] = v[i];
    u32 mu = 0;
#pragma unroll
    for (int i = 0; i < 9; i += 3)
      mu = max(mu, fx::max3(fx::mag_hi(v[i]), fx::mag_hi(v[i + 1]), fx::mag_hi(v[i + 2])));
    ok = ok && mu < kTop;
    eu[c] = mu >= (123u << 20) ? (int)(mu >> 20) - 1081 : -100000;  // below 2^-900 it counts as zero
  }
  const int em_u = max(max(eu[0], eu[1]), 123 - 1081);
  const bool far = em_u - min(eu[0], eu[1]) - 7u < 50000u;  // apart by 7 or more, neither zero
  if (!far) eu[0] = eu[1] = em_u;
  i64 vel[2], D[2][2], xx[2], yy[2], xy[2];  // D[axis][component]
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    i64 v[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) v[i] = fd_term(ub[c][i], eu[c] + 1086);
    vel[c] = v[0];
    D[0][c] = PRED ? v[1] - v[0] : v[0] - v[2];
    D[1][c] = PRED ? v[3] - v[0] : v[0] - v[4];
    xx[c] = v[1] + v[2] - 2 * v[0];
    yy[c] = v[3] + v[4] - 2 * v[0];
    xy[c] = (v[5] - v[8]) - (v[6] - v[7]);
  }
  if (far) {
    vel[0] = fx::shr_s(vel[0], em_u - eu[0]);
    vel[1] = fx::shr_s(vel[1], em_u - eu[1]);
  }
  // advection: cA u . grad u_c in units of 2^(em_u + eu_c + 124 + eA)
  const Factor cA = factor(k.cA), ux2 = factor(2 * vel[0]), uy2 = factor(2 * vel[1]);
  const i64 y0 = mulhi_k(cA, factor(up(mulhi2(ux2, factor(D[0][0]), uy2, factor(D[1][0])), 3)));
  const i64 y1 = mulhi_k(cA, factor(up(mulhi2(ux2, factor(D[0][1]), uy2, factor(D[1][1])), 3)));
  const int ey0 = em_u + eu[0] + 124 + k.eA, ey1 = em_u + eu[1] + 124 + k.eA;
  int ed = em_u;  // the differences' unit from here on: set by the largest of them if far
  if (far) {
    int g[2];
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const u64 any = mag(D[0][c]) | mag(D[1][c]) | mag(xx[c]) | mag(yy[c]) | mag(xy[c]);
      g[c] = any ? eu[c] - max(fx::clz64(any) - 4, 0) : -100000;  // zeros set none
    }
    ed = max(g[0], g[1]);
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const int to = eu[c] - ed;
      D[0][c] = moved(D[0][c], to);
      D[1][c] = moved(D[1][c], to);
      xx[c] = moved(xx[c], to);
      yy[c] = moved(yy[c], to);
      xy[c] = moved(xy[c], to);
    }
  }
  const i64 Dv = D[0][0] + D[1][1], Sh = D[0][1] + D[1][0];
  // rho and p at the point and its one-sided neighbours
  const u64 rb[3] = {at(a.rho, 0, 0), at(a.rho, PRED ? 1 : -1, 0), at(a.rho, 0, PRED ? 1 : -1)};
  const u64 pb[3] = {at(a.p, 0, 0), at(a.p, PRED ? 1 : -1, 0), at(a.p, 0, PRED ? 1 : -1)};
  const u32 mr = max(max(fx::hi32(rb[0]), fx::hi32(rb[1])), fx::hi32(rb[2]));
  const u32 mn = min(min(fx::hi32(rb[0]), fx::hi32(rb[1])), fx::hi32(rb[2]));
  const u32 mp = max(max(fx::mag_hi(pb[0]), fx::mag_hi(pb[1])), fx::mag_hi(pb[2]));
  ok = ok && mr < kTop && mn >= (703u << 20) && mp < kTop;
  const int egr = (int)(mr >> 20) + 3, er = egr - 1086;
  const int egp = max((int)(mp >> 20), 703) + 3;
  i64 r[3], p[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    r[i] = (i64)fx::shr_u(fx::significand(rb[i]), egr - (int)(fx::hi32(rb[i]) >> 20));
    p[i] = fd_term(pb[i], egp);
  }
  const i64 Dr0 = PRED ? r[1] - r[0] : r[0] - r[1], Dr1 = PRED ? r[2] - r[0] : r[0] - r[2];
  const i64 Dp0 = PRED ? p[1] - p[0] : p[0] - p[1], Dp1 = PRED ? p[2] - p[0] : p[0] - p[2];
  const Factor ux = factor(vel[0]), uy = factor(vel[1]), fDv = factor(Dv), fSh = factor(Sh);
  // mass: -cA (rho div u + u . grad rho)
  i64 div = mulhi(factor(r[0]), fDv);
  if (far) div = fx::shr_s(div, em_u - ed);
  const i64 m = div + mulhi2(ux, factor(Dr0), uy, factor(Dr1));
  const int er0 = er + em_u + 125 + k.eA, er1 = max(er0, kLowest);
  *drho = fx::frame_to_double(fx::shr_s(-mulhi_k(cA, factor(up(m, 3))), er1 - er0), er1);
  // viscous terms
  i64 v1 = k.v1, v2 = k.v2, v3 = k.v3, v4 = k.v4, w1 = k.v1;  // w1: the one of rho U_yy
  if (VV) {
    // mu = rho n1, n1 = g0 + g1 rho, mu_B = rho n2, n2 = e0 - g1 rho; d mu / d rho = n1 + g1 rho
    const int d = k.ev - (er + 62 + k.g1.e);  // two places up: 0 or more for rho up to 2 rho_l
    ok = ok && d >= 0;
    const i64 gr = fx::shr_s(up(mulhi(factor(k.g1.m), factor(r[0])), 2), d);
    ok = ok && (u32)(i32_of(gr) + 0x10000000u) < 0x20000000u;
    const i64 n1 = k.g0 + gr, n2 = k.e0 - gr;
    w1 = n1;
    v1 = n1 + gr;
    v2 = n2 - gr;
    v3 = 2 * n1 + n2;
    v4 = (n1 + n2) >> 2;
  }
  const Factor f1 = factor(v1), f2 = factor(v2), f3 = factor(v3), f4 = factor(v4), fw = factor(w1);
  const Factor dr0 = factor(2 * Dr0), dr1 = factor(2 * Dr1), r2 = factor(2 * r[0]);
  const i64 V0 = mulhi_k(f1, factor(up(mulhi2(dr0, factor(D[0][0]), factor(Dr1), fSh), 1))) +
                 mulhi_k(f2, factor(mulhi(dr0, fDv))) +
                 mulhi(r2, factor(mulhi_k(f3, factor(xx[0])) + mulhi_k(f4, factor(xy[1])) + mulhi_k(fw, factor(yy[0]))));
  const i64 V1 = mulhi_k(f1, factor(up(mulhi2(dr1, factor(D[1][1]), factor(Dr0), fSh), 1))) +
                 mulhi_k(f2, factor(mulhi(dr1, fDv))) +
                 mulhi(r2, factor(mulhi_k(f3, factor(yy[1])) + mulhi_k(f4, factor(xy[0])) + mulhi_k(fw, factor(xx[1]))));
  // (V - F - cA dp) / rho
  const int eV = er + ed + 127 + k.ev, eF = 2 * es + 125 + k.eF, eP = egp - 1086 + 64 + k.eA;
  const int e = max(max(eV, eF), eP);
  // the three in a unit that the largest of them sets (of the two components): 2^-60 of it;
  // zeros set none
  const i64 P0 = mulhi_k(cA, factor(Dp0)), P1 = mulhi_k(cA, factor(Dp1));
  auto free_places = [&](i64 x, i64 y, int ex) {
    const u64 both = mag(x) | mag(y);
    return both ? fx::clz64(both) + (e - ex) : 4096;
  };
  const int n = min(min(free_places(V0, V1, eV), free_places(F0, F1, eF)), free_places(P0, P1, eP)) - 4;
  ok = ok && n >= 0;
  const int nV = n - (e - eV), nF = n - (e - eF), nP = n - (e - eP);
  const i64 a0 = moved(V0, nV) - moved(F0, nF) - moved(P0, nP);
  const i64 a1 = moved(V1, nV) - moved(F1, nF) - moved(P1, nP);
  const Factor inv = factor(fx::reciprocal<8>(fx::significand(rb[0])));
  const int e1 = e - n + 1025 - (int)(fx::hi32(rb[0]) >> 20);
  const int em0 = max(max(e1, ey0), kLowest), em1 = max(max(e1, ey1), kLowest);
  *dux = fx::frame_to_double(fx::shr_s(mulhi(factor(a0), inv), em0 - e1) - fx::shr_s(y0, em0 - ey0), em0);
  *duy = fx::frame_to_double(fx::shr_s(mulhi(factor(a1), inv), em1 - e1) - fx::shr_s(y1, em1 - ey1), em1);
  return ok;
}

template <bool PRED, bool VV>
__global__ void __launch_bounds__(kFDThreads, kFDBlocks) k_fd_update(const __grid_constant__ FDKernelArgs g) {
  begin_dependent();
  const FDArgs& a = g.a;
  const int x = blockIdx.x * 32 + threadIdx.x;
  const int y = tile_row() * (kFDThreads / 32) + threadIdx.y;
  if (x >= a.nx || y >= a.ny) return;
  const int nx = a.nx, ny = a.ny;
  // periodic columns and row offsets of the 5 x 5 neighbourhood, wrapped once (offsets
  // reach +-2, so a grid of width 1 or 2 wraps twice)
  auto wrap = [](int v, int n) {
    if (v < 0) v += n;
    if (v < 0) v += n;
    if (v >= n) v -= n;
    if (v >= n) v -= n;
    return v;
  };
  int cx[5], ry[5];
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    cx[k] = wrap(x + k - 2, nx);
    ry[k] = (a.walls ? y + k : wrap(y + k - 2, ny)) * nx;  // walls: padded rows, no wrap
  }
  double drho, dux, duy;
  if (!fd_update_fixed<PRED, VV>(a, g.k, cx, ry, &drho, &dux, &duy)) {
    fd_update_general<PRED, VV>(a, x, y);
    return;
  }
  const int i = ry[2] + x, c = ry[2] + cx[2];
  const double rho = a.rho[c], ux = a.ux[c], uy = a.uy[c];
  if (PRED) {
    a.orho[i] = rho + drho;
    a.oux[i] = ux + dux;
    a.ouy[i] = uy + duy;
  } else {
    a.orho[i] = 0.5 * (a.rho0[i] + (rho + drho));
    a.oux[i] = 0.5 * (a.ux0[i] + (ux + dux));
    a.ouy[i] = 0.5 * (a.uy0[i] + (uy + duy));
  }
}

// The general form at every point, with 64-bit offsets: planes of 2^31 values or more, and
// constants outside the frames (fd_fix), with which every point of k_fd_update would go through
// the frames first (1024^2: 442 us per step, 275 so). 3 blocks per SM: 80 registers.
template <bool PRED, bool VV>
__global__ void __launch_bounds__(256, 3) k_fd_update_general(const __grid_constant__ FDKernelArgs g) {
  begin_dependent();
  const int x = blockIdx.x * 32 + threadIdx.x, y = blockIdx.y * 8 + threadIdx.y;
  if (x < g.a.nx && y < g.a.ny) fd_update_general<PRED, VV>(g.a, x, y);
}

// The constants of one sum, m 2^e with |m| < 2^62 for the largest of them: e from the
// largest, 0 for zeros; *ok is cleared outside 2^-60 .. 2^60
int frame_of(std::initializer_list<double> v, int* ok) {
  double big = 0.0;
  for (double x : v) big = std::fmax(big, std::fabs(x));
  if (big == 0.0) return -62;
  int e;
  std::frexp(big, &e);
  if (!std::isfinite(big) || e < -60 || e > 60) *ok = 0;
  return e - 62;
}

fx::i64 in_frame(double x, int e) { return (fx::i64)std::llrint(std::ldexp((long double)x, -e)); }

FDFix fd_fix(const FDArgs& a, bool vary, double rho_l) {
  FDFix k;
  std::memset(&k, 0, sizeof(k));
  k.ok = 1;
  k.eF = frame_of({0.25 * a.kS, a.kL, a.kD}, &k.ok);
  k.eA = frame_of({a.cA}, &k.ok);
  // tau_nu(rho): room for the combinations with rho up to 2 rho_l (denser points take the general form)
  k.ev = vary ? frame_of({4.0 * a.g0, 4.0 * a.e0, 8.0 * rho_l * a.g1}, &k.ok) : frame_of({a.v1, a.v2, a.v3, a.v4}, &k.ok);
  if (!k.ok) return k;
  k.kS4 = in_frame(0.25 * a.kS, k.eF);
  k.kL = in_frame(a.kL, k.eF);
  k.kD = in_frame(a.kD, k.eF);
  k.cA = in_frame(a.cA, k.eA);
  if (vary) {
    k.g0 = in_frame(a.g0, k.ev);
    k.e0 = in_frame(a.e0, k.ev);
    k.g1 = fixnum(a.g1, 1);
  } else {
    k.v1 = in_frame(a.v1, k.ev);
    k.v2 = in_frame(a.v2, k.ev);
    k.v3 = in_frame(a.v3, k.ev);
    k.v4 = in_frame(a.v4, k.ev);
  }
  return k;
}

template <bool PRED, bool VV>
void launch_fd_update(const FDKernelArgs& g, int64_t plane, cudaStream_t s) {
  const int rows = kFDThreads / 32;
  if (g.k.ok && plane < (int64_t)INT32_MAX)
    launch_dependent(k_fd_update<PRED, VV>, tile_grid((g.a.nx + 31) / 32, (g.a.ny + rows - 1) / rows), dim3(32, rows), s, g);
  else
    launch_dependent(k_fd_update_general<PRED, VV>, dim3((g.a.nx + 31) / 32, (g.a.ny + 7) / 8), dim3(32, 8), s, g);
}

}  // namespace
}  // namespace pplbm

using namespace pplbm;

struct pplbm_fd {
  int nx, ny;
  int64_t n;     // fluid nodes
  bool walls;
  int64_t np;    // values per plane: n, or nx (ny + 4) with walls
  int64_t off;   // first fluid value of a plane: 0, or 2 nx with walls
  EosConst eos;
  FDEosArgs eos_args;
  pplbm_eos_derived derived;
  double G, eps, dx, mu_c, muB_c, tau_e;
  double kappa;   // surface-tension control, 0 = off
  bool var_visc;  // tau_nu(rho) = ta + tb rho instead of a constant
  double ta, tb;
  double* U;   // rho, ux, uy
  double* S;   // predictor state
  double* psi;
  double* p;
  cudaStream_t stream;
  int64_t steps;
};

extern "C" {

namespace {
// 0: periodic y, 1: walls, -1: not accepted
int fd_walls(const pplbm_lattice* l) {
  if (l->bc == (PPLBM_BC_PERIODIC_X | PPLBM_BC_PERIODIC_Y)) return 0;
  if (l->bc == (PPLBM_BC_PERIODIC_X | PPLBM_BC_WALL_BOTTOM | PPLBM_BC_WALL_TOP) && l->ny >= 2) return 1;
  return -1;
}
}  // namespace

size_t pplbm_fd_workspace_bytes(const pplbm_lattice* lattice) {
  if (!lattice || lattice->nx < 1 || lattice->ny < 1 || lattice->ny > 65535 * 8) return 0;
  const int w = fd_walls(lattice);
  if (w < 0) return 0;
  return sizeof(double) * 8 * (size_t)lattice->nx * (size_t)(lattice->ny + 4 * w);
}

pplbm_status pplbm_fd_create(pplbm_fd** out, const pplbm_lattice* lattice, const pplbm_eos_params* eos, double G,
                             double tau_nu, double tau_e, double dx, void* workspace, size_t workspace_bytes,
                             void* stream) {
  if (!out) return PPLBM_ERR_ARG;
  *out = nullptr;
  if (!lattice || !eos || !workspace || lattice->nx < 1 || lattice->ny < 1 || lattice->reserved != 0) return PPLBM_ERR_ARG;
  if (lattice->ny > 65535 * 8) return PPLBM_ERR_ARG;  // k_fd_update_general's grid: 8-row tiles on its y axis
  if (fd_walls(lattice) < 0) return PPLBM_ERR_ARG;
  if (!(tau_nu > 0.5) || !(tau_e > 0.0) || !(dx > 0.0)) return PPLBM_ERR_ARG;
  if (workspace_bytes < pplbm_fd_workspace_bytes(lattice)) return PPLBM_ERR_ARG;
  pplbm_eos_derived d;
  const pplbm_status st = pplbm_eos_setup(eos, G, &d);
  if (st != PPLBM_OK) return st;
  pplbm_fd* f = new (std::nothrow) pplbm_fd();
  if (!f) return PPLBM_ERR_ARG;
  f->nx = lattice->nx;
  f->ny = lattice->ny;
  f->n = (int64_t)f->nx * f->ny;
  f->walls = fd_walls(lattice) == 1;
  f->np = (int64_t)f->nx * (f->ny + (f->walls ? 4 : 0));
  f->off = f->walls ? 2 * (int64_t)f->nx : 0;
  f->derived = d;
  f->eos = make_eos_const(d);
  f->eos_args.eos = f->eos;
  f->eos_args.fix = make_eos_fix(d, G);
  f->eos_args.half = (fx::i64)std::ldexp(-0.5 * G, 63 + f->eos_args.fix.s);
  f->G = G;
  f->eps = d.eps;
  f->dx = dx;
  f->mu_c = (tau_nu - 0.5) / 3.0;
  f->muB_c = (tau_e - tau_nu) / 3.0;
  f->tau_e = tau_e;
  f->kappa = 0.0;
  f->var_visc = false;
  double* w = (double*)workspace;
  f->U = w;
  f->S = w + 3 * f->np;
  f->psi = w + 6 * f->np;
  f->p = w + 7 * f->np;
  f->stream = (cudaStream_t)stream;
  *out = f;
  return PPLBM_OK;
}

pplbm_status pplbm_fd_set_state(pplbm_fd* f, const double* rho, const double* ux, const double* uy) {
  if (!f || !rho || !ux || !uy) return PPLBM_ERR_ARG;
  const double* src[3] = {rho, ux, uy};
  for (int k = 0; k < 3; ++k)
    if (cudaMemcpyAsync(f->U + k * f->np + f->off, src[k], sizeof(double) * f->n, cudaMemcpyDefault, f->stream) !=
        cudaSuccess)
      return PPLBM_ERR_CUDA;
  return cudaStreamSynchronize(f->stream) == cudaSuccess ? PPLBM_OK : PPLBM_ERR_CUDA;
}

pplbm_status pplbm_fd_get_state(pplbm_fd* f, double* rho, double* ux, double* uy) {
  if (!f) return PPLBM_ERR_ARG;
  double* dst[3] = {rho, ux, uy};
  for (int k = 0; k < 3; ++k)
    if (dst[k] &&
        cudaMemcpyAsync(dst[k], f->U + k * f->np + f->off, sizeof(double) * f->n, cudaMemcpyDefault, f->stream) !=
            cudaSuccess)
      return PPLBM_ERR_CUDA;
  return cudaStreamSynchronize(f->stream) == cudaSuccess ? PPLBM_OK : PPLBM_ERR_CUDA;
}

pplbm_status pplbm_fd_step(pplbm_fd* f, int64_t nsteps, double dt) {
  if (!f || nsteps < 0 || !(dt > 0.0)) return PPLBM_ERR_ARG;
  const unsigned eb = (unsigned)((f->n + 127) / 128);
  FDKernelArgs g;
  std::memset(&g, 0, sizeof(g));
  FDArgs& a = g.a;
  a.nx = f->nx;
  a.ny = f->ny;
  a.walls = f->walls ? 1 : 0;
  const double h = 1.0 / f->dx, h2 = h * h, h3 = h2 * h;
  a.cA = dt * h;
  a.kS = dt * 0.5 * h3 * (f->G / 6.0 - f->eps * f->G / 4.0 - f->kappa * f->G / 6.0);
  a.kL = dt * 0.5 * h3 * (f->G / 12.0 + f->kappa * f->G / 6.0);
  a.kD = dt * 0.5 * h3 * (f->G / 4.0);
  a.v1 = dt * h2 * f->mu_c;
  a.v2 = dt * h2 * f->muB_c;
  a.v3 = dt * h2 * (2.0 * f->mu_c + f->muB_c);
  a.v4 = dt * h2 * (f->mu_c + f->muB_c) * 0.25;
  if (f->var_visc) {
    a.g0 = dt * h2 * (f->ta - 0.5) / 3.0;
    a.g1 = dt * h2 * f->tb / 3.0;
    a.e0 = dt * h2 * (f->tau_e - f->ta) / 3.0;
  }
  a.psi = f->psi;
  a.p = f->p;
  g.k = fd_fix(a, f->var_visc, f->derived.rho_l);
  const int64_t n = f->n, np = f->np, off = f->off;
  const unsigned wb = (unsigned)((f->nx + 63) / 64);
  const double two_dy = 2.0 * f->dx, psi_l = f->derived.psi_l;
  // psi and p of the state in X, then its wall layers
  auto eos_pass = [&](double* X) {
    launch_dependent(k_fd_eos, eb, 128, f->stream, f->eos_args, X + off, f->psi + off, f->p + off, n);
    if (f->walls)
      launch_dependent(k_fd_walls, wb, 64, f->stream, f->eos, X, X + np, X + 2 * np, f->psi, f->p, f->nx, f->ny, two_dy,
                       psi_l);
  };
  for (int64_t s = 0; s < nsteps; ++s) {
    // predictor: U* = U + dt R_f(U)
    eos_pass(f->U);
    a.rho = f->U;
    a.ux = f->U + np;
    a.uy = f->U + 2 * np;
    a.orho = f->S;
    a.oux = f->S + np;
    a.ouy = f->S + 2 * np;
    if (f->var_visc)
      launch_fd_update<true, true>(g, np, f->stream);
    else
      launch_fd_update<true, false>(g, np, f->stream);
    // corrector: U <- (U + U* + dt R_b(U*)) / 2
    eos_pass(f->S);
    a.rho = f->S;
    a.ux = f->S + np;
    a.uy = f->S + 2 * np;
    a.rho0 = f->U;
    a.ux0 = f->U + np;
    a.uy0 = f->U + 2 * np;
    a.orho = f->U;
    a.oux = f->U + np;
    a.ouy = f->U + 2 * np;
    if (f->var_visc)
      launch_fd_update<false, true>(g, np, f->stream);
    else
      launch_fd_update<false, false>(g, np, f->stream);
  }
  f->steps += nsteps;
  return cudaGetLastError() == cudaSuccess ? PPLBM_OK : PPLBM_ERR_CUDA;
}

pplbm_status pplbm_fd_set_two_phase_viscosity(pplbm_fd* f, double tau_l, double visc_ratio) {
  if (!f || !(tau_l > 0.5) || !(visc_ratio > 0.0)) return PPLBM_ERR_ARG;
  const double tau_v = 0.5 + visc_ratio * (tau_l - 0.5);
  const double rv = f->derived.rho_v, rl = f->derived.rho_l;
  f->tb = (tau_l - tau_v) / (rl - rv);
  f->ta = tau_l - f->tb * rl;
  f->var_visc = true;
  return PPLBM_OK;
}

pplbm_status pplbm_fd_set_surface_tension(pplbm_fd* f, double kappa) {
  if (!f || !std::isfinite(kappa) || !(kappa < 1.0)) return PPLBM_ERR_ARG;
  f->kappa = kappa;
  return PPLBM_OK;
}

pplbm_status pplbm_fd_sync(pplbm_fd* f) {
  if (!f) return PPLBM_ERR_ARG;
  return cudaStreamSynchronize(f->stream) == cudaSuccess ? PPLBM_OK : PPLBM_ERR_CUDA;
}

void pplbm_fd_destroy(pplbm_fd* f) { delete f; }

}  // extern "C"
