// Host derivation of the collision arguments from a relaxation set, shared by the
// single-lattice context, the batched engine and the no-allocation entry point.
#include <cmath>

#include "internal.h"

namespace pplbm {

int collision_kind(const pplbm_relax* r) {
  if (!r || r->reserved != 0) return -1;
  if (!std::isfinite(r->kappa) || !(r->kappa < 1.0)) return -1;
  if (r->forcing != PPLBM_FORCING_GUO && r->forcing != PPLBM_FORCING_LI) return -1;
  if (r->kind == PPLBM_RELAX_TWO_PHASE) {
    if (!(r->tau_l > 0.5) || !(r->visc_ratio > 0.0) || !std::isfinite(r->tau_l) || !std::isfinite(r->visc_ratio))
      return -1;
    return kShearTau;
  }
  if (r->kind != PPLBM_RELAX_MRT) return -1;
  const double t[6] = {r->tau_rho, r->tau_e, r->tau_zeta, r->tau_j, r->tau_q, r->tau_nu};
  for (double v : t)
    if (!(v > 0.5) || !std::isfinite(v)) return -1;
  if (r->tau_rho == 1.0 && r->tau_e == 1.0 && r->tau_zeta == 1.0 && r->tau_j == 1.0 && r->tau_q == 1.0)
    return r->tau_nu == 1.0 ? kUnitTau : kShearTau;
  return kFullMrt;
}

fx::FixNum fixnum(double x, int div) {
  fx::FixNum r{0, -4096, 0};
  if (x == 0.0) return r;
  if (!std::isfinite(x)) return fx::FixNum{1ll << 62, 4096, 0};
  int e;
  const int64_t s = (int64_t)std::ldexp(std::frexp(std::fabs(x), &e), 53);  // |x| = s 2^(e - 53)
  unsigned __int128 q = ((unsigned __int128)s << 72) / (unsigned)div;       // |x| / div = q 2^(e - 125)
  e -= 125;
  while (q >> 63) {
    q = (q >> 1) + (q & 1 && !(q >> 64));
    ++e;
  }
  r.m = x < 0.0 ? -(int64_t)q : (int64_t)q;
  r.e = e;
  return r;
}

// round(x 2^k) when it is below 2^bits in magnitude; *ok is cleared otherwise
static int64_t fixed(long double x, int k, int bits, int* ok) {
  const long double v = std::ldexp(x, k);
  if (!(std::fabs(v) < std::ldexp(1.0L, bits))) {
    *ok = 0;
    return 0;
  }
  return (int64_t)std::llrint(v);
}

// A branch psi^2 2^-s = k3 rho + A + B g((rho - rho0) / a), rho up to rho_top: an ellipse
// (|rho - rho0| <= a) or the cubic (a its span). *ok is cleared when a is not positive and
// finite: a block that no set-up made.
static LoopFix loop_branch(bool ellipse, long double rho_top, long double rho0, long double a, long double A,
                           long double B, int* ok) {
  LoopFix L{};
  if (!(a > 0.0L) || !std::isfinite(a) || !std::isfinite(rho_top)) {
    *ok = 0;
    return L;
  }
  int e;
  std::frexp(ellipse ? std::fmax(rho_top, 2.0L * a) : rho_top, &e);  // < 2^e
  L.q = (ellipse ? 63 : 62) - e;
  if (ellipse) {
    L.c = fixed(a, L.q, 62, ok);
    B = B / a * std::ldexp(1.0L, 62 - L.q);
  } else {
    while (L.up <= 12 && std::ldexp(1.0L / a, 126 - L.up - L.q) >= 0x1.8p62L) ++L.up;
    if (L.up > 12) *ok = 0;  // the span is far below a frame this coarse
    L.c = fixed(1.0L / a, 126 - L.up - L.q, 63, ok);
  }
  L.rho0 = fixed(rho0, L.q, 63, ok);
  L.A = fixnum((double)A, 1);
  L.B = fixnum((double)B, 1);
  return L;
}

EosFix make_eos_fix(const pplbm_eos_derived& d, double G) {
  EosFix e{};
  int lb;
  e.ok = std::frexp(d.b / 4.0, &lb) == 0.5 ? 1 : 0;
  e.log2_b4 = lb - 1;
  if (e.log2_b4 < -30 || e.log2_b4 > 30) e.ok = 0;
  const long double sc = 2.0L / (long double)G, k3 = -sc / 3.0L;
  std::frexp(k3, &e.s);
  const long double one = std::ldexp(1.0L, -e.s);  // every constant times 2^-s
  e.k3_57 = fixed(k3 * one, 57, 57, &e.ok);
  e.k3_60 = fixed(k3 * one, 60, 60, &e.ok);
  const bool smooth = d.mode == PPLBM_EOS_SMOOTH || d.mode == PPLBM_EOS_SMOOTH_MOD;
  for (int i = 0; i < 2; ++i) {
    const bool v = i == 0 && smooth;
    CsFix& k = e.cs[i];
    k.c1 = fixed(2.0L * sc * (long double)d.R * (v ? d.T_v : d.T_l) * one, 62, 63, &e.ok);
    k.k2 = fixed(-sc * (v ? d.a_v : d.a_l) * one, 58, 62, &e.ok);
    const double k4 = v ? 0.0 : (double)(sc * d.dP * one);
    k.k4 = fixnum(k4, 1);
    k.k4.m >>= 2;  // room for the sum with rho x
    k.k4.e += 2;
  }
  if (smooth) {
    e.loop = 1;
    const long double pM = d.p_max, pm = d.p_min, b1 = d.b1, b3 = d.b3, s = sc * one;
    e.loops[0] = loop_branch(true, d.rho_max, d.rho_max, std::sqrt((long double)d.a1sq), s * (pM - b1), s * b1, &e.loop);
    e.loops[1] = loop_branch(true, d.rho_l, d.rho_min, std::sqrt((long double)d.a3sq), s * (pm + b3), -s * b3, &e.loop);
    e.loops[2] = loop_branch(false, d.rho_min, d.rho_max, (long double)d.rho_min - d.rho_max, s * pM, s * (pm - pM), &e.loop);
  }
  return e;
}

void set_collision_args(StepArgs& a, int kind, const pplbm_relax& r, const pplbm_eos_derived& d, double G) {
  // Li forcing parameter (Eq. LiFS): 0 for the Guo scheme (Eq. GFS), or from eps of
  // Eq. VaporLiqEq for the EOS in use (Sec. III.A)
  const double sigma = r.forcing == PPLBM_FORCING_GUO ? 0.0 : r.sigma_auto ? -d.eps / (16.0 * G) : r.sigma;
  a.tau_a = a.tau_b = 0.0;
  if (kind == kShearTau) {
    if (r.kind == PPLBM_RELAX_TWO_PHASE) {
      // tau = tau_l (rho - rho_v)/(rho_l - rho_v) + tau_v (rho - rho_l)/(rho_v - rho_l),
      // tau_v = 1/2 + v_r (tau_l - 1/2) (Eq. RelaxationTime)
      const double tv = 0.5 + r.visc_ratio * (r.tau_l - 0.5);
      a.tau_b = (r.tau_l - tv) / (d.rho_l - d.rho_v);
      a.tau_a = r.tau_l - a.tau_b * d.rho_l;
    } else {
      a.tau_a = r.tau_nu;
    }
  }
  a.zz_scale = sigma * G * G / 432.0;
  a.kappa_q = r.kappa * G / 24.0;
  a.efix = make_eos_fix(d, G);
  a.fix.ch = fixnum(a.half_force, 36);
  a.fix.zz = fixnum(a.zz_scale, 1);
  a.fix.kq = fixnum(a.kappa_q, 36);
  a.fix.tb = fixnum(a.tau_b, 1);
  int fits = 1;
  a.fix.ta = kind == kShearTau ? fixed(a.tau_a, 58, 62, &fits) : 0;
  if (!fits) a.fix.ta = INT64_MIN;  // |tau_a| >= 16: every node takes the general collision
  if (kind == kFullMrt) {
    const double t[9] = {r.tau_rho, r.tau_e, r.tau_zeta, r.tau_j, r.tau_q, r.tau_j, r.tau_q, r.tau_nu, r.tau_nu};
    for (int k = 0; k < 9; ++k) a.omega[k] = 1.0 / t[k];
    a.li_e = 12.0 * sigma / (r.tau_e - 0.5);
    a.li_z = 12.0 * sigma / (r.tau_zeta - 0.5);
    int ok = 1;
    a.fix.we = fixed(a.omega[1], 61, 62, &ok);
    a.fix.wz = fixed(a.omega[2], 61, 62, &ok);
    a.fix.wq = fixed(a.omega[4], 61, 62, &ok);
    a.fix.wn = fixed(a.omega[7], 61, 62, &ok);
    a.fix.le = fixnum(a.li_e * G * G / 144.0, 36);
    a.fix.lz = fixnum(a.li_z * G * G / 144.0, 36);
  }
}

}  // namespace pplbm
