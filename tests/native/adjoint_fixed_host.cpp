// Host build of the fixed-point reverse of the collision (csrc/adjoint_fixed.cuh), for the
// CPU tests.
#include "../../paper_2107_06355_gb300/csrc/adjoint_fixed.cuh"
#include "../../paper_2107_06355_gb300/csrc/collision_args.cpp"
#include "../../paper_2107_06355_gb300/csrc/eos_setup.cpp"

extern "C" {

// rows of 23 (psi at C, E, W, N, S, NE, NW, SW, SE; rho, jx, jy, m7, m8; mu_0..8) -> out
// rows of 17: rho_b, jx_b, jy_b, m7_b, m8_b, psi_b, gx_b, gy_b, zs_b, u6, u7, u8, omega, 6 t,
// sd, xd and 1 if the row is in the domain. c: half_force, zz_scale, tau_a, tau_b as in StepArgs.
void af_reverse(long long n, int shear, const double* c, const double* in, double* out) {
  using namespace pplbm::fx;
  CollideFix k{};
  k.ch = pplbm::fixnum(c[0], 36);
  k.zz = pplbm::fixnum(c[1], 1);
  k.ta = (i64)std::ldexp(c[2], 58);
  k.tb = pplbm::fixnum(c[3], 1);
  for (long long i = 0; i < n; ++i) {
    const double* r = in + 23 * i;
    u64 p[9];
    double mu[9];
    for (int j = 0; j < 9; ++j) {
      p[j] = bits_of(r[j]);
      mu[j] = r[14 + j];
    }
    ReverseOut o = {};
    const bool ok = shear ? collide_reverse_fixed<true, true>(k, p, r[9], r[10], r[11], r[12], r[13], mu, &o)
                          : collide_reverse_fixed<false, true>(k, p, r[9], r[10], r[11], r[12], r[13], mu, &o);
    const double v[17] = {o.rho_b, o.jx_b, o.jy_b, o.m7_b, o.m8_b, o.psi_b, o.gx_b, o.gy_b, o.zs_b,
                          o.u6, o.u7, o.u8, o.om, o.t6, o.sd, o.xd, ok ? 1.0 : 0.0};
    for (int j = 0; j < 17; ++j) out[17 * i + j] = v[j];
  }
}

// d psi^2 / d rho of the vapour (branch 0) or liquid C-S branch of the EOS p = {mode, Tr,
// a_liq, a_vap, b, R, alpha}, its constants {b, R T, a} in k, and 1/(2 rho)
int af_slope(const double* p, double G, int branch, long long n, const double* rho, double* k, double* slope,
             double* half, int* ok) {
  pplbm_eos_params q{(int32_t)p[0], 0, p[1], p[2], p[3], p[4], p[5], p[6], 0.0};
  pplbm_eos_derived d;
  if (pplbm_eos_setup(&q, G, &d)) return 1;
  k[0] = d.b;
  k[1] = d.R * (branch ? d.T_l : d.T_v);
  k[2] = branch ? d.a_l : d.a_v;
  const pplbm::EosFix e = pplbm::make_eos_fix(d, G);
  for (long long i = 0; i < n; ++i) {
    const pplbm::fx::u64 b = pplbm::fx::bits_of(rho[i]);
    ok[i] = pplbm::fx::cs_slope_fixed(e, e.cs[branch], pplbm::fx::significand(b), (int)(b >> 52), slope + i);
    half[i] = pplbm::fx::half_reciprocal(b);
  }
  return 0;
}
}
