// Host build of the fixed-point EOS of csrc/eos_fixed.cuh (the same source the density
// kernels compile) with the library's EOS set-up, for the CPU tests.
#include "../../paper_2107_06355_gb300/csrc/collision_args.cpp"
#include "../../paper_2107_06355_gb300/csrc/eos_setup.cpp"

extern "C" {

// set-up of one EOS: p = {mode, Tr, a_liq, a_vap, b, R, alpha, r_theta}; out: G, b, R T_l,
// R T_v, a_l, a_v, dP, rho_v, rho_max, rho_min, rho_l, p_max, b1, a1sq, p_min, b3, a3sq
int ef_setup(const double* p, double G, double* out) {
  pplbm_eos_params q{(int32_t)p[0], 0, p[1], p[2], p[3], p[4], p[5], p[6], p[7]};
  pplbm_eos_derived d;
  const int s = (int)pplbm_eos_setup(&q, G, &d);
  if (s) return s;
  const double v[17] = {d.G, d.b, d.R * d.T_l, d.R * d.T_v, d.a_l, d.a_v, d.dP, d.rho_v, d.rho_max, d.rho_min,
                        d.rho_l, d.p_max, d.b1, d.a1sq, d.p_min, d.b3, d.a3sq};
  std::memcpy(out, v, sizeof(v));
  return 0;
}

// rho (n) -> psi (n), ok (n): 1 in the fixed-point domain
int ef_psi(const double* p, double G, long long n, const double* rho, double* psi, int* ok) {
  pplbm_eos_params q{(int32_t)p[0], 0, p[1], p[2], p[3], p[4], p[5], p[6], p[7]};
  pplbm_eos_derived d;
  if (pplbm_eos_setup(&q, G, &d)) return 1;
  const pplbm::EosConst c = pplbm::make_eos_const(d);
  const pplbm::EosFix e = pplbm::make_eos_fix(d, G);
  for (long long i = 0; i < n; ++i) {
    const pplbm::fx::u64 b = pplbm::fx::bits_of(rho[i]);
    pplbm::fx::i64 P = 0;
    int ex = 0;
    ok[i] = e.ok && pplbm::psi2_fixed(e, c, pplbm::fx::significand(b), (int)(b >> 52), (pplbm::fx::i64)b, &P, &ex);
    psi[i] = ok[i] ? pplbm::fx::sqrt_double(P, ex) : 0.0;
  }
  return 0;
}

// sqrt(P 2^ex) as a double
void ef_sqrt(long long n, const long long* P, const int* ex, double* out) {
  for (long long i = 0; i < n; ++i) out[i] = pplbm::fx::sqrt_double(P[i], ex[i]);
}
}
