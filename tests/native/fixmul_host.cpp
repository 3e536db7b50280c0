// Host build of the fixed-point collision of csrc/collide_fixed.cuh (the same source the
// collision kernels compile), for the CPU tests.
#include "../../paper_2107_06355_gb300/csrc/collision_args.cpp"

using namespace pplbm::fx;

namespace {

template <int FORM, bool ST>
bool one(const CollideFix& k, const double* in, double (&f)[9]) {
  u64 p[9];
  for (int i = 0; i < 9; ++i) p[i] = bits_of(in[i]);
  const double m[6] = {in[12], in[13], in[14], in[15], in[16], in[17]};
  return collide_fixed<FORM, ST, 4>(k, p, in[9], in[10], in[11], m, f);
}

}  // namespace

extern "C" {

// rows of 18 (psi at C, E, W, N, S, NE, NW, SW, SE; rho, jx, jy; the moments: m7, m8 for form
// 1, rows 1, 2, 4, 6, 7, 8 for form 2) -> out rows of 10: the nine populations, then 1 if the
// row is in the domain. c: half_force, zz_scale, kappa_q, tau_a, tau_b as in StepArgs, then
// for form 2 the rates of rows 1, 2, (4, 6), (7, 8) and li_e G^2/144, li_z G^2/144.
void fm_collide(long long n, int form, int st, const double* c, const double* in, double* out) {
  CollideFix k{};
  k.ch = pplbm::fixnum(c[0], 36);
  k.zz = pplbm::fixnum(c[1], 1);
  k.kq = pplbm::fixnum(c[2], 36);
  k.tb = pplbm::fixnum(c[4], 1);
  k.ta = (i64)std::ldexp(c[3], 58);
  if (form == 2) {
    i64* w[4] = {&k.we, &k.wz, &k.wq, &k.wn};
    for (int i = 0; i < 4; ++i) *w[i] = (i64)std::ldexp(c[5 + i], 61);
    k.le = pplbm::fixnum(c[9], 36);
    k.lz = pplbm::fixnum(c[10], 36);
  }
  for (long long i = 0; i < n; ++i) {
    double f[9];
    const double* r = in + 18 * i;
    bool ok;
    switch (2 * form + st) {
      case 0: ok = one<0, false>(k, r, f); break;
      case 1: ok = one<0, true>(k, r, f); break;
      case 2: ok = one<1, false>(k, r, f); break;
      case 3: ok = one<1, true>(k, r, f); break;
      case 4: ok = one<2, false>(k, r, f); break;
      default: ok = one<2, true>(k, r, f); break;
    }
    for (int j = 0; j < 9; ++j) out[10 * i + j] = f[j];
    out[10 * i + 9] = ok ? 1.0 : 0.0;
  }
}

// L (significands) -> 9 2^59 / m as signed integers
void fm_reciprocal(long long n, const unsigned long long* L, long long* out) {
  for (long long i = 0; i < n; ++i) out[i] = reciprocal<9>(L[i]);
}

// integers >= 2^32 -> doubles
void fm_to_double(long long n, const long long* in, double* out) {
  for (long long i = 0; i < n; ++i) out[i] = double_of(to_double_int(in[i]));
}
}
