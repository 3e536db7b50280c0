// Host build of the fixed-point collision of csrc/collide_fixed.cuh (the same source the
// collision kernels compile), for the CPU tests.
#include "../../paper_2107_06355_gb300/csrc/collision_args.cpp"

using namespace pplbm::fx;

namespace {

template <bool SHEAR, bool ST>
bool one(const CollideFix& k, const double* in, double (&f)[9]) {
  u64 p[9];
  for (int i = 0; i < 9; ++i) p[i] = bits_of(in[i]);
  return collide_fixed<SHEAR, ST, 4>(k, p, in[9], in[10], in[11], in[12], in[13], f);
}

}  // namespace

extern "C" {

// rows of 14 (psi at C, E, W, N, S, NE, NW, SW, SE; rho, jx, jy, m7, m8) -> out rows of 10:
// the nine populations, then 1 if the row is in the domain. c: half_force, zz_scale,
// kappa_q, tau_a, tau_b as in StepArgs.
void fm_collide(long long n, int shear, int st, const double* c, const double* in, double* out) {
  const CollideFix k{pplbm::fixnum(c[0], 36), pplbm::fixnum(c[1], 1), pplbm::fixnum(c[2], 36),
                     pplbm::fixnum(c[4], 1), (i64)std::ldexp(c[3], 58)};
  for (long long i = 0; i < n; ++i) {
    double f[9];
    const double* r = in + 14 * i;
    const bool ok = shear ? (st ? one<true, true>(k, r, f) : one<true, false>(k, r, f))
                          : (st ? one<false, true>(k, r, f) : one<false, false>(k, r, f));
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
