// Host build of the products of csrc/fixmul.cuh, for the CPU tests.
#include "../../paper_2107_06355_gb300/csrc/fixmul.cuh"

using namespace pplbm::fx;

extern "C" {

void mh_product(long long n, const long long* x, const long long* y, long long* out) {
  for (long long i = 0; i < n; ++i) out[i] = mulhi(factor(x[i]), factor(y[i]));
}

// k x, k a constant
void mh_constant(long long n, long long k, const long long* x, long long* out) {
  for (long long i = 0; i < n; ++i) out[i] = mulhi_k(factor(k), factor(x[i]));
}

// x y + z w
void mh_pair(long long n, const long long* x, const long long* y, const long long* z, const long long* w,
             long long* out) {
  for (long long i = 0; i < n; ++i) out[i] = mulhi2(factor(x[i]), factor(y[i]), factor(z[i]), factor(w[i]));
}
}
