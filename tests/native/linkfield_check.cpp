// Host build of the fixed-point field test (csrc/fixedpt.cuh) for tests/test_fixedpt_components_host.py.
#include <cstring>

#include "../../paper_0910_1048_gb300/csrc/fixedpt.cuh"

using namespace ovl;

// Whether n links u[n][3][3] (complex) may be kept in fixed point: what k_fx_links and k_fx_field decide.
extern "C" int field_usable(const double* u, long long n) {
  double lo = 1e308, hi = 0;
  unsigned weak = 0;
  for (long long l = 0; l < n; ++l) {
    Mat3<double> m;
    for (int k = 0; k < 9; ++k) m.m[k / 3][k % 3] = mk<double>(u[18 * l + 2 * k], u[18 * l + 2 * k + 1]);
    double top, need;
    bool w;
    fx_link_range(m, top, need, w);
    lo = top < lo ? top : lo;
    hi = need > hi ? need : hi;
    weak += w;
  }
  int uexp;
  return fx_field_scale(lo, hi, &uexp) && fx_field_mixes(weak, (size_t)n);
}

// Fixed-point copies of n components and what the library's conversion is to equal: x 2^(58 - uexp), ties to even.
extern "C" void convert(const double* x, long long n, int uexp, long long* got, long long* want) {
  for (long long i = 0; i < n; ++i) {
    got[i] = fx_link_fixed(x[i], uexp);
    want[i] = std::llrint(std::ldexp(x[i], 58 - uexp));
  }
}
