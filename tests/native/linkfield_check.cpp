// Host build of the fixed-point field test (csrc/fixedpt.cuh) for tests/test_fixedpt_components_host.py.
#include <cstring>
#include <vector>

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

namespace {
struct Load {
  const double* p;  // [12][V] complex
  int vol;
  void operator()(int s, Spin<double>& o) const {
    for (int c = 0; c < 12; ++c) {
      const double* q = p + 2 * ((size_t)c * vol + s);
      o.c[c / 3][c % 3] = mk<double>(q[0], q[1]);
    }
  }
};
}  // namespace

// Per spin and site, whether the sum of the eight hops (scale 2^0, antiperiodic time) is large in the sense of fx_large.
extern "C" void large_spins(const int* d, double mu, const double* u, const double* psi, int* large) {
  Geom g;
  g.lx = d[0], g.ly = d[1], g.lz = d[2], g.lt = d[3];
  g.vol = d[0] * d[1] * d[2] * d[3];
  g.sy = d[0], g.sz = d[0] * d[1], g.st = d[0] * d[1] * d[2];
  g.t_bc = -1;
  std::vector<FxC> fx((size_t)36 * g.vol);
  for (size_t e = 0; e < fx.size(); ++e) fx[e] = fx_link_entry(mk<double>(u[2 * e], u[2 * e + 1]), 0);
  const FxCoef c = fx_coef(-2.0, mu);
  for (int s = 0; s < g.vol; ++s) {
    FxAcc a;
    fx_clear(a);
    FxSizes z;
    int E;
    const bool ok = fx_hops(g, fx.data(), s, 0, 8, c, Load{psi, g.vol}, false, a, E, z);
    for (int i = 0; i < 4; ++i) large[(size_t)i * g.vol + s] = ok && fx_large(a.re[i], a.im[i]);
  }
}
