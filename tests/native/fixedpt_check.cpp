// Host build of the fixed-point hops (csrc/fixedpt.cuh) for tests/test_fixedpt_host.py: D_W psi by fixed
// point, by the FP64 hops and in extended precision on the same inputs.
#include <cstring>

#include "../../paper_0910_1048_gb300/csrc/fixedpt.cuh"

using namespace ovl;

namespace {

template <class R>
struct Load {
  const double* p;  // [12][V] complex
  int vol;
  bool g5;
  void operator()(int s, Spin<R>& o) const {
    for (int c = 0; c < 12; ++c) {
      const double* q = p + 2 * ((size_t)c * vol + s);
      const R sg = g5 && c >= 6 ? (R)-1 : (R)1;
      o.c[c / 3][c % 3] = mk<R>(sg * (R)q[0], sg * (R)q[1]);
    }
  }
};

Geom geom(const int* d, int t_bc) {
  Geom g;
  g.lx = d[0], g.ly = d[1], g.lz = d[2], g.lt = d[3];
  g.vol = d[0] * d[1] * d[2] * d[3];
  g.sy = d[0], g.sz = d[0] * d[1], g.st = d[0] * d[1] * d[2];
  g.t_bc = t_bc;
  return g;
}

void run(const Geom& g, double m_w, double mu, const FxC* fx, int uexp, const double* psi, bool g5in, double* out,
         int* usable) {
  const FxCoef c = fx_coef(m_w, mu);
  for (int s = 0; s < g.vol; ++s) {
    FxAcc a;
    int E;
    fx_clear(a);
    const Load<double> ld{psi, g.vol, false};
    usable[s] = c.ok && fx_hops(g, fx, s, 0, 8, c, ld, g5in, a, E);
    Spin<double> o;
    Load<double>{psi, g.vol, g5in}(s, o);
    const double f = usable[s] ? fx_unit(E, c, uexp) : 0.0;
    for (int i = 0; i < 12; ++i) {
      double* q = out + 2 * ((size_t)i * g.vol + s);
      q[0] = std::fma(f, (double)a.re[i / 3][i % 3], o.c[i / 3][i % 3].re);
      q[1] = std::fma(f, (double)a.im[i / 3][i % 3], o.c[i / 3][i % 3].im);
    }
  }
}

template <class R>
void plain(const Geom& g, double m_w, double mu, const double* u, const double* psi, bool g5in, R* out) {
  Links U;
  U.f64 = (const double2*)u;
  const R kap = 1 / (2 * (R)m_w + 8);
  HopCoef<R> c;
  c.ks = -kap;
  c.ktf = -kap * (R)std::exp(mu);  // the factors both paths are given, rounded to FP64
  c.ktb = -kap * (R)std::exp(-mu);
  for (int s = 0; s < g.vol; ++s) {
    Spin<R> o;
    dslash_site<LINK_F64>(g, U, s, c, Load<R>{psi, g.vol, g5in}, o);
    for (int i = 0; i < 12; ++i) {
      R* q = out + 2 * ((size_t)i * g.vol + s);
      q[0] = o.c[i / 3][i % 3].re;
      q[1] = o.c[i / 3][i % 3].im;
    }
  }
}

}  // namespace

extern "C" {

// u: [4][9][V] complex. Returns 1 and fills the outputs if the field has a fixed-point scale, else 0.
// err_fx / err_f64: per component, distance from the extended-precision value.
int dslash_check(const int* dims, int t_bc, double m_w, double mu, int g5in, const double* u, const double* psi,
                 double* out_fx, double* out_f64, double* err_fx, double* err_f64, int* usable) {
  const Geom g = geom(dims, t_bc);
  double lo = 1e308, hi = 0;
  for (int mu_ = 0; mu_ < 4; ++mu_)
    for (int s = 0; s < g.vol; ++s) {
      Mat3<double> m;
      for (int k = 0; k < 9; ++k) {
        const double* q = u + 2 * (((size_t)mu_ * 9 + k) * g.vol + s);
        m.m[k / 3][k % 3] = mk<double>(q[0], q[1]);
      }
      double top, need;
      fx_link_range(m, top, need);
      lo = top < lo ? top : lo;
      hi = need > hi ? need : hi;
    }
  int uexp;
  if (!fx_field_scale(lo, hi, &uexp)) return 0;
  std::vector<FxC> fx((size_t)36 * g.vol);
  for (size_t e = 0; e < fx.size(); ++e) fx[e] = fx_link_entry(mk<double>(u[2 * e], u[2 * e + 1]), uexp);
  run(g, m_w, mu, fx.data(), uexp, psi, g5in, out_fx, usable);
  plain<double>(g, m_w, mu, u, psi, g5in, out_f64);
  std::vector<long double> ref((size_t)24 * g.vol);
  plain<long double>(g, m_w, mu, u, psi, g5in, ref.data());
  for (size_t i = 0; i < ref.size(); ++i) {
    err_fx[i] = (double)std::fabs(out_fx[i] - ref[i]);
    err_f64[i] = (double)std::fabs(out_f64[i] - ref[i]);
  }
  return 1;
}

}
