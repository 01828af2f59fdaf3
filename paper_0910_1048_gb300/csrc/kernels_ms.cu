// Multishift BiCG kernels (Algorithm 3 on M = A^2, A = H_W(mu); Section 5's rational sign).
//
// One iteration k is three launches:
//   pair1:  t = A p,  t~ = A^H p~  (A^H = H_W(-mu));  alpha_k = rho / (t~^H t - s1 p~^H p);
//           last block: zeta^i_{k+1}, alpha^i_k for every live shift
//   pair2:  r -= alpha_k q, q = A t - s1 p = (M - s1) p;  r~ -= conj(alpha_k) q~, q~ = A^H t~ - s1 p~;
//           rho' = r~^H r, |r|; last block: beta_k = rho'/rho, beta^i_k = beta_k (zeta^i_{k+1}/zeta^i_k)^2,
//           shifts with |zeta^i_{k+1}| |r| <= tol |r_0| are retired after this step
//   dirs:   X += sum_i omega_i alpha^i_k p^i;  p^i = zeta^i_{k+1} r + beta^i_k p^i;
//           p = r + beta_k p,  p~ = r~ + conj(beta_k) p~
// The shifted recurrences follow from the BiCG residual polynomials: r_k = R_k(M0) r_0 with
// R_{k+1}(t) = (1 + a_k b_{k-1}/a_{k-1} - a_k t) R_k(t) - (a_k b_{k-1}/a_{k-1}) R_{k-1}(t), and the
// residual of (M0 - d) x = r_0 in the same Krylov space is R_k(d)^-1 r_k, i.e. zeta = 1/R_k(d).
#include "devutil.cuh"
#include "kernels.h"

namespace ovl {

template <class R>
__device__ __forceinline__ size_t voff(int rhs, size_t n) { return (size_t)rhs * n; }

// start: r = b - R L^H b, r~ = b - L R^H b, x_P; p = r, p~ = r~, p^i = r, X = 0
template <class R>
__global__ void __launch_bounds__(kBlock) k_ms_start(Geom g, MsDev ms, MsVecs v, const double2* b, int m,
                                                     const double2* Rv, const double2* Lv, const double* lam_sign,
                                                     const double2* dots) {
  using T = typename V2<R>::T;
  const int rhs = blockIdx.y;
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  const size_t n = (size_t)12 * g.vol;
  double acc[4] = {0, 0, 0, 0};
  if (s < g.vol) {
    const double2* dr = dots + (size_t)rhs * 2 * m;
    for (int c = 0; c < 12; ++c) {
      zd bv = ldc<double>(b, (size_t)rhs * n + (size_t)s * 12 + c);
      zd r = bv, rt = bv, x = mk(0.0, 0.0);
      for (int i = 0; i < m; ++i) {
        zd ci = ldc<double>(dr, i), di = ldc<double>(dr, m + i);
        zd ri = ldc<double>(Rv, (size_t)i * n + (size_t)c * g.vol + s);
        zd li = ldc<double>(Lv, (size_t)i * n + (size_t)c * g.vol + s);
        r = r - ci * ri;
        x = x + lam_sign[i] * (ci * ri);
        rt = rt - di * li;
      }
      const size_t e = voff<R>(rhs, n) + (size_t)c * g.vol + s;
      if (v.xp) stc<double>(v.xp, e, x);
      if (v.r64) stc<double>(v.r64, e, r);
      if (v.xs)
        for (int i = 0; i < ms.s; ++i) stc<double>(v.xs, ((size_t)rhs * ms.s + i) * n + (size_t)c * g.vol + s, mk(0.0, 0.0));
      stc<double>(v.X, e, mk(0.0, 0.0));
      cplx<R> rr = mk<R>((R)r.re, (R)r.im), rtt = mk<R>((R)rt.re, (R)rt.im);
      stc<R>((T*)v.r, e, rr);
      stc<R>((T*)v.p, e, rr);
      stc<R>((T*)v.rt, e, rtt);
      stc<R>((T*)v.pt, e, rtt);
      if (v.ps)
        for (int i = 0; i < ms.s; ++i) stc<R>((T*)v.ps, ((size_t)rhs * ms.s + i) * n + (size_t)c * g.vol + s, rr);
      // rho and |r| from the stored (rounded) vectors, so the recurrences start consistent
      zd rd = mk((double)rr.re, (double)rr.im), rtd = mk((double)rtt.re, (double)rtt.im);
      zd ip = cdot(rtd, rd);
      acc[0] += ip.re;
      acc[1] += ip.im;
      acc[2] += norm2(rd);
    }
  }
  block_sum<4>(acc);
  double* part = ms.part + (size_t)rhs * ms.nblk * 4;
  if (publish_partials<4>(acc, part, ms.count + rhs)) {
    reduce_partials<4>(part, gridDim.x, acc);
    const int t = lin_tid();
    double2* sd = ms.seed + (size_t)rhs * 8;
    if (t == 0) {
      double rn = sqrt(acc[2]);
      sd[0] = make_double2(acc[0], acc[1]);  // rho
      sd[1] = make_double2(0, 0);
      sd[2] = make_double2(1, 0);  // alpha_{-1}
      sd[3] = make_double2(0, 0);  // beta_{-1}
      sd[4] = make_double2(rn, rn);
      sd[5] = make_double2(0, 0);
      ms.k[rhs] = 0;
      ms.status[rhs] = acc[2] == 0.0 ? 3 : ((acc[0] != 0.0 || acc[1] != 0.0) ? 0 : 1);
    }
    for (int i = t; i < ms.s; i += lin_nthreads()) {
      double2* z = ms.zeta + ((size_t)rhs * ms.s + i) * 3;
      z[0] = z[1] = z[2] = make_double2(1, 0);
      ms.active[(size_t)rhs * ms.s + i] = 1;
      ms.ash[(size_t)rhs * ms.s + i] = make_double2(0, 0);
      ms.bsh[(size_t)rhs * ms.s + i] = make_double2(0, 0);
    }
  }
}

// Every FP64 instruction is slow on GB300's narrow FP64 pipe, so the last blocks' recurrences keep
// their dependent chains short (one division per shift, comparisons on squares). Blocks have at
// least as many threads as shifts (s <= 127), so thread t holds shift t.
struct MsAlphaIn {
  zd rho, akm, bkm;  // rho_k, alpha_{k-1}, beta_{k-1}
  int act;           // shift t: 0 retired, 1 live, 2 last direction update done
  zd zm, z0;         // zeta^t_{k-1}, zeta^t_k
  double dsig;       // sigma_t - sigma_1
};

__device__ __forceinline__ MsAlphaIn ms_alpha_inputs(const MsDev& ms, int rhs) {
  MsAlphaIn in{};
  const double2* sd = ms.seed + (size_t)rhs * 8;
  const int t = lin_tid();
  in.rho = ldc<double>(sd, 0);
  in.akm = ldc<double>(sd, 2);
  in.bkm = ldc<double>(sd, 3);
  if (t < ms.s) {
    const size_t si = (size_t)rhs * ms.s + t;
    in.act = ms.active[si];
    const double2* z = ms.zeta + si * 3;
    in.zm = ldc<double>(z, 0);
    in.z0 = ldc<double>(z, 1);
    in.dsig = ms.dsig[t];
  }
  return in;
}

// last block of pair1: alpha_k, then zeta^i_{k+1} and alpha^i_k of the live shifts
__device__ __forceinline__ void ms_alpha_and_shifts(MsDev& ms, int rhs, const double (&pv)[4], const MsAlphaIn& in) {
  __shared__ zd alpha_sh;
  __shared__ int bad;
  const int t = lin_tid();
  double2* sd = ms.seed + (size_t)rhs * 8;
  if (t == 0) {
    zd den = mk(pv[0], pv[1]);
    double dd = norm2(den);
    bad = !(dd > 0.0) || !(dd < 1e300);
    zd alpha = bad ? mk(0.0, 0.0) : (1.0 / dd) * (in.rho * conj(den));
    alpha_sh = alpha;
    if (bad) ms.status[rhs] = 1;
    sd[1] = make_double2(alpha.re, alpha.im);
  }
  __syncthreads();
  if (bad) return;
  const zd ak = alpha_sh, akm = in.akm, bkm = in.bkm;
  for (int i = t; i < ms.s; i += lin_nthreads()) {
    const size_t si = (size_t)rhs * ms.s + i;
    double2* z = ms.zeta + si * 3;
    const bool mine = i == t;
    int act = mine ? in.act : ms.active[si];
    if (act == 2) ms.active[si] = act = 0;
    if (!act) continue;
    const zd zm = mine ? in.zm : ldc<double>(z, 0), z0 = mine ? in.z0 : ldc<double>(z, 1);
    const double ds = mine ? in.dsig : ms.dsig[i];
    zd d1 = mk(1.0 - ak.re * ds, -ak.im * ds);
    zd den = akm * zm * d1 + ak * bkm * (zm - z0);
    zd num = z0 * zm * akm;
    const double dn = norm2(den), z0n = norm2(z0);
    const zd nc = num * conj(den);
    zd zp = mk(0.0, 0.0), ai = mk(0.0, 0.0);
    const double prod = dn * z0n;
    if (prod > 1e-300 && prod < 1e300) {  // zeta^i_{k+1} = num / den, alpha^i_k = alpha_k zeta^i_{k+1} / zeta^i_k
      const double inv = 1.0 / prod;
      zp = (z0n * inv) * nc;
      ai = ak * (inv * (nc * conj(z0)));
    } else {  // the same with one division each (a product outside the safe range)
      if (dn > 0) zp = (1.0 / dn) * nc;
      if (z0n > 0) ai = ak * ((1.0 / z0n) * (zp * conj(z0)));
    }
    z[2] = make_double2(zp.re, zp.im);
    ms.ash[si] = make_double2(ai.re, ai.im);
  }
}

struct MsBetaIn {
  double tol, r0;
  zd rho, z1, z2;  // rho_k, zeta^t_k, zeta^t_{k+1}
  int act;
};
__device__ __forceinline__ MsBetaIn ms_beta_inputs(const MsDev& ms, int rhs) {
  MsBetaIn in{};
  const double2* sd = ms.seed + (size_t)rhs * 8;
  const int t = lin_tid();
  in.tol = ms.tolv ? ms.tolv[rhs] : ms.tol;
  in.rho = ldc<double>(sd, 0);
  in.r0 = sd[4].x;
  if (t < ms.s) {
    const size_t si = (size_t)rhs * ms.s + t;
    in.act = ms.active[si];
    in.z1 = ldc<double>(ms.zeta + si * 3, 1);
    in.z2 = ldc<double>(ms.zeta + si * 3, 2);
  }
  return in;
}

// last block of pair2: rho_{k+1} and |r_{k+1}| (pv), beta_k, the shifts' beta^i_k and states
__device__ __forceinline__ void ms_beta_and_status(MsDev& ms, int rhs, const double (&pv)[4], const MsBetaIn& in) {
  const int t = lin_tid();
  double2* sd = ms.seed + (size_t)rhs * 8;
  __shared__ zd beta_sh;
  __shared__ double r2_sh;
  __shared__ int live;
  if (t == 0) {
    zd rhon = mk(pv[0], pv[1]);
    double rr = norm2(in.rho);
    zd beta = rr > 0 ? (1.0 / rr) * (rhon * conj(in.rho)) : mk(0.0, 0.0);
    double rn = sqrt(pv[2]);
    beta_sh = beta;
    r2_sh = pv[2];
    live = 0;
    sd[0] = make_double2(rhon.re, rhon.im);
    sd[2] = sd[1];  // alpha_{k-1} <- alpha_k
    sd[3] = make_double2(beta.re, beta.im);
    sd[5] = make_double2(beta.re, beta.im);
    sd[4].y = rn;
    ms.k[rhs] += 1;
    // breakdown of the BiCG recurrence (rho' = 0 while r is not small) or non-finite values
    if (!(rn < 1e300) || !(norm2(rhon) < 1e300) || (norm2(rhon) == 0.0 && rn > in.tol * sd[4].x))
      ms.status[rhs] = 1;
  }
  __syncthreads();
  const zd beta = beta_sh;
  const double r2 = r2_sh, lim = (in.tol * in.r0) * (in.tol * in.r0);
  int mylive = 0;
  for (int i = t; i < ms.s; i += lin_nthreads()) {
    const size_t si = (size_t)rhs * ms.s + i;
    const bool mine = i == t;
    if (!(mine ? in.act : ms.active[si])) continue;
    double2* z = ms.zeta + si * 3;
    const zd z0 = mine ? in.z1 : ldc<double>(z, 1), zp = mine ? in.z2 : ldc<double>(z, 2);
    double z0n = norm2(z0);
    zd ratio = z0n > 0 ? (1.0 / z0n) * (zp * conj(z0)) : mk(0.0, 0.0);
    zd bi = beta * (ratio * ratio);
    ms.bsh[si] = make_double2(bi.re, bi.im);
    z[0] = make_double2(z0.re, z0.im);
    z[1] = make_double2(zp.re, zp.im);
    if (norm2(zp) * r2 <= lim)  // |zeta^i_{k+1}| |r_{k+1}| <= tol |r_0|, on squares
      ms.active[si] = 2;  // this step's direction update is its last
    else
      mylive = 1;
  }
  if (mylive) atomicOr(&live, 1);
  __syncthreads();
  if (t == 0 && !live && ms.status[rhs] == 0) ms.status[rhs] = 4;
}

// pair1 (MODE 0): t = A p, t~ = A^H p~, and the denominator of alpha: with q = (A^2 - s1) p,
// p~^H q = t~^H t - s1 p~^H p, so alpha is known before q is.
// pair2 (MODE 1): r -= alpha (A t - s1 p), r~ -= conj(alpha) (A^H t~ - s1 p~) as q comes out of the stencil, and
// rho' = r~^H r, |r|^2. The two roles of a site (p and p~ side) exchange components through shared memory for
// the products and share their float-float sums: the p side takes |r|^2 and colour 0, the other the rest.
// With the denominator from q itself, q and q~ were written here and read back by a kernel of their own: 22 vector
// passes a step in a correction instead of 18, and 16^4, 4 sources, 20 poles took 636 ms instead of 555 (FP32 with
// 5 blocks per SM, 96 registers; 738 at 228 registers, 561 at 80).
template <class R, int MODE>
struct MsPairSum {
  static constexpr int kValues = MODE == 0 ? 2 : 3;
  Red<R> acc[kValues];
  __device__ __forceinline__ void dot(cplx<R> y, cplx<R> x) {  // y^H x
    acc[0].dot2(y.re, x.re, y.im, x.im);
    acc[1].dot2(y.re, x.im, -y.im, x.re);
  }
  // The block's sums published, and the last block's share of the recurrence. (Its inputs are loaded after
  // the sum: held across it they cost the whole stencil kernel registers, 80 -> 106, and occupancy.)
  __device__ __forceinline__ void finish(MsDev& ms, int rhs) {
    double tot[kValues];
    block_reduce<R, kValues>(acc, tot);
    double* part = ms.part + (size_t)rhs * ms.nblk * 4;
    double pv[4] = {tot[0], tot[1], MODE == 0 ? 0.0 : tot[kValues - 1], 0.0};
    if (publish_partials<4>(pv, part, ms.count + rhs)) {
      reduce_partials<4>(part, gridDim.x, pv);
      if (MODE == 0)
        ms_alpha_and_shifts(ms, rhs, pv, ms_alpha_inputs(ms, rhs));
      else
        ms_beta_and_status(ms, rhs, pv, ms_beta_inputs(ms, rhs));
    }
  }
};

template <class R, int LF, int MODE, class Coef>
__global__ void __launch_bounds__(2 * kPairSites, std::is_same_v<Coef, FxCoef> ? 3 : sizeof(R) == 8 ? 1 : 5)
    k_ms_pair(Geom g, Links U, Coef cp, Coef cm, MsDev ms, MsVecs v) {
  using T = typename V2<R>::T;
  __shared__ cplx<R> xch[12][kPairSites];
  const int rhs = blockIdx.y;
  if (MODE == 0 && blockIdx.x == 0 && lin_tid() == 0 && ms.status[rhs] == 4) ms.status[rhs] = 2;
  if (ms.status[rhs] != 0) return;
  const size_t n = (size_t)12 * g.vol;
  const int tx = threadIdx.x, s = blockIdx.x * kPairSites + tx;
  const bool is_t = threadIdx.y == 1, live = s < g.vol;
  const T* in = (const T*)(MODE == 0 ? (is_t ? v.pt : v.p) : (is_t ? v.tt : v.t)) + voff<R>(rhs, n);
  const T* p = (const T*)v.p + voff<R>(rhs, n);
  const T* pt = (const T*)v.pt + voff<R>(rhs, n);
  const double s1d = ms.sig1v ? ms.sig1v[rhs] : ms.sigma1;
  R s1v[1], akv[2];
  scalars_in<R, 1>(&s1d, s1v);
  if (MODE == 1) scalars_in<R, 2>((const double*)(ms.seed + (size_t)rhs * 8 + 1), akv);
  const R s1 = s1v[0];
  MsPairSum<R, MODE> sum;
  cplx<R> x[12];
  if (live) {
    Spin<R> o;
    stencil_site<LF, R>(g, U, s, is_t ? cm : cp, in, o);
#pragma unroll
    for (int c = 0; c < 12; ++c) x[c] = c >= 6 ? -o.c[c / 3][c % 3] : o.c[c / 3][c % 3];  // gamma5
    if constexpr (MODE == 0) {
      T* out = (T*)(is_t ? v.tt : v.t) + voff<R>(rhs, n);
      if (is_t) {
        if (s1 != (R)0) {
          cplx<R> a = mk<R>(0, 0);
#pragma unroll
          for (int c = 0; c < 12; ++c)
            a = a + cdot(ldc<R>(pt, (size_t)c * g.vol + s), ldc<R>(p, (size_t)c * g.vol + s));
          sum.acc[0].add(-s1 * a.re);
          sum.acc[1].add(-s1 * a.im);
        }
#pragma unroll
        for (int c = 0; c < 12; ++c) xch[c][tx] = x[c];
      }
#pragma unroll
      for (int c = 0; c < 12; ++c) stc<R>(out, (size_t)c * g.vol + s, x[c]);
    } else {
      const cplx<R> ak = mk<R>(akv[0], is_t ? -akv[1] : akv[1]);
      const T* pp = is_t ? pt : p;
      T* r = (T*)(is_t ? v.rt : v.r) + voff<R>(rhs, n);
      // every load before the first store (stores that might alias would otherwise serialise twelve
      // memory round trips)
      cplx<R> pv[12], rv[12];
#pragma unroll
      for (int c = 0; c < 12; ++c) {
        pv[c] = ldc<R>(pp, (size_t)c * g.vol + s);
        rv[c] = ldc<R>(r, (size_t)c * g.vol + s);
      }
#pragma unroll
      for (int c = 0; c < 12; ++c) {
        x[c] = cmsub(rv[c], ak, x[c] - s1 * pv[c]);
        stc<R>(r, (size_t)c * g.vol + s, x[c]);
        if (is_t == (c % 3 == 0)) xch[c][tx] = x[c];
      }
    }
  }
  __syncthreads();
  if (live) {
    if constexpr (MODE == 0) {
      if (!is_t) {
        cplx<R> a = mk<R>(0, 0);
#pragma unroll
        for (int c = 0; c < 12; ++c) a = a + cdot(xch[c][tx], x[c]);
        sum.acc[0].add(a.re);
        sum.acc[1].add(a.im);
      }
    } else if (is_t) {
#pragma unroll
      for (int c = 0; c < 12; ++c)
        if (c % 3 != 0) sum.dot(x[c], xch[c][tx]);
    } else {
#pragma unroll
      for (int c = 0; c < 12; ++c) {
        if (c % 3 == 0) sum.dot(xch[c][tx], x[c]);
        sum.acc[2].dot2(x[c].re, x[c].re, x[c].im, x[c].im);
      }
    }
  }
  sum.finish(ms, rhs);
}

// The same with eight threads per site (pair_split): each thread finishes one spin of its site.
template <class R, int LF, int MODE, class Coef>
__global__ void __launch_bounds__(8 * kSplitSites) k_ms_pair_split(Geom g, Links U, Coef cp, Coef cm, MsDev ms, MsVecs v) {
  using T = typename V2<R>::T;
  __shared__ SplitSmem<R> sm;
  __shared__ cplx<R> xch[12][kSplitSites];
  const int rhs = blockIdx.y;
  if (MODE == 0 && blockIdx.x == 0 && lin_tid() == 0 && ms.status[rhs] == 4) ms.status[rhs] = 2;
  if (ms.status[rhs] != 0) return;
  const size_t n = (size_t)12 * g.vol;
  const T* in0 = (const T*)(MODE == 0 ? v.p : v.t) + voff<R>(rhs, n);
  const T* in1 = (const T*)(MODE == 0 ? v.pt : v.tt) + voff<R>(rhs, n);
  const T* p = (const T*)v.p + voff<R>(rhs, n);
  const T* pt = (const T*)v.pt + voff<R>(rhs, n);
  const double s1d = ms.sig1v ? ms.sig1v[rhs] : ms.sigma1;
  R s1v[1], akv[2];
  scalars_in<R, 1>(&s1d, s1v);
  if (MODE == 1) scalars_in<R, 2>((const double*)(ms.seed + (size_t)rhs * 8 + 1), akv);
  const R s1 = s1v[0];
  MsPairSum<R, MODE> sum;
  cplx<R> x[3];
  pair_split<R, LF, Coef>(g, U, cp, cm, in0, in1, sm, [&](int which, int s, int sp, cplx<R> (&o)[3]) {
    const R g5 = sp >= 2 ? (R)-1 : (R)1;
    if constexpr (MODE == 0) {
      T* out = (T*)(which ? v.tt : v.t) + voff<R>(rhs, n);
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const size_t e = (size_t)(sp * 3 + a) * g.vol + s;
        x[a] = g5 * o[a];
        if (which) {
          if (s1 != (R)0) sum.dot(-s1 * ldc<R>(pt, e), ldc<R>(p, e));
          xch[sp * 3 + a][threadIdx.x] = x[a];
        }
        stc<R>(out, e, x[a]);
      }
    } else {
      const cplx<R> ak = mk<R>(akv[0], which ? -akv[1] : akv[1]);
      const T* pp = which ? pt : p;
      T* r = (T*)(which ? v.rt : v.r) + voff<R>(rhs, n);
      cplx<R> pv[3], rv[3];  // loads first (see k_ms_pair)
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        pv[a] = ldc<R>(pp, (size_t)(sp * 3 + a) * g.vol + s);
        rv[a] = ldc<R>(r, (size_t)(sp * 3 + a) * g.vol + s);
      }
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        x[a] = cmsub(rv[a], ak, g5 * o[a] - s1 * pv[a]);
        stc<R>(r, (size_t)(sp * 3 + a) * g.vol + s, x[a]);
        if ((which == 1) == (a == 0)) xch[sp * 3 + a][threadIdx.x] = x[a];
      }
    }
  });
  __syncthreads();
  if (blockIdx.x * kSplitSites + threadIdx.x < g.vol) {
    const int which = threadIdx.y >> 2, c0 = (threadIdx.y & 3) * 3;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const cplx<R> y = xch[c0 + a][threadIdx.x];
      if constexpr (MODE == 0) {
        if (!which) sum.dot(y, x[a]);
      } else {
        if (which && a != 0) sum.dot(x[a], y);
        if (!which && a == 0) sum.dot(y, x[a]);
        if (!which) sum.acc[2].dot2(x[a].re, x[a].re, x[a].im, x[a].im);
      }
    }
  }
  sum.finish(ms, rhs);
}

// dirs: X += sum_i omega_i alpha^i p^i; p^i = zeta^i r + beta^i p^i; p, p~ updates.
// FP64 kernels accumulate X term by term in double. FP32 kernels sum the iteration's terms
// over the shifts in float-float and add that sum to the FP64 X once (the FP64 pipe is 1/64 of
// the FP32 rate); with per-shift solutions kept (refinement), x^(i) is held in float-float
// (re hi, re lo, im hi, im lo: the 16 bytes of a complex double) during the pass, so the
// increments alpha^i p^i need no FP64 arithmetic; it is converted to FP64 in place afterwards.
// XS: per-shift solutions kept (v.xs set), a compile-time choice so that neither path's
// instructions are issued predicated-off in the other (predicated-off FP64 instructions still hold
// the FP64 pipe).
template <class R, bool XS>
__global__ void __launch_bounds__(kVecBlock) k_ms_dirs(Geom g, MsDev ms, MsVecs v) {
  using T = typename V2<R>::T;
  const int rhs = blockIdx.y;
  const int st = ms.status[rhs];
  if (st != 0 && st != 4) return;
  const size_t n = (size_t)12 * g.vol;
  const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;  // one vector element per thread
  // the shift coefficients in the kernel's own precision (FP32 kernels convert them once per
  // block here, not per element: a double -> float conversion runs on the FP64 pipe)
  using T2 = typename V2<R>::T;
  __shared__ T2 coefx[kMaxShifts], coefz[kMaxShifts], coefb[kMaxShifts], coefa[kMaxShifts];
  __shared__ int act[kMaxShifts];
  for (int i = threadIdx.x; i < ms.s; i += blockDim.x) {
    const size_t si = (size_t)rhs * ms.s + i;
    act[i] = ms.active[si];
    const zd ai = ldc<double>(ms.ash, si);
    const double2 z = ms.zeta[si * 3 + 1], b = ms.bsh[si];  // zeta_{k+1} after the rotation in update
    coefa[i].x = (R)ai.re;
    coefa[i].y = (R)ai.im;
    coefx[i].x = (R)(ms.omega[i] * ai.re);
    coefx[i].y = (R)(ms.omega[i] * ai.im);
    coefz[i].x = (R)z.x;
    coefz[i].y = (R)z.y;
    coefb[i].x = (R)b.x;
    coefb[i].y = (R)b.y;
  }
  __syncthreads();
  R bkr[2];
  scalars_in<R, 2>((const double*)(ms.seed + (size_t)rhs * 8 + 5), bkr);
  if (e >= n) return;
  const cplx<R> b = mk<R>(bkr[0], bkr[1]), bc = mk<R>(bkr[0], -bkr[1]);
  const T* r = (const T*)v.r + voff<R>(rhs, n);
  const T* rt = (const T*)v.rt + voff<R>(rhs, n);
  T* p = (T*)v.p + voff<R>(rhs, n);
  T* pt = (T*)v.pt + voff<R>(rhs, n);
  T* ps = (T*)v.ps + (size_t)rhs * ms.s * n;
  double2* X = v.X + voff<R>(rhs, n);
  {
    const cplx<R> rv = ldc<R>(r, e);
    zd xa = XS ? mk(0.0, 0.0) : ldc<double>(X, e);  // X is not used when x^(i) are kept
    Red<R> sre, sim;  // FP32: this iteration's sum over the shifts
    for (int i = 0; i < ms.s; ++i) {
      if (!act[i]) continue;
      T* pi = ps + (size_t)i * n;
      const cplx<R> pv = ldc<R>(pi, e);
      if constexpr (XS) {  // keep x^(i) itself: x^(i) += alpha^i p^i
        const T2 ca = coefa[i];
        if constexpr (sizeof(R) == 8) {
          double2* xi = v.xs + ((size_t)rhs * ms.s + i) * n;
          stc<double>(xi, e, ldc<double>(xi, e) + mk(ca.x, ca.y) * pv);
        } else {
          float4* xi = reinterpret_cast<float4*>(v.xs + ((size_t)rhs * ms.s + i) * n);
          const cplx<R> inc = mk<R>(ca.x, ca.y) * pv;
          float4 x4 = xi[e];
          const FF re = ff_add(FF{x4.x, x4.y}, FF{inc.re, 0.f}), im = ff_add(FF{x4.z, x4.w}, FF{inc.im, 0.f});
          xi[e] = make_float4(re.hi, re.lo, im.hi, im.lo);
        }
      } else {
        const T2 cx = coefx[i];
        if constexpr (sizeof(R) == 8) {
          xa = xa + mk(cx.x, cx.y) * pv;
        } else {
          const cplx<R> c = mk<R>(cx.x, cx.y);
          sre.add(fma(c.re, pv.re, -(c.im * pv.im)));
          sim.add(fma(c.re, pv.im, c.im * pv.re));
        }
      }
      if (act[i] == 1) {
        const T2 cz = coefz[i], cb = coefb[i];
        cplx<R> nv = mk<R>(cz.x, cz.y) * rv + mk<R>(cb.x, cb.y) * pv;
        stc<R>(pi, e, nv);
      }
    }
    if constexpr (!XS) {
      if constexpr (sizeof(R) == 4) {
        xa.re += sre.get();
        xa.im += sim.get();
      }
      stc<double>(X, e, xa);
    }
    if (st == 0) {
      stc<R>(p, e, rv + b * ldc<R>(p, e));
      stc<R>(pt, e, ldc<R>(rt, e) + bc * ldc<R>(pt, e));
    }
  }
}

// float -> double by its bits (normal numbers; the conversion instruction runs on the FP64 pipe, four of
// whose operations per component bound the kernel below).
__device__ __forceinline__ double widen(float x) {
  const unsigned u = __float_as_uint(x), e = (u >> 23) & 0xffu;
  if (e == 0u || e == 0xffu) return (double)x;
  return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + (896u << 20))), (int)(u << 29));
}

// dirs for one system without shifts (the FP32 corrections of the reliable updates: s = 1, dsig = 0, so
// p^1 = p, alpha^1 = alpha and omega = 1): X += alpha p; p = r + beta p, p~ = r~ + conj(beta) p~. Two elements
// per thread and pass. HBM-bound: 80 bytes an element. The general kernel, which carries p^1 beside p and
// spent eight FP64 operations an element on X, took 526 us on average over the 80 systems of 16^4 (at most a
// third running at a time), this one 249.
constexpr int kSeedBlock = 256, kSeedPasses = 4;
__global__ void __launch_bounds__(kSeedBlock) k_ms_dirs_seed(Geom g, MsDev ms, MsVecs v) {
  const int rhs = blockIdx.y;
  const int st = ms.status[rhs];
  if (st != 0 && st != 4) return;
  const size_t n = (size_t)12 * g.vol;  // a multiple of 192: pairs stay aligned and inside one system
  const double2* sd = ms.seed + (size_t)rhs * 8;
  const double src[4] = {sd[1].x, sd[1].y, sd[5].x, sd[5].y};
  float c[4];
  scalars_in<float, 4>(src, c);
  const float4* r = (const float4*)((const float2*)v.r + voff<float>(rhs, n));
  const float4* rt = (const float4*)((const float2*)v.rt + voff<float>(rhs, n));
  float4* p = (float4*)((float2*)v.p + voff<float>(rhs, n));
  float4* pt = (float4*)((float2*)v.pt + voff<float>(rhs, n));
  double2* X = v.X + voff<float>(rhs, n);
  const cplx<float> al = mk<float>(c[0], c[1]), be = mk<float>(c[2], c[3]), bc = mk<float>(c[2], -c[3]);
#pragma unroll
  for (int q = 0; q < kSeedPasses; ++q) {
    const size_t i = ((size_t)blockIdx.x * kSeedPasses + q) * kSeedBlock + threadIdx.x;
    if (i >= n / 2) break;
    const float4 pv = p[i];
    const cplx<float> p0 = mk<float>(pv.x, pv.y), p1 = mk<float>(pv.z, pv.w);
    const double2 x0 = X[2 * i], x1 = X[2 * i + 1];
    const cplx<float> a0 = al * p0, a1 = al * p1;
    X[2 * i] = make_double2(x0.x + widen(a0.re), x0.y + widen(a0.im));
    X[2 * i + 1] = make_double2(x1.x + widen(a1.re), x1.y + widen(a1.im));
    if (st == 0) {
      const float4 rv = r[i], rtv = rt[i], qv = pt[i];
      const cplx<float> n0 = mk<float>(rv.x, rv.y) + be * p0, n1 = mk<float>(rv.z, rv.w) + be * p1;
      const cplx<float> m0 = mk<float>(rtv.x, rtv.y) + bc * mk<float>(qv.x, qv.y);
      const cplx<float> m1 = mk<float>(rtv.z, rtv.w) + bc * mk<float>(qv.z, qv.w);
      p[i] = make_float4(n0.re, n0.im, n1.re, n1.im);
      pt[i] = make_float4(m0.re, m0.im, m1.re, m1.im);
    }
  }
}

cudaError_t launch_ms_start(const Geom& g, bool f64, const MsDev& ms, const MsVecs& v, const double2* b, int m,
                            const double2* R, const double2* L, const double* lam_sign, double2* dots, cudaStream_t st) {
  dim3 grid((g.vol + kBlock - 1) / kBlock, ms.nrhs);
  if (m > 0) {
    cudaError_t e = launch_defl_dots(g, ms.nrhs, m, b, R, L, ms.part, ms.count, dots, st);
    if (e != cudaSuccess) return e;
  }
  if (f64)
    k_ms_start<double><<<grid, kBlock, 0, st>>>(g, ms, v, b, m, R, L, lam_sign, dots);
  else
    k_ms_start<float><<<grid, kBlock, 0, st>>>(g, ms, v, b, m, R, L, lam_sign, dots);
  return cudaGetLastError();
}

bool ms_pair_split(const Geom& g, int key) {
  const int tv = tuned_pair_variant(g.vol, key);
  return tv < 0 ? use_split(g) : (tv == 1 || tv == 4 || tv == 5);  // 0, 2, 3, 6, 7, 8: one thread per site
}

template <class R, int LF, class Coef>
static cudaError_t ms_step_t(const Geom& g, const Links& U, const Coef& cp, const Coef& cm, const MsDev& ms,
                             const MsVecs& v, cudaStream_t st, cudaEvent_t* ev) {
  dim3 grid(vec_blocks(g), ms.nrhs);
  dim3 pgrid((g.vol + kPairSites - 1) / kPairSites, ms.nrhs), pblock(kPairSites, 2);
  dim3 sgrid((g.vol + kSplitSites - 1) / kSplitSites, ms.nrhs), sblock(kSplitSites, 8);
  const bool split = ms_pair_split(g, sizeof(R) == 8 ? 0 : LF);
  cudaError_t e;
  if (ev && (e = record_timing(ev[0], st))) return e;
  e = split ? launch_plain(k_ms_pair_split<R, LF, 0, Coef>, sgrid, sblock, st, g, U, cp, cm, ms, v)
            : launch_plain(k_ms_pair<R, LF, 0, Coef>, pgrid, pblock, st, g, U, cp, cm, ms, v);
  if (e) return e;
  if (ev && (e = record_timing(ev[1], st))) return e;
  e = split ? launch_plain(k_ms_pair_split<R, LF, 1, Coef>, sgrid, sblock, st, g, U, cp, cm, ms, v)
            : launch_plain(k_ms_pair<R, LF, 1, Coef>, pgrid, pblock, st, g, U, cp, cm, ms, v);
  if (e) return e;
  if (ev && (e = record_timing(ev[2], st))) return e;
  if (sizeof(R) == 4 && ms.s == 1 && ms.sig1v) {  // a correction batch (each system its own shift as the seed)
    const size_t pairs = (size_t)6 * g.vol;
    const unsigned nb = (unsigned)((pairs + (size_t)kSeedBlock * kSeedPasses - 1) / ((size_t)kSeedBlock * kSeedPasses));
    e = launch_plain(k_ms_dirs_seed, dim3(nb, ms.nrhs), dim3(kSeedBlock), st, g, ms, v);
  } else {
    e = v.xs ? launch_plain(k_ms_dirs<R, true>, grid, dim3(kVecBlock), st, g, ms, v)
             : launch_plain(k_ms_dirs<R, false>, grid, dim3(kVecBlock), st, g, ms, v);
  }
  if (e) return e;
  if (ev && (e = record_timing(ev[3], st))) return e;
  return cudaGetLastError();
}

cudaError_t launch_ms_step(const Geom& g, const Links& U, int lf, bool f64, double m_w, double mu, const MsDev& ms,
                           const MsVecs& v, cudaStream_t st, cudaEvent_t* ev) {
  if (f64) {
    // fixed-point hops where the field and the factors fit them; FP64 ones inlined otherwise (their fallback inside
    // the fixed-point kernels: unit links, 12^4 pair1 + pair2 129 us against 107 here)
    const FxCoef cp = fx_coef(m_w, mu), cm = fx_coef(m_w, -mu);
    if (U.fits && cp.ok && cm.ok) return ms_step_t<double, LINK_F64>(g, U, cp, cm, ms, v, st, ev);
    return ms_step_t<double, LINK_F64>(g, U, cp.k, cm.k, ms, v, st, ev);
  }
  const HopCoef<float> cp = hop_coef<float>(m_w, mu), cm = hop_coef<float>(m_w, -mu);
  if (lf == LINK_F16R12) return ms_step_t<float, LINK_F16R12>(g, U, cp, cm, ms, v, st, ev);
  return ms_step_t<float, LINK_F32>(g, U, cp, cm, ms, v, st, ev);
}

__global__ void __launch_bounds__(kVecBlock) k_ms_residual_batch(int vol, int j0, int s, const double2* r64,
                                                                 const double2* t2, const double2* x,
                                                                 const double* sigma, double2* res, double* part,
                                                                 unsigned* count, double* out) {
  const size_t n = (size_t)12 * vol;
  const int j = blockIdx.y, jj = j0 + j, rhs = jj / s, i = jj % s;
  const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  double acc[1] = {0};
  if (e < n) {
    const size_t o = (size_t)j * n + e;
    zd a = ldc<double>(r64, (size_t)rhs * n + e) - (ldc<double>(t2, o) - sigma[i] * ldc<double>(x, o));
    stc<double>(res, o, a);
    acc[0] = norm2(a);
  }
  block_sum<1>(acc);
  if (publish_partials<1>(acc, part + (size_t)j * gridDim.x, count + j)) {
    reduce_partials<1>(part + (size_t)j * gridDim.x, gridDim.x, acc);
    if (lin_tid() == 0) out[j] = acc[0];
  }
}

cudaError_t launch_ms_residual_batch(const Geom& g, int j0, int gn, int s, const double2* r64, const double2* t2,
                                     const double2* x, const double* sigma, double2* res, double* part,
                                     unsigned* count, double* out, cudaStream_t st) {
  dim3 grid(vec_blocks(g), gn);
  k_ms_residual_batch<<<grid, kVecBlock, 0, st>>>(g.vol, j0, s, r64, t2, x, sigma, res, part, count, out);
  return cudaGetLastError();
}

__global__ void k_axpy_f64_masked(size_t n, const int* status, const double2* e, double2* x) {
  const int j = blockIdx.y;
  if (status[j] == 1) return;  // breakdown of this correction solve: keep x_j
  size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) stc<double>(x, (size_t)j * n + i, ldc<double>(x, (size_t)j * n + i) + ldc<double>(e, (size_t)j * n + i));
}

cudaError_t launch_axpy_f64_masked(const Geom& g, int gn, const int* status, const double2* e, double2* x,
                                   cudaStream_t st) {
  size_t n = (size_t)12 * g.vol;
  dim3 grid((unsigned)((n + 255) / 256), gn);
  k_axpy_f64_masked<<<grid, 256, 0, st>>>(n, status, e, x);
  return cudaGetLastError();
}

// Float-float complex (re hi, re lo, im hi, im lo) -> complex double, in place.
__global__ void k_ff_to_f64(size_t n, double2* x) {
  size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float4 f = reinterpret_cast<const float4*>(x)[i];
  x[i] = make_double2((double)f.x + (double)f.y, (double)f.z + (double)f.w);
}

cudaError_t launch_ff_to_f64(size_t n, double2* x, cudaStream_t st) {
  k_ff_to_f64<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(n, x);
  return cudaGetLastError();
}

__global__ void k_ms_combine_shifts(size_t n, int s, const double* omega, const double2* xs, double2* X) {
  const int rhs = blockIdx.y;
  size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  zd a = mk(0.0, 0.0);
  for (int j = 0; j < s; ++j) a = a + omega[j] * ldc<double>(xs, ((size_t)rhs * s + j) * n + i);
  stc<double>(X, (size_t)rhs * n + i, a);
}

cudaError_t launch_ms_combine_shifts(const Geom& g, int nrhs, int s, const double* omega, const double2* xs,
                                     double2* X, cudaStream_t st) {
  size_t n = (size_t)12 * g.vol;
  dim3 grid((unsigned)((n + 255) / 256), nrhs);
  k_ms_combine_shifts<<<grid, 256, 0, st>>>(n, s, omega, xs, X);
  return cudaGetLastError();
}

__global__ void k_ms_finish(int vol, const double2* ax, const double2* xp, double2* x) {
  const size_t n = (size_t)12 * vol;
  const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int rhs = blockIdx.y;
  if (e >= n) return;
  zd a = ldc<double>(ax, (size_t)rhs * n + e);
  if (xp) a = a + ldc<double>(xp, (size_t)rhs * n + e);
  int c = (int)(e / vol), s = (int)(e % vol);
  x[(size_t)rhs * n + (size_t)s * 12 + c] = make_double2(a.re, a.im);
}

cudaError_t launch_ms_finish(const Geom& g, int nrhs, const double2* ax, const double2* xp, double2* x, cudaStream_t st) {
  size_t n = (size_t)12 * g.vol;
  dim3 grid((unsigned)((n + 255) / 256), nrhs);
  k_ms_finish<<<grid, 256, 0, st>>>(g.vol, ax, xp, x);
  return cudaGetLastError();
}

}  // namespace ovl
