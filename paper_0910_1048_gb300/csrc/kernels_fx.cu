// The FP64 direct method's Lanczos step with its vectors in fixed point (fixedpt.cuh).
//
// GB300's FP64 pipe (about two lanes per SM and clock) bound every kernel of the FP64 step: the pair
// stencil at 12^4 took 84 us and the update 24.5 us against 4.2 and 4.8 us of HBM time. Here the
// recurrence vectors vhat_j, vhat_{j-1}, what_j, what_{j-1} are kept as limbs with one exponent per site
// (59 bits of the site's largest component, so at least as much as FP64 holds of it), and both the
// stencil and the update are integer arithmetic: products of limbs by mad.wide.s32, sums in 64 bits.
// FP64 is left for the basis columns (one conversion per component), the step's scalars and the sums
// over blocks. Every sum inside a block is an integer sum with one rounding per term, so the
// results do not depend on the shape or the order of the launch.
//
// Step j:
//   k_fx_pair:   A v = H(mu) vhat_j / k, A w = H(-mu) what_j / k (k = the hop coefficient ks times the links'
//                scale; unscaled otherwise), normalised per site, and the chunk sums of what_j^H (A v)
//   k_fx_update: alpha_j from the chunk sums; vhat_{j+1}, what_{j+1} in place of vhat_{j-1}, what_{j-1}, the
//                basis column in FP64, and the chunk sums of what^H vhat, |vhat|^2, |what|^2
//   k_fx_settle: delta_j, beta_j, the next scales (behind the next pair stencil, which needs none of them)
#include "devutil.cuh"
#include "kernels.h"
#include "lzscalars.cuh"

namespace ovl {

// (h 2^30 + l) from a 60-bit value.
__device__ __forceinline__ void fx_split(fx64 q, int& h, int& l) {
  h = (int)(q >> 30);
  l = (int)((unsigned)q & 0x3fffffffu);
}

__device__ __forceinline__ fx64 fx_sar_round(fx64 v, int n) {  // v >> n to nearest, n in [0, 62]
  return n > 0 ? (v + ((fx64)1 << (n - 1))) >> n : v;
}

// v 2^k: on the exponent where the result is normal.
__device__ __forceinline__ double fx_scalb(double v, int k) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  const int e = (int)(b >> 52) & 0x7ff;
  if (e != 0 && e + k > 0 && e + k < 0x7ff)
    return __longlong_as_double((long long)(b + ((unsigned long long)(long long)k << 52)));
  const int k1 = max(-1000, min(1000, k / 2)), k2 = max(-1000, min(1000, k - k1));
  return v * fx_pow2(1023 + k1) * fx_pow2(1023 + k2);
}

// Largest high word of |v| over a set of values (the site's normalisation): see fx_norm_shift.
__device__ __forceinline__ int fx_top(int m, fx64 v) {
  const int w = (int)(v >> 32);
  return max(m, w ^ (w >> 31));
}
// Shift that takes values whose largest high word is m to at most 2^59: right if positive, left if not.
__device__ __forceinline__ int fx_norm_shift(int m) { return 5 - __clz(m); }  // (32 - clz) + 32 - 59
__device__ __forceinline__ fx64 fx_normalise(fx64 v, int r) { return r > 0 ? fx_sar_round(v, r) : v << -r; }

// Product of two complex numbers in limbs, T = H + (X >> 30), in units of 2^-58 of their scales' product.
// CONJ: conj(a) b.
template <bool CONJ>
__device__ __forceinline__ void fx_cmul(const FxC& a, const FxC& b, fx64& re, fx64& im) {
  const int ih = CONJ ? -a.ih : a.ih, il = CONJ ? -a.il : a.il, nh = -ih, nl = -il;
  fx64 hr = fx_mul(a.rh, b.rh), hi = fx_mul(a.rh, b.ih), xr = fx_mul(a.rh, b.rl), xi = fx_mul(a.rh, b.il);
  fx_mad(hr, nh, b.ih);
  fx_mad(hi, ih, b.rh);
  fx_mad(xr, a.rl, b.rh);
  fx_mad(xi, a.rl, b.ih);
  fx_mad(xr, nh, b.il);
  fx_mad(xi, ih, b.rl);
  fx_mad(xr, nl, b.ih);
  fx_mad(xi, il, b.rh);
  re = hr + (xr >> 30);
  im = hi + (xi >> 30);
}
__device__ __forceinline__ fx64 fx_rmul(int ah, int al, int bh, int bl) {
  fx64 x = fx_mul(ah, bl);
  fx_mad(x, al, bh);
  return fx_mul(ah, bh) + (x >> 30);
}

// ------------------------------------------------------------------ chunk sums
// A chunk is 32 consecutive sites (a warp). Its sum: the sites' values aligned to the chunk's largest
// exponent with five bits of headroom, each rounded once; stored as an integer and that exponent.
constexpr int kFxNone = -(1 << 28);  // exponent of a value that is not there

__device__ __forceinline__ fx64 warp_sum(fx64 v) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  return v;
}
__device__ __forceinline__ fx64 fx_align(fx64 v, int d) { return fx_sar_round(v, min(d, 61)); }

// Partials of a rhs inside its part block: alpha sums (re, im), the update's four sums, and their exponents.
struct FxParts {
  longlong2* a;  // [nchunk]
  fx64* u;       // [4][nchunk]
  int* ae;       // [nchunk]
  int* ue;       // [4][nchunk]
};
__device__ __forceinline__ FxParts fx_parts(const LzDev& lz, int rhs, int nchunk) {
  char* p = (char*)(lz.part + (size_t)rhs * lz.nblk * 4);
  FxParts f;
  f.a = (longlong2*)p;
  f.u = (fx64*)(p + (size_t)nchunk * 16);
  f.ae = (int*)(p + (size_t)nchunk * 48);
  f.ue = f.ae + nchunk;
  return f;
}

// ------------------------------------------------------------------ start
// vhat_1 (basis column 1) and what_1 (FP64, in `w1`) to limbs in slot 1. One thread per site.
__global__ void __launch_bounds__(64) k_fx_begin(Geom g, LzDev lz, FxVecs fx, const double2* vh, const double2* w1) {
  const int rhs = blockIdx.y, s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= g.vol) return;
  const size_t n = (size_t)12 * g.vol;
#pragma unroll 1
  for (int role = 0; role < 2; ++role) {
    const double2* in = role ? w1 + (size_t)rhs * n : vh + (size_t)rhs * lz.vcols * n;
    Spin<double> p;
    StrideLoader{in, 1, g.vol}(s, p);
    const int e = max(fx_exponent(p), 64);
    FxSpin q;
    fx_spin(p, e, q);
    FxC* out = (role ? fx.w[1] : fx.v[1]) + (size_t)rhs * n;
#pragma unroll
    for (int i = 0; i < 12; ++i)
      out[(size_t)i * g.vol + s] = FxC{q.rh[i / 3][i % 3], q.rl[i / 3][i % 3], q.ih[i / 3][i % 3], q.il[i / 3][i % 3]};
    (role ? fx.ew[1] : fx.ev[1])[(size_t)rhs * g.vol + s] = e;
  }
}

// ------------------------------------------------------------------ pair stencil
// Block (32 sites, 2 T): warp y computes the hops of role y / T (0: H(mu) vhat_j, 1: H(-mu) what_j) whose
// index is in [8 t / T, 8 (t+1) / T), t = y % T. T = 1: one thread per site and role; T = 4: one direction
// per thread, for lattices too small to fill the GPU with one (each thread finishes one spin).
struct FxSelf {
  int h, l, e;  // 1 / ks = (h 2^30 + l) 2^-59 2^e
};

template <int T>
__global__ void __launch_bounds__(64 * T, T == 1 ? 6 : 1)
    k_fx_pair(Geom g, Links U, FxCoef cp, FxCoef cm, FxSelf self, LzDev lz, FxVecs fx) {
  const int rhs = blockIdx.y;
  const int lane = threadIdx.x, role = threadIdx.y / T, t = threadIdx.y % T;
  // launched early behind k_fx_settle (programmatic dependent launch): status and j are final since the
  // update, and the step's scalars are not used here, so the only wait is the one at the end
  const bool run = lz.status[rhs] == 0;
  const int j = lz.j[rhs];
  const int s = blockIdx.x * 32 + lane;
  const bool live = run && s < g.vol;
  const size_t n = (size_t)12 * g.vol;
  const FxCoef& c = role ? cm : cp;
  const FxC* q = (role ? fx.w : fx.v)[j & 1] + (size_t)rhs * n;
  const int* ex = (role ? fx.ew : fx.ev)[j & 1] + (size_t)rhs * g.vol;
  FxAcc acc;
  fx_clear(acc);
  int E = 0, es = 0;
  const int se = self.e - U.fxf->uexp;  // exponent of the diagonal's coefficient
  if (live) {
    const unsigned long long xyzt = fx_coords(g, s);
    es = ex[s];
    int en[8];
    bool wraps;
#pragma unroll
    for (int k = 0; k < 8; ++k) en[k] = ex[fx_neighbour(g, s, xyzt, k, &wraps)];
    // the diagonal's scale is at most 2^5 of the hops': |A| < 2^61.8 units
    E = es + se - 3;
#pragma unroll
    for (int k = 0; k < 8; ++k) E = max(E, fx_hop_exponent(k, en[k], c));
#pragma unroll 1
    for (int k = t * (8 / T); k < (t + 1) * (8 / T); ++k) {
      const int nb = fx_neighbour(g, s, xyzt, k, &wraps);
      const int eh = fx_hop_exponent(k, ex[nb], c);
      FxHalf h;
      {
        FxSpin p;
#pragma unroll
        for (int i = 0; i < 12; ++i) {
          const FxC x = q[(size_t)i * g.vol + nb];
          p.rh[i / 3][i % 3] = x.rh;
          p.rl[i / 3][i % 3] = x.rl;
          p.ih[i / 3][i % 3] = x.ih;
          p.il[i / 3][i % 3] = x.il;
        }
        fx_half(k, p, false, h);
      }
      fx_hop(k, E - eh, h, U.fx + (size_t)(k >> 1) * 9 * g.vol + ((k & 1) ? nb : s), (size_t)g.vol, c,
             wraps && g.t_bc < 0, acc);
    }
  }
  // the diagonal psi / ks, and gamma5: A of spin sp
  auto finish = [&](int sp, fx64 (&ar)[3], fx64 (&ai)[3]) {
    const int sh = E - es - se + 3;  // from units of 2^-59 2^(es + se - 1022)
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const FxC x = q[(size_t)(sp * 3 + a) * g.vol + s];
      fx64 xr = fx_mul(x.rh, self.l), xi = fx_mul(x.ih, self.l);
      fx_mad(xr, x.rl, self.h);
      fx_mad(xi, x.il, self.h);
      ar[a] += fx_align(2 * fx_mul(x.rh, self.h) + (xr >> 29), sh);
      ai[a] += fx_align(2 * fx_mul(x.ih, self.h) + (xi >> 29), sh);
      if (sp >= 2) ar[a] = -ar[a], ai[a] = -ai[a];
    }
  };
  // normalised A of spin sp to HBM; what_j^H (A v) of the spin in units of 2^-58
  FxC* out = (role ? fx.aw : fx.av) + (size_t)rhs * n;
  auto emit = [&](int sp, int r, const fx64 (&ar)[3], const fx64 (&ai)[3], fx64& dr, fx64& di) {
    const FxC* w = fx.w[j & 1] + (size_t)rhs * n;
    fx64 hr = 0, hi = 0, xr = 0, xi = 0;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      FxC y;
      fx_split(fx_normalise(ar[a], r), y.rh, y.rl);
      fx_split(fx_normalise(ai[a], r), y.ih, y.il);
      out[(size_t)(sp * 3 + a) * g.vol + s] = y;
      if (role == 0) {
        const FxC x = w[(size_t)(sp * 3 + a) * g.vol + s];
        const int nh = -x.ih, nl = -x.il;  // conj(what)
        fx_mad(hr, x.rh, y.rh);
        fx_mad(hr, x.ih, y.ih);
        fx_mad(hi, x.rh, y.ih);
        fx_mad(hi, nh, y.rh);
        fx_mad(xr, x.rh, y.rl);
        fx_mad(xr, x.rl, y.rh);
        fx_mad(xr, x.ih, y.il);
        fx_mad(xr, x.il, y.ih);
        fx_mad(xi, x.rh, y.il);
        fx_mad(xi, x.rl, y.ih);
        fx_mad(xi, nh, y.rl);
        fx_mad(xi, nl, y.rh);
      }
    }
    dr = hr + (xr >> 30);
    di = hi + (xi >> 30);
  };
  fx64 dr = 0, di = 0;
  int de = kFxNone;
  if constexpr (T == 1) {
    if (live) {
      int m = 0;
#pragma unroll
      for (int sp = 0; sp < 4; ++sp) {
        finish(sp, acc.re[sp], acc.im[sp]);
#pragma unroll
        for (int a = 0; a < 3; ++a) m = fx_top(fx_top(m, acc.re[sp][a]), acc.im[sp][a]);
      }
      const int r = fx_norm_shift(m), ea = E + r + 3;
#pragma unroll
      for (int sp = 0; sp < 4; ++sp) {
        fx64 x, y;
        emit(sp, r, acc.re[sp], acc.im[sp], x, y);
        dr += x;
        di += y;
      }
      (role ? fx.eaw : fx.eav)[(size_t)rhs * g.vol + s] = ea;
      if (role == 0) de = ea + fx.ew[j & 1][(size_t)rhs * g.vol + s];
    }
  } else {
    // each thread keeps its own direction's part of spin t and hands the other spins over
    __shared__ fx64 part[2][3][12][2][32];  // [role][slot of the contributing thread][component][re, im][site]
    __shared__ int top[2][4][32];
    __shared__ fx64 dot[4][2][32];
    if (live) {
#pragma unroll
      for (int sp = 0; sp < 4; ++sp)
        if (sp != t)
#pragma unroll
          for (int a = 0; a < 3; ++a) {
            part[role][t < sp ? t : t - 1][sp * 3 + a][0][lane] = acc.re[sp][a];
            part[role][t < sp ? t : t - 1][sp * 3 + a][1][lane] = acc.im[sp][a];
          }
    }
    __syncthreads();
    fx64 ar[3] = {0, 0, 0}, ai[3] = {0, 0, 0};
    if (live) {
#pragma unroll
      for (int sp = 0; sp < 4; ++sp)
        if (sp == t)
#pragma unroll
          for (int a = 0; a < 3; ++a) {
            ar[a] = acc.re[sp][a] + part[role][0][sp * 3 + a][0][lane] + part[role][1][sp * 3 + a][0][lane] +
                    part[role][2][sp * 3 + a][0][lane];
            ai[a] = acc.im[sp][a] + part[role][0][sp * 3 + a][1][lane] + part[role][1][sp * 3 + a][1][lane] +
                    part[role][2][sp * 3 + a][1][lane];
          }
      finish(t, ar, ai);
      int m = 0;
#pragma unroll
      for (int a = 0; a < 3; ++a) m = fx_top(fx_top(m, ar[a]), ai[a]);
      top[role][t][lane] = m;
    }
    __syncthreads();
    if (live) {
      const int m = max(max(top[role][0][lane], top[role][1][lane]), max(top[role][2][lane], top[role][3][lane]));
      const int r = fx_norm_shift(m), ea = E + r + 3;
      fx64 x, y;
      emit(t, r, ar, ai, x, y);
      if (role == 0) {
        dot[t][0][lane] = x;
        dot[t][1][lane] = y;
      }
      if (t == 0) {
        (role ? fx.eaw : fx.eav)[(size_t)rhs * g.vol + s] = ea;
        if (role == 0) de = ea + fx.ew[j & 1][(size_t)rhs * g.vol + s];
      }
    }
    __syncthreads();
    if (role == 0 && t == 0 && live) {
      dr = dot[0][0][lane] + dot[1][0][lane] + dot[2][0][lane] + dot[3][0][lane];
      di = dot[0][1][lane] + dot[1][1][lane] + dot[2][1][lane] + dot[3][1][lane];
    }
  }
  if (role == 0 && t == 0 && run) {  // the chunk's sum
    const int em = __reduce_max_sync(0xffffffffu, de), d = em - de + 5;
    dr = warp_sum(fx_align(dr, d));
    di = warp_sum(fx_align(di, d));
    if (lane == 0) {
      const FxParts f = fx_parts(lz, rhs, gridDim.x);
      f.a[blockIdx.x] = make_longlong2(dr, di);
      f.ae[blockIdx.x] = em + 5;
    }
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");  // the settle kernel has finished before this one does
}

// ------------------------------------------------------------------ sums over chunks
// Sums of NV values over the chunk partials: value v of chunk c is t(v, c) 2^e(v, c). Every thread of the
// block takes chunks tid, tid + nthreads, ...; the terms are aligned to the largest exponent and added
// as two words, exactly. Results (sum hi, sum lo with 2^31 between them, exponent) in all lanes of warp 0.
struct FxSum {
  fx64 hi, lo;
  int e;
  __device__ __forceinline__ double get(int k) const {  // (hi 2^31 + lo) 2^(e + k)
    return fx_scalb(fma((double)hi, 2147483648.0, (double)lo), e + k);
  }
};

template <int NV, class LoadT, class LoadE>
__device__ __forceinline__ void fx_sum_chunks(int nchunk, LoadT tv, LoadE ev, FxSum (&out)[NV]) {
  __shared__ int se[NV][32];
  __shared__ fx64 sh[NV][2][32];
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
  fx64 t0[NV];
  int e0[NV], em[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) {  // the first chunk's values: one round trip for most lattices
    t0[v] = tid < nchunk ? tv(v, tid) : 0;
    em[v] = e0[v] = tid < nchunk ? ev(v, tid) : kFxNone;
  }
  for (int c = tid + nt; c < nchunk; c += nt)
#pragma unroll
    for (int v = 0; v < NV; ++v) em[v] = max(em[v], ev(v, c));
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    em[v] = __reduce_max_sync(0xffffffffu, em[v]);
    if (lane == 0) se[v][warp] = em[v];
  }
  __syncthreads();
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    em[v] = __reduce_max_sync(0xffffffffu, lane < nw ? se[v][lane] : kFxNone);
    fx64 a = fx_align(t0[v], em[v] - e0[v]);
    fx64 hi = a >> 31, lo = a & 0x7fffffff;
    for (int c = tid + nt; c < nchunk; c += nt) {
      a = fx_align(tv(v, c), em[v] - ev(v, c));
      hi += a >> 31;
      lo += a & 0x7fffffff;
    }
    hi = warp_sum(hi);
    lo = warp_sum(lo);
    if (lane == 0) sh[v][0][warp] = hi, sh[v][1][warp] = lo;
  }
  __syncthreads();
  if (warp == 0)
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      out[v].hi = warp_sum(lane < nw ? sh[v][0][lane] : 0);
      out[v].lo = warp_sum(lane < nw ? sh[v][1][lane] : 0);
      out[v].e = em[v];
    }
}

// ------------------------------------------------------------------ update
// One block per SM, block b taking the chunks [nchunk b / G, nchunk (b+1) / G); a group of four warps per
// chunk, warp sp of the group its spin sp. Groups synchronise by themselves (named barriers).
// Every block forms the coefficients from the pair stencil's chunk sums (a microsecond, instead of a
// one-block kernel between the two). The block that takes the last ticket at the start (every block
// has read j by then) advances j and marks the step pending for k_fx_settle.
constexpr int kFxGroups = 5;  // chunks in flight per block (96 registers a thread)

struct FxCoefSh {
  FxC c;
  int e;
};

__device__ __forceinline__ void group_sync(int grp) { asm volatile("bar.sync %0, 128;" ::"r"(grp + 1) : "memory"); }

template <bool STORE, bool XACC>
__global__ void __launch_bounds__(128 * kFxGroups, 1)
    k_fx_update(Geom g, double ks, const FxField* fxf, LzDev lz, FxVecs fx, double2* vh) {
  const int rhs = blockIdx.y;
  if (lz.status[rhs]) return;
  __shared__ int jsh;
  __shared__ FxCoefSh cs[6];
  __shared__ fx64 dots[kFxGroups][4][4][32];
  __shared__ int tops[kFxGroups][2][4][32];
  const int tid = threadIdx.x, lane = tid & 31;
  if (tid == 0) {
    jsh = lz.j[rhs];
    __threadfence();  // this block's read of j completes before its ticket
    if (atomicAdd(lz.count + rhs, 1u) == gridDim.x - 1) {
      lz.count[rhs] = 0u;
      lz.j[rhs] = jsh + 1;
      lz.pending[rhs] = 1;
    }
  }
  __syncthreads();
  const int j = jsh;
  const int nchunk = (g.vol + 31) >> 5;
  const size_t n = (size_t)12 * g.vol, o = (size_t)rhs * (lz.kmax + 2);
  const FxParts parts = fx_parts(lz, rhs, nchunk);
  {
    // warp 0, one coefficient per lane (lanes 0..5: A v, vhat_j, vhat_{j-1}, A w, what_j, what_{j-1}; 6: alpha_j)
    zd p = mk(0.0, 0.0), q = mk(0.0, 0.0);
    if (tid < 32) {
      const double kse = fx_scalb(ks, fxf->uexp), sv = lz.sv[o + j];
      const zd sw = ldc<double>(lz.sw, o + j);
      const zd k1 = (sv * kse) * conj(sw);  // alpha_j = k1 (sum of what^H A v)
      if (lane == 0) p = mk(sv, 0.0), q = mk(kse, 0.0);
      if (lane == 1) p = -(sv * k1);
      if (lane == 2 && j > 1) p = mk(-lz.sv[o + j - 1], 0.0), q = ldc<double>(lz.beta, o + j - 1);
      if (lane == 3) p = sw, q = mk(kse, 0.0);
      if (lane == 4) p = -(sw * conj(k1));
      if (lane == 5 && j > 1) p = mk(-lz.delta[o + j - 1], 0.0), q = ldc<double>(lz.sw, o + j - 1);
      if (lane == 6) p = k1;
    }
    FxSum sum[2];
    fx_sum_chunks<2>(
        nchunk, [&](int v, int c) { return v ? parts.a[c].y : parts.a[c].x; }, [&](int, int c) { return parts.ae[c]; }, sum);
    if (tid < 7) {
      const zd al = mk(sum[0].get(-58 - 2044), sum[1].get(-58 - 2044));
      if (lane == 1 || lane == 6) q = al;
      if (lane == 4) q = conj(al);
      const zd r = p * q;
      if (lane < 6) {
        int hr, hi;
        unsigned lr, li;
        fx_words(r.re, hr, lr);
        fx_words(r.im, hi, li);
        const int e = max(max(hr & 0x7fffffff, hi & 0x7fffffff) >> 20, 64);
        FxCoefSh& d = cs[lane];
        fx_limbs(hr, lr, e, d.c.rh, d.c.rl);
        fx_limbs(hi, li, e, d.c.ih, d.c.il);
        d.e = r.re == 0.0 && r.im == 0.0 ? kFxNone : e;  // (the vectors before the first may hold anything)
      } else if (blockIdx.x == 0) {
        lz.alpha[o + j] = make_double2(r.re, r.im);
      }
    }
    __syncthreads();
  }
  const int grp = tid >> 7, sp = (tid >> 5) & 3;
  const int ngrp = blockDim.x >> 7;
  const int c0 = (int)((long long)nchunk * blockIdx.x / gridDim.x), c1 = (int)((long long)nchunk * (blockIdx.x + 1) / gridDim.x);
  const zd xc = XACC ? ldc<double>(lz.xcoef, o + j + 1) : mk(0.0, 0.0);
#pragma unroll 1
  for (int ch = c0 + grp; ch < c1; ch += ngrp) {
    const bool live = ch * 32 + lane < g.vol;
    const int s = live ? ch * 32 + lane : g.vol - 1;  // (a lane past the end reads the chunk's last site)
    const size_t base = (size_t)rhs * n + (size_t)sp * 3 * g.vol + s;
    const size_t es = (size_t)rhs * g.vol + s;
    FxC nv[2][3];  // new limbs of vhat and what
    int en[2];
#pragma unroll
    for (int role = 0; role < 2; ++role) {
      const FxC* A = (role ? fx.aw : fx.av) + base;
      const FxC* V = (role ? fx.w : fx.v)[j & 1] + base;
      FxC* P = (role ? fx.w : fx.v)[(j + 1) & 1] + base;  // column j-1, overwritten
      int* pe = (role ? fx.ew : fx.ev)[(j + 1) & 1] + es;
      const FxCoefSh& k0 = cs[3 * role];
      const FxCoefSh& k1 = cs[3 * role + 1];
      const FxCoefSh& k2 = cs[3 * role + 2];
      const bool prev = k2.e != kFxNone;
      // biased exponents of the three products
      const int e0 = (role ? fx.eaw : fx.eav)[es] + k0.e - 1022, e1 = (role ? fx.ew : fx.ev)[j & 1][es] + k1.e - 1022;
      const int e2 = prev ? *pe + k2.e - 1022 : kFxNone;
      const int E = max(max(e0, e1), e2);
      fx64 x[3][2];
      int m = 0;
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const FxC va = A[(size_t)a * g.vol], vv = V[(size_t)a * g.vol];
        const FxC vp = prev ? P[(size_t)a * g.vol] : FxC{0, 0, 0, 0};
        fx64 r, i;
        if (role == 0) {  // a real coefficient
          r = fx_rmul(k0.c.rh, k0.c.rl, va.rh, va.rl);
          i = fx_rmul(k0.c.rh, k0.c.rl, va.ih, va.il);
        } else {
          fx_cmul<false>(k0.c, va, r, i);
        }
        fx64 xr = fx_align(r, E - e0), xi = fx_align(i, E - e0);
        fx_cmul<false>(k1.c, vv, r, i);
        xr += fx_align(r, E - e1);
        xi += fx_align(i, E - e1);
        fx_cmul<false>(k2.c, vp, r, i);
        xr += fx_align(r, E - e2);
        xi += fx_align(i, E - e2);
        x[a][0] = xr;
        x[a][1] = xi;
        m = fx_top(fx_top(m, xr), xi);
      }
      tops[grp][role][sp][lane] = m;
      group_sync(grp);
      m = max(max(tops[grp][role][0][lane], tops[grp][role][1][lane]),
              max(tops[grp][role][2][lane], tops[grp][role][3][lane]));
      const int r = fx_norm_shift(m);
      en[role] = E + r + 1;
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const fx64 qr = fx_normalise(x[a][0], r), qi = fx_normalise(x[a][1], r);
        FxC y;
        fx_split(qr, y.rh, y.rl);
        fx_split(qi, y.ih, y.il);
        nv[role][a] = y;
        if (live) {
          P[(size_t)a * g.vol] = y;
          if (role == 0 && (STORE || XACC)) {
            const zd d = mk(fx_scalb((double)qr, en[0] - 1022 - 59), fx_scalb((double)qi, en[0] - 1022 - 59));
            const size_t at = (size_t)(sp * 3 + a) * g.vol + s;
            if (STORE) stc<double>(vh, ((size_t)rhs * lz.vcols + j) * n + at, d);  // column j + 1
            if (XACC) {
              double2* xa = lz.xacc + (size_t)rhs * n;
              stc<double>(xa, at, ldc<double>(xa, at) + xc * d);
            }
          }
        }
      }
      if (live && sp == 0) *pe = en[role];
    }
    // what^H vhat, |vhat|^2, |what|^2 of this spin
    fx64 h[4] = {0, 0, 0, 0}, xx[4] = {0, 0, 0, 0};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const FxC x = nv[0][a], y = nv[1][a];
      const int nh = -y.ih, nl = -y.il;
      fx_mad(h[0], y.rh, x.rh);
      fx_mad(h[0], y.ih, x.ih);
      fx_mad(xx[0], y.rh, x.rl);
      fx_mad(xx[0], y.rl, x.rh);
      fx_mad(xx[0], y.ih, x.il);
      fx_mad(xx[0], y.il, x.ih);
      fx_mad(h[1], y.rh, x.ih);
      fx_mad(h[1], nh, x.rh);
      fx_mad(xx[1], y.rh, x.il);
      fx_mad(xx[1], y.rl, x.ih);
      fx_mad(xx[1], nh, x.rl);
      fx_mad(xx[1], nl, x.rh);
      fx_mad(h[2], x.rh, x.rh);
      fx_mad(h[2], x.ih, x.ih);
      fx_mad(xx[2], x.rh, x.rl);
      fx_mad(xx[2], x.ih, x.il);
      fx_mad(h[3], y.rh, y.rh);
      fx_mad(h[3], y.ih, y.ih);
      fx_mad(xx[3], y.rh, y.rl);
      fx_mad(xx[3], y.ih, y.il);
    }
    dots[grp][sp][0][lane] = h[0] + (xx[0] >> 30);
    dots[grp][sp][1][lane] = h[1] + (xx[1] >> 30);
    dots[grp][sp][2][lane] = h[2] + (xx[2] >> 29);
    dots[grp][sp][3][lane] = h[3] + (xx[3] >> 29);
    group_sync(grp);
    {  // warp v of the group sums value v over the chunk
      const int v = sp;
      const fx64 d = dots[grp][0][v][lane] + dots[grp][1][v][lane] + dots[grp][2][v][lane] + dots[grp][3][v][lane];
      const int e = !live ? kFxNone : v < 2 ? en[0] + en[1] : 2 * en[v - 2];
      const int em = __reduce_max_sync(0xffffffffu, e);
      const fx64 t = warp_sum(live ? fx_align(d, em - e + 5) : 0);
      if (lane == 0) {
        parts.u[(size_t)v * nchunk + ch] = t;
        parts.ue[(size_t)v * nchunk + ch] = em + 5;
      }
    }
    group_sync(grp);  // dots and tops are free again
  }
}

// ------------------------------------------------------------------ settle
constexpr int kFxSettle = 512;

__global__ void __launch_bounds__(kFxSettle) k_fx_settle(LzDev lz, int nchunk) {
  asm volatile("griddepcontrol.launch_dependents;");  // the pair stencil that follows may start
  const int rhs = blockIdx.y;
  __shared__ int go, jsh;
  if (threadIdx.x == 0) {
    go = lz.pending[rhs] && !lz.status[rhs];
    jsh = lz.j[rhs];
  }
  __syncthreads();
  if (!go) return;
  const int j = jsh;
  const FxParts f = fx_parts(lz, rhs, nchunk);
  FxSum sum[4];
  fx_sum_chunks<4>(
      nchunk, [&](int v, int c) { return f.u[(size_t)v * nchunk + c]; },
      [&](int v, int c) { return f.ue[(size_t)v * nchunk + c]; }, sum);
  if (threadIdx.x == 0) {
    const double sums[4] = {sum[0].get(-58 - 2044), sum[1].get(-58 - 2044), sum[2].get(-58 - 2044),
                            sum[3].get(-58 - 2044)};
    const BetaVals b = lz_beta_vals(sums);
    lz_beta_store(lz, rhs, (size_t)rhs * (lz.kmax + 2), j - 1, b);
    if (!b.ok) lz.j[rhs] = j - 1;
    lz.pending[rhs] = 0;
  }
}

// ------------------------------------------------------------------ launches
static FxSelf fx_self(double ks) {
  FxSelf s;
  const double m = std::frexp(1.0 / ks, &s.e);
  const fx64 q = std::llrint(std::ldexp(m, 59));
  s.h = (int)(q >> 30);
  s.l = (int)(q & ((1 << 30) - 1));
  return s;
}

bool fx_step_usable(double m_w, double mu) {
  const FxCoef c = fx_coef(m_w, mu);
  const double k = std::fabs(c.k.ks);
  return c.ok && k >= 0x1p-10 && k <= 0x1p10;
}

cudaError_t launch_fx_begin(const Geom& g, const LzDev& lz, const FxVecs& fx, const void* vh, const void* w1,
                            cudaStream_t st) {
  return launch_plain(k_fx_begin, dim3((g.vol + 63) / 64, lz.nrhs), dim3(64), st, g, lz, fx, (const double2*)vh,
                      (const double2*)w1);
}

cudaError_t launch_fx_settle(const Geom& g, const LzDev& lz, cudaStream_t st) {
  return launch_plain(k_fx_settle, dim3(1, lz.nrhs), dim3(kFxSettle), st, lz, (g.vol + 31) >> 5);
}

cudaError_t launch_fx_pair(const Geom& g, const Links& U, double m_w, double mu, const LzDev& lz, const FxVecs& fx,
                           cudaStream_t st, int variant, cudaEvent_t mid, cudaEvent_t first) {
  cudaError_t e;
  if ((e = launch_fx_settle(g, lz, st))) return e;
  if (first && (e = record_timing(first, st))) return e;
  const FxCoef cp = fx_coef(m_w, mu), cm = fx_coef(m_w, -mu);
  const bool split = variant == 1 || variant == 4 || variant == 5;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((g.vol + 31) / 32, lz.nrhs);
  cfg.blockDim = dim3(32, split ? 8 : 2);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  if (!first) {  // (a timing event between the two kernels orders them anyway)
    cfg.attrs = attr;
    cfg.numAttrs = 1;
  }
  e = split ? cudaLaunchKernelEx(&cfg, k_fx_pair<4>, g, U, cp, cm, fx_self(cp.k.ks), lz, fx)
            : cudaLaunchKernelEx(&cfg, k_fx_pair<1>, g, U, cp, cm, fx_self(cp.k.ks), lz, fx);
  if (e == cudaSuccess && mid) e = record_timing(mid, st);
  return e;
}

cudaError_t launch_fx_update(const Geom& g, const Links& U, double m_w, const LzDev& lz, const FxVecs& fx, void* vh,
                             cudaStream_t st, cudaEvent_t mid) {
  int dev = 0, nsm = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  const int nchunk = (g.vol + 31) >> 5;
  const int nb = std::min(nsm, nchunk);
  const int grp = std::min(kFxGroups, (nchunk + nb - 1) / nb);
  const dim3 grid(nb, lz.nrhs), block(128 * grp);
  const double ks = hop_coef<double>(m_w, 0.0).ks;
  const bool store = fx.store != 0, xacc = lz.xacc != nullptr;
  e = xacc    ? launch_plain(k_fx_update<false, true>, grid, block, st, g, ks, U.fxf, lz, fx, (double2*)vh)
      : store ? launch_plain(k_fx_update<true, false>, grid, block, st, g, ks, U.fxf, lz, fx, (double2*)vh)
              : launch_plain(k_fx_update<false, false>, grid, block, st, g, ks, U.fxf, lz, fx, (double2*)vh);
  if (e == cudaSuccess && mid) e = record_timing(mid, st);
  return e;
}

}  // namespace ovl
