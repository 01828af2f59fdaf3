// The FP64 direct method's Lanczos step with its vectors in fixed point (fixedpt.cuh).
//
// GB300's FP64 pipe (about two lanes per SM and clock) bound every kernel of the FP64 step: the pair
// stencil at 12^4 took 84 us and the update 24.5 us against 4.2 and 4.8 us of HBM time. Here the
// recurrence vectors vhat_j, vhat_{j-1}, what_j, what_{j-1} are kept as limbs with one exponent per site
// (59 bits of the site's largest component, 56 where sites share an exponent: in the norm more than FP64
// holds, of a component 2^-m of the largest m bits less), and both the stencil and the update are
// integer arithmetic: products of limbs by mad.wide.s32, sums in 64 bits. FP64 is left for the basis
// columns (one conversion per component), the step's scalars and the sums over blocks. Every sum inside a
// block is an integer sum with one rounding per term, so the results do not depend on the shape or the
// order of the launch.
//
// Step j:
//   k_fx_pair:   A v = H(mu) vhat_j / k, A w = H(-mu) what_j / k (k = the hop coefficient ks times the links'
//                scale; unscaled otherwise), normalised per site, and the chunk sums of what_j^H (A v). It
//                needs none of the step's scalars, so one more block settles the previous step
//                meanwhile: delta, beta, the next scales and the coefficients the update needs
//   k_fx_update: alpha_j from the chunk sums; vhat_{j+1}, what_{j+1} in place of vhat_{j-1}, what_{j-1}, the
//                basis column in FP64, and the chunk sums of what^H vhat, |vhat|^2, |what|^2
// Both are launched early (programmatic dependent launch). Each waits for its predecessor, then lets its
// successor launch; what comes before the wait reads only what the kernel before the predecessor has
// finished (vectors, exponents, links, j).
#include <map>
#include <mutex>

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

// ------------------------------------------------------------------ sums over chunks
// Sum over the chunks c = q 32 + lane, + 32 nshare, ... of t(c) 2^e(c), by one warp: the terms aligned to the
// largest exponent met and added as two words, exactly. In units of 2^k; every lane gets it.
template <class LoadT, class LoadE>
__device__ __forceinline__ double fx_warp_sum_chunks(int nchunk, int q, int nshare, LoadT tv, LoadE ev, int k) {
  const int first = q * 32 + (threadIdx.x & 31), step = 32 * nshare;
  constexpr int NK = 4;  // terms kept in registers: one round trip for most lattices
  fx64 t[NK];
  int e[NK], em = kFxNone;
#pragma unroll
  for (int i = 0; i < NK; ++i) {
    const int c = first + i * step;
    t[i] = c < nchunk ? tv(c) : 0;
    e[i] = c < nchunk ? ev(c) : kFxNone;
  }
#pragma unroll
  for (int i = 0; i < NK; ++i) em = max(em, e[i]);
  for (int c = first + NK * step; c < nchunk; c += step) em = max(em, ev(c));
  em = __reduce_max_sync(0xffffffffu, em);
  fx64 hi = 0, lo = 0;
#pragma unroll
  for (int i = 0; i < NK; ++i) {
    const fx64 a = fx_align(t[i], em - e[i]);
    hi += a >> 31;
    lo += a & 0x7fffffff;
  }
#pragma unroll 4
  for (int c = first + NK * step; c < nchunk; c += step) {
    const fx64 a = fx_align(tv(c), em - ev(c));
    hi += a >> 31;
    lo += a & 0x7fffffff;
  }
  hi = warp_sum(hi);
  lo = warp_sum(lo);
  return fx_scalb(fma((double)hi, 2147483648.0, (double)lo), em + k);
}

// ------------------------------------------------------------------ settle
// A complex coefficient in limbs, |components| < 2^(e - 1022).
struct FxCoefSh {
  FxC c;
  int e;
};
__device__ __forceinline__ FxCoefSh fx_coefficient(zd r) {
  FxCoefSh d;
  int hr, hi;
  unsigned lr, li;
  fx_words(r.re, hr, lr);
  fx_words(r.im, hi, li);
  const int e = max(max(hr & 0x7fffffff, hi & 0x7fffffff) >> 20, 64);
  fx_limbs(hr, lr, e, d.c.rh, d.c.rl);
  fx_limbs(hi, li, e, d.c.ih, d.c.il);
  d.e = r.re == 0.0 && r.im == 0.0 ? kFxNone : e;  // (the vectors before the first may hold anything)
  return d;
}

// What the update of step j needs beside alpha_j (formed where sv_j, sw_j are):
//   vhat_{j+1} = c0 A v + (kv a) vhat_j + c2 vhat_{j-1}, what_{j+1} = c0w A w + (kw conj(a)) what_j + c2w what_{j-1},
//   alpha_j = k1 a, a the sum of what_j^H A v.
struct FxStep {
  FxCoefSh c[4];    // c0, c2, c0w, c2w
  double2 k[3];     // kv, kw, k1
  // largest site exponent of column j of vhat and what, slot j & 1 (see k_fx_update)
  int emax[2][2];
};
size_t fx_step_bytes() { return (sizeof(FxStep) + 255) & ~(size_t)255; }

__device__ __forceinline__ FxStep* fx_step(const FxVecs& fx, int rhs) {
  return (FxStep*)((char*)fx.step + (size_t)rhs * ((sizeof(FxStep) + 255) & ~(size_t)255));
}

// By one warp: lane i < 4 one coefficient, lane 4 the factors of the sum.
__device__ __forceinline__ void fx_step_store(FxStep* st, double kse, double sv, zd sw, double svp, zd bt, double dp,
                                              zd swp) {
  const int lane = threadIdx.x & 31;
  if (lane < 4) {
    const zd p = lane == 0 ? mk(sv, 0.0) : lane == 1 ? mk(-svp, 0.0) : lane == 2 ? sw : mk(-dp, 0.0);
    const zd q = lane == 1 ? bt : lane == 3 ? swp : mk(kse, 0.0);
    st->c[lane] = fx_coefficient(p * q);
  } else if (lane == 4) {
    const zd k1 = (sv * kse) * conj(sw), kv = -(sv * k1), kw = -(sw * conj(k1));
    st->k[0] = make_double2(kv.re, kv.im);
    st->k[1] = make_double2(kw.re, kw.im);
    st->k[2] = make_double2(k1.re, k1.im);
  }
}

// Ends the update of step j - 1 (j has been advanced): its sums, delta, beta, the scales of column j, the
// coefficients of the update of step j. By one block.
__device__ __forceinline__ void fx_settle(const LzDev& lz, const FxVecs& fx, int rhs, int nchunk, double ks,
                                          const FxField* fxf) {
  __shared__ double sh[4][2];
  const int t = lin_tid(), warp = t >> 5, lane = t & 31, nw = lin_nthreads() >> 5;
  const int go = lz.pending[rhs] && !lz.status[rhs];
  const int j = lz.j[rhs];
  const size_t o = (size_t)rhs * (lz.kmax + 2);
  const double svp = j > 1 ? lz.sv[o + j - 1] : 0.0;
  const zd swp = j > 1 ? ldc<double>(lz.sw, o + j - 1) : mk(0.0, 0.0);
  const FxParts f = fx_parts(lz, rhs, nchunk);
  constexpr int nshare = 2;  // per sum, whatever the block: the shares are added in FP64
  if (go)
    for (int i = warp; i < 4 * nshare; i += nw) {
      const int v = i & 3, q = i >> 2;
      const double x = fx_warp_sum_chunks(
          nchunk, q, nshare, [&](int c) { return f.u[(size_t)v * nchunk + c]; },
          [&](int c) { return f.ue[(size_t)v * nchunk + c]; }, -58 - 2044);
      if (lane == 0) sh[v][q] = x;
    }
  __syncthreads();
  if (!go || warp != 0) return;
  double sums[4];
#pragma unroll
  for (int v = 0; v < 4; ++v) {
    sums[v] = sh[v][0];
    for (int q = 1; q < nshare; ++q) sums[v] += sh[v][q];
  }
  const BetaVals b = lz_beta_vals(sums);
  if (b.ok) fx_step_store(fx_step(fx, rhs), fx_scalb(ks, fxf->uexp), b.id, b.swv, svp, b.bt, b.d, swp);
  if (lane == 0) {
    lz_beta_store(lz, rhs, o, j - 1, b);
    if (!b.ok) lz.j[rhs] = j - 1;
    lz.pending[rhs] = 0;
    fx_step(fx, rhs)->emax[0][(j + 1) & 1] = kFxNone;  // column j - 1's, replaced by the next update
    fx_step(fx, rhs)->emax[1][(j + 1) & 1] = kFxNone;
  }
}

constexpr int kFxSettle = 256;
__global__ void __launch_bounds__(kFxSettle) k_fx_settle(LzDev lz, const __grid_constant__ FxVecs fx, int nchunk, double ks,
                                                        const FxField* fxf) {
  fx_settle(lz, fx, blockIdx.y, nchunk, ks, fxf);
}

// ------------------------------------------------------------------ start
// vhat_1 (basis column 1) and what_1 (FP64, in `w1`) to limbs in slot 1. One thread per site.
__global__ void __launch_bounds__(64) k_fx_begin(Geom g, LzDev lz, FxVecs fx, const double2* vh, const double2* w1,
                                                 double ks, const FxField* fxf) {
  const int rhs = blockIdx.y, s = blockIdx.x * blockDim.x + threadIdx.x;
  if (blockIdx.x == 0 && threadIdx.x < 32) {
    if (threadIdx.x < 4) fx_step(fx, rhs)->emax[threadIdx.x >> 1][threadIdx.x & 1] = kFxNone;
    const size_t o = (size_t)rhs * (lz.kmax + 2) + 1;
    fx_step_store(fx_step(fx, rhs), fx_scalb(ks, fxf->uexp), lz.sv[o], ldc<double>(lz.sw, o), 0.0, mk(0.0, 0.0), 0.0,
                  mk(0.0, 0.0));
  }
  if (s >= g.vol) return;
  const size_t n = (size_t)12 * g.vol;
#pragma unroll 1
  for (int role = 0; role < 2; ++role) {
    const double2* in = role ? w1 + (size_t)rhs * n : vh + (size_t)rhs * lz.vcols * n;
    Spin<double> p;
    StrideLoader{in, 1, g.vol}(s, p);
    const int e = max(fx_top_word(p) >> 20, 64);
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
// per thread, for lattices too small to fill the GPU with one (each thread finishes one spin). Block 0
// settles the previous step, block b > 0 takes chunk b - 1. A source that has ended (status above 1:
// retired by the host, or without a Krylov part) costs its blocks' launch: seven beside one at 12^4 take a step from
// 44.9 to 45.7 us, where running their hops took it to 231. Every thread of a block sees such a status alike, since
// only stream work before the step writes it; a breakdown (1) is also written by block 0, and the host retires it.
// (A barrier that caught it at once cost 0.4 us a step; the test before the wait cost 0.7.)
// With 8.5 warps per SM (12^4) the latency of the loads is not hidden by other warps, so a hop's inputs are
// copied to shared memory while the previous one is computed: the neighbour's 12 components per thread,
// and the link's nine once for the two roles; what_j for the dot during the last hop (12^4 step 45.7 -> 44.2 us;
// loaded where it is used, the end of the kernel took 9000 clocks instead of 4000). At 12^4 the pair takes
// 34 us, two 20000-clock warps or three per scheduler. Two threads per site and role, or the last 40 of the 648
// chunks split over twice the warps, were no faster (49.7, 44.5).
struct FxSelf {
  int h, l, e;  // 1 / ks = (h 2^30 + l) 2^-59 2^e
};
struct FxPairArgs {  // indexed by the role
  FxCoef c[2];
  const FxC* q[2][2];  // [role][slot]
  const int* e[2][2];
  FxC* out[2];
  int* eo[2];
};

__device__ __forceinline__ void copy_async(void* smem, const void* gmem) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(smem)), "l"(gmem)
               : "memory");
}
__device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <int T>
struct FxPairSmem {
  FxC q[2][12][64 * T];   // [stage][component][thread]
  FxC u[2][T][9][32];     // [stage][direction set][entry][site]
  fx64 part[T > 1 ? 2 : 1][T > 1 ? T - 1 : 1][12][2][T > 1 ? 32 : 1];  // [role][slot][component][re, im][site]
  int top[2][T][32];
  fx64 dot[T][2][32];
};

template <int T>
__global__ void __launch_bounds__(64 * T, T == 1 ? 5 : 1)
    k_fx_pair(Geom g, Links U, const __grid_constant__ FxPairArgs args, FxSelf self, LzDev lz,
              const __grid_constant__ FxVecs fx, double ks) {
  extern __shared__ __align__(16) unsigned char raw[];
  FxPairSmem<T>& sm = *reinterpret_cast<FxPairSmem<T>*>(raw);
  const int rhs = blockIdx.y;
  if (blockIdx.x == 0) {
    grid_wait();
    grid_launch();
    fx_settle(lz, fx, rhs, gridDim.x - 1, ks, U.fxf);
    return;
  }
  const int chunk = blockIdx.x - 1;
  const int lane = threadIdx.x, role = threadIdx.y / T, t = threadIdx.y % T, tid = lin_tid();
  const bool live = chunk * 32 + lane < g.vol;
  const int s = live ? chunk * 32 + lane : g.vol - 1;  // (a lane past the end repeats the last site)
  const size_t n = (size_t)12 * g.vol;
  const FxCoef& c = args.c[role];
  constexpr int NH = 8 / T;
  const unsigned long long xyzt = fx_coords(g, s);
  auto fetch_link = [&](int k, int nb) {  // the roles share the nine rows
    const FxC* u = U.fx + (size_t)(k >> 1) * 9 * g.vol + ((k & 1) ? nb : s);
#pragma unroll
    for (int i = 0; i < 5; ++i) {
      const int row = role * 5 + i;  // of a backward hop's link, transposed
      if (row < 9) copy_async(&sm.u[k & 1][t][row][lane], u + (size_t)((k & 1) ? (row % 3) * 3 + row / 3 : row) * g.vol);
    }
  };
  bool wraps;
  int nb = fx_neighbour(g, s, xyzt, t * NH, &wraps);
  fetch_link(t * NH, nb);
  grid_wait();
  grid_launch();
  const int status = lz.status[rhs], j = lz.j[rhs];
  if (status > 1 || j == 0) {  // ended before this launch, or broke down at the start (no column 1)
    copy_wait();
    return;
  }
  const FxC* q = args.q[role][j & 1] + (size_t)rhs * n;
  const int* ex = args.e[role][j & 1] + (size_t)rhs * g.vol;
  auto fetch_spinor = [&](int stage, const FxC* p) {
#pragma unroll
    for (int i = 0; i < 12; ++i) copy_async(&sm.q[stage][i][tid], p + (size_t)i * g.vol);
  };
  fetch_spinor(0, q + nb);
  FxAcc acc;
  fx_clear(acc);
  const int se = self.e - U.fxf->uexp;  // exponent of the diagonal's coefficient
  const int es = ex[s], ew = args.e[1][j & 1][(size_t)rhs * g.vol + s];
  // the diagonal's scale is at most 2^2 of the hops': |A| < 2^62.8 units
  int E = es + se - 2;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    bool w;
    E = max(E, fx_hop_exponent(k, ex[fx_neighbour(g, s, xyzt, k, &w)], c));
  }
  const FxC* w = args.q[1][j & 1] + (size_t)rhs * n + s;
#pragma unroll 1
  for (int i = 0; i < NH; ++i) {
    const int k = t * NH + i, eh = fx_hop_exponent(k, ex[nb], c);
    const bool flip = wraps && g.t_bc < 0;
    copy_wait();
    __syncthreads();  // hop k's inputs are there, and the other stage has been read
    if (i + 1 < NH) {
      nb = fx_neighbour(g, s, xyzt, k + 1, &wraps);
      fetch_spinor((i + 1) & 1, q + nb);
      fetch_link(k + 1, nb);
    } else if (T == 1) {  // the site's own components, for the diagonal
      fetch_spinor(0, q + s);
    } else {  // of the thread's spin, and of what_j
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        copy_async(&sm.q[0][a][tid], q + (size_t)(t * 3 + a) * g.vol + s);
        copy_async(&sm.q[0][3 + a][tid], w + (size_t)(t * 3 + a) * g.vol);
      }
    }
    FxHalf h;
    {
      FxSpin p;
#pragma unroll
      for (int r = 0; r < 12; ++r) {
        const FxC x = sm.q[i & 1][r][tid];
        p.rh[r / 3][r % 3] = x.rh;
        p.rl[r / 3][r % 3] = x.rl;
        p.ih[r / 3][r % 3] = x.ih;
        p.il[r / 3][r % 3] = x.il;
      }
      fx_half(k, p, false, h);
    }
    if (T == 1 && i + 1 == NH && role == 0)  // what_j, in the thread's slots of the stage just read
#pragma unroll
      for (int a = 0; a < 12; ++a) copy_async(&sm.q[i & 1][a][tid], w + (size_t)a * g.vol);
    const FxC* u = &sm.u[k & 1][t][0][lane];
    fx_hop(k, E - eh, __any_sync(0xffffffffu, E != eh), h, [&](int a, int b) { return u[(a * 3 + b) * 32]; }, c, flip,
           acc);
  }
  copy_wait();
  // the diagonal psi / ks, and gamma5: A of spin sp
  const int sh = E - es - se + 2;  // from units of 2^-59 2^(es + se - 1022)
  const int shc = min(sh, 61);
  const fx64 half = shc > 0 ? (fx64)1 << (shc - 1) : 0;
  auto finish = [&](int sp, int row, fx64 (&ar)[3], fx64 (&ai)[3]) {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const FxC x = sm.q[0][row + a][tid];
      fx64 xr = fx_mad_to(x.rh, self.l, (fx64)1 << 28), xi = fx_mad_to(x.ih, self.l, (fx64)1 << 28);
      fx_mad(xr, x.rl, self.h);
      fx_mad(xi, x.il, self.h);
      ar[a] += fx_sar(2 * fx_mul(x.rh, self.h) + (xr >> 29) + half, shc);
      ai[a] += fx_sar(2 * fx_mul(x.ih, self.h) + (xi >> 29) + half, shc);
      if (sp >= 2) ar[a] = -ar[a], ai[a] = -ai[a];
    }
  };
  // normalised A of spin sp to HBM; what_j^H (A v) of the spin in units of 2^-58
  FxC* out = args.out[role] + (size_t)rhs * n;
  auto emit = [&](int sp, int r, const fx64 (&ar)[3], const fx64 (&ai)[3], fx64& dr, fx64& di) {
    const int rr = max(r, 0), rl = max(-r, 0);
    const fx64 hn = rr > 0 ? (fx64)1 << (rr - 1) : 0;
    fx64 hr = 0, hi = 0, xr = 0, xi = 0;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      FxC y;
      fx_split(((ar[a] + hn) >> rr) << rl, y.rh, y.rl);
      fx_split(((ai[a] + hn) >> rr) << rl, y.ih, y.il);
      if (live) out[(size_t)(sp * 3 + a) * g.vol + s] = y;
      if (role == 0) {
        const FxC x = T == 1 ? sm.q[(NH - 1) & 1][sp * 3 + a][tid] : sm.q[0][3 + a][tid];
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
  int ea;
  if constexpr (T == 1) {
    int m = 0;
#pragma unroll
    for (int sp = 0; sp < 4; ++sp) {
      finish(sp, sp * 3, acc.re[sp], acc.im[sp]);
#pragma unroll
      for (int a = 0; a < 3; ++a) m = fx_top(fx_top(m, acc.re[sp][a]), acc.im[sp][a]);
    }
    const int r = fx_norm_shift(m);
    ea = E + r + 2;
#pragma unroll
    for (int sp = 0; sp < 4; ++sp) {
      fx64 x, y;
      emit(sp, r, acc.re[sp], acc.im[sp], x, y);
      dr += x;
      di += y;
    }
  } else {
    // each thread keeps its own direction's part of spin t and hands the other spins over
#pragma unroll
    for (int sp = 0; sp < 4; ++sp)
      if (sp != t)
#pragma unroll
        for (int a = 0; a < 3; ++a) {
          sm.part[role][t < sp ? t : t - 1][sp * 3 + a][0][lane] = acc.re[sp][a];
          sm.part[role][t < sp ? t : t - 1][sp * 3 + a][1][lane] = acc.im[sp][a];
        }
    __syncthreads();
    fx64 ar[3] = {0, 0, 0}, ai[3] = {0, 0, 0};
#pragma unroll
    for (int sp = 0; sp < 4; ++sp)
      if (sp == t)
#pragma unroll
        for (int a = 0; a < 3; ++a) ar[a] = acc.re[sp][a], ai[a] = acc.im[sp][a];
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
      for (int p = 0; p < T - 1; ++p) {
        ar[a] += sm.part[role][p][t * 3 + a][0][lane];
        ai[a] += sm.part[role][p][t * 3 + a][1][lane];
      }
    finish(t, 0, ar, ai);
    int m = 0;
#pragma unroll
    for (int a = 0; a < 3; ++a) m = fx_top(fx_top(m, ar[a]), ai[a]);
    sm.top[role][t][lane] = m;
    __syncthreads();
#pragma unroll
    for (int p = 0; p < T; ++p) m = max(m, sm.top[role][p][lane]);
    const int r = fx_norm_shift(m);
    ea = E + r + 2;
    fx64 x, y;
    emit(t, r, ar, ai, x, y);
    if (role == 0) {
      sm.dot[t][0][lane] = x;
      sm.dot[t][1][lane] = y;
    }
    __syncthreads();
    if (role == 0 && t == 0)
#pragma unroll
      for (int p = 0; p < T; ++p) {
        dr += sm.dot[p][0][lane];
        di += sm.dot[p][1][lane];
      }
  }
  if (live && t == 0) args.eo[role][(size_t)rhs * g.vol + s] = ea;
  if (role == 0 && t == 0) {  // the chunk's sum
    const int de = live ? ea + ew : kFxNone;
    const int em = __reduce_max_sync(0xffffffffu, de), d = em - de + 5;
    dr = warp_sum(live ? fx_align(dr, d) : 0);
    di = warp_sum(live ? fx_align(di, d) : 0);
    if (lane == 0) {
      const FxParts f = fx_parts(lz, rhs, gridDim.x - 1);
      f.a[chunk] = make_longlong2(dr, di);
      f.ae[chunk] = em + 5;
    }
  }
}

// ------------------------------------------------------------------ update
// One block per SM, block b taking the chunks [nchunk b / G, nchunk (b+1) / G); a group of four warps per
// chunk, warp sp of the group its spin sp. Groups synchronise by themselves (named barriers).
// A chunk's inputs are copied to shared memory asynchronously, the first chunk's before anything else,
// so that their latency passes during the prologue: every block forms the coefficients from the pair
// stencil's chunk sums (a microsecond, instead of a one-block kernel between the two). The block that takes
// the last ticket at the start (every block has read j by then) advances j and marks the step pending
// for k_fx_settle.
constexpr int kFxGroups = 5;  // chunks in flight per block (96 registers a thread)
constexpr int kFxRows = 18;   // 16-byte inputs per thread: three colours of A, column j, column j-1, twice

__device__ __forceinline__ void group_sync(int grp) { asm volatile("bar.sync %0, 128;" ::"r"(grp + 1) : "memory"); }

// H and X of a b (complex limbs) added to hr, hi, xr, xi.
__device__ __forceinline__ void fx_cmad(const FxC& a, int nh, int nl, const FxC& b, fx64& hr, fx64& hi, fx64& xr, fx64& xi) {
  fx_mad(hr, a.rh, b.rh);
  fx_mad(hi, a.rh, b.ih);
  fx_mad(xr, a.rh, b.rl);
  fx_mad(xi, a.rh, b.il);
  fx_mad(xr, a.rl, b.rh);
  fx_mad(xi, a.rl, b.ih);
  fx_mad(hr, nh, b.ih);
  fx_mad(hi, a.ih, b.rh);
  fx_mad(xr, nh, b.il);
  fx_mad(xi, a.ih, b.rl);
  fx_mad(xr, nl, b.ih);
  fx_mad(xi, a.il, b.rh);
}
// A coefficient's limbs moved down by d bits (to another exponent).
__device__ __forceinline__ FxC fx_lower(const FxC& c, int d) {
  const int n = min(d, 62);
  const fx64 half = n > 0 ? (fx64)1 << (n - 1) : 0;
  FxC r;
  fx_split(fx_sar(((fx64)c.rh << 30) + c.rl + half, n), r.rh, r.rl);
  fx_split(fx_sar(((fx64)c.ih << 30) + c.il + half, n), r.ih, r.il);
  return r;
}

template <bool STORE, bool XACC>
__global__ void __launch_bounds__(128 * kFxGroups, 1)
    k_fx_update(Geom g, LzDev lz, const __grid_constant__ FxVecs fx, double2* vh) {
  extern __shared__ FxC rows[];  // [row][thread]
  const int rhs = blockIdx.y;
  __shared__ FxCoefSh cs[6];  // c0, (kv a), c2, c0w, (kw conj(a)), c2w
  __shared__ double ash[2][4];
  __shared__ fx64 dots[kFxGroups][4][4][32];
  __shared__ int tops[kFxGroups][2][4][32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nt = blockDim.x;
  const int ended = lz.status[rhs];
  const int j = lz.j[rhs];  // (the settle block may take it back, with a status: see below)
  if (ended > 1 || j == 0) {  // see k_fx_pair
    grid_wait();
    return;
  }
  const int nchunk = (g.vol + 31) >> 5;
  const size_t n = (size_t)12 * g.vol, o = (size_t)rhs * (lz.kmax + 2);
  const int grp = tid >> 7, sp = (tid >> 5) & 3, ngrp = nt >> 7;
  const int c0 = (int)((long long)nchunk * blockIdx.x / gridDim.x), c1 = (int)((long long)nchunk * (blockIdx.x + 1) / gridDim.x);
  // rows 0..2 and 9..11: A (after the wait); 3..8, 12..17: columns j and j - 1 (before it)
  const FxC* in[6] = {fx.av, fx.v[j & 1], fx.v[(j + 1) & 1], fx.aw, fx.w[j & 1], fx.w[(j + 1) & 1]};
  auto fetch = [&](int ch, bool a) {  // this thread's inputs of chunk ch (a lane past the end takes the last site's)
    const size_t base = (size_t)rhs * n + (size_t)sp * 3 * g.vol + min(ch * 32 + lane, g.vol - 1);
#pragma unroll
    for (int i = 0; i < kFxRows; ++i)
      if ((i % 9 < 3) == a) copy_async(rows + i * nt + tid, in[i / 3] + base + (size_t)(i % 3) * g.vol);
  };
  const bool any = c0 + grp < c1;
  const size_t es0 = (size_t)rhs * g.vol + min((c0 + grp) * 32 + lane, g.vol - 1);
  int ex[6] = {0, 0, 0, 0, 0, 0};  // exponents of A, columns j and j - 1, twice
  auto fetch_e = [&](size_t es, bool a) {
    if (a)
      ex[0] = fx.eav[es], ex[3] = fx.eaw[es];
    else
      ex[1] = fx.ev[j & 1][es], ex[2] = fx.ev[(j + 1) & 1][es], ex[4] = fx.ew[j & 1][es], ex[5] = fx.ew[(j + 1) & 1][es];
  };
  if (any) {
    fetch(c0 + grp, false);
    fetch_e(es0, false);
  }
  grid_wait();
  grid_launch();
  const int status = lz.status[rhs];
  const FxParts parts = fx_parts(lz, rhs, nchunk);
  const FxStep* st = fx_step(fx, rhs);
  const int er0 = st->emax[0][j & 1], er1 = st->emax[1][j & 1];
  {
    const int nshare = min(4, nt >> 6);
    zd k = mk(0.0, 0.0);
    if (warp == 0 && lane < 3) k = mk(st->k[lane].x, st->k[lane].y);
    if (warp == 1 && lane < 4) cs[lane < 2 ? 2 * lane : 2 * lane - 1] = st->c[lane];
    if (any) {
      fetch(c0 + grp, true);
      fetch_e(es0, true);
    }
    if (warp < 2 * nshare) {  // the sum of what^H A v: warp (value, share)
      const int v = warp & 1, q = warp >> 1;
      const double x = fx_warp_sum_chunks(
          nchunk, q, nshare, [&](int c) { return v ? parts.a[c].y : parts.a[c].x; }, [&](int c) { return parts.ae[c]; },
          -58 - 2044);
      if (lane == 0) ash[v][q] = x;
    }
    if (status) {  // (uniform)
      copy_wait();
      return;
    }
    __syncthreads();
    if (warp == 0) {
      zd a = mk(ash[0][0], ash[1][0]);
      for (int q = 1; q < nshare; ++q) a = a + mk(ash[0][q], ash[1][q]);
      const zd r = k * (lane == 1 ? conj(a) : a);
      if (lane < 2) cs[3 * lane + 1] = fx_coefficient(r);
      if (lane == 2 && blockIdx.x == 0) lz.alpha[o + j] = make_double2(r.re, r.im);
    }
    if (tid == 32) {
      // (every thread of the block has read j: the barrier above)
      __threadfence();
      if (atomicAdd(lz.count + rhs, 1u) == gridDim.x - 1) {
        lz.count[rhs] = 0u;
        lz.j[rhs] = j + 1;
        lz.pending[rhs] = 1;
      }
    }
    __syncthreads();
  }
  const zd xc = XACC ? ldc<double>(lz.xcoef, o + j + 1) : mk(0.0, 0.0);
  const int eref[2] = {er0, er1};
#pragma unroll 1
  for (int ch = c0 + grp; ch < c1; ch += ngrp) {
    const bool live = ch * 32 + lane < g.vol;
    const int s = live ? ch * 32 + lane : g.vol - 1;
    const size_t base = (size_t)rhs * n + (size_t)sp * 3 * g.vol + s;
    const size_t es = (size_t)rhs * g.vol + s;
    fx64 x[2][3][2];
    int en[2];
#pragma unroll
    for (int role = 0; role < 2; ++role) {
      const FxCoefSh& k0 = cs[3 * role];
      const FxCoefSh& k1 = cs[3 * role + 1];
      const FxCoefSh& k2 = cs[3 * role + 2];
      const bool prev = k2.e != kFxNone;
      // biased exponents of the three products; the coefficients are moved to the largest, so that the
      // products add up without shifts
      const int e0 = ex[3 * role] + k0.e - 1022, e1 = ex[3 * role + 1] + k1.e - 1022;
      const int e2 = prev ? ex[3 * role + 2] + k2.e - 1022 : kFxNone;
      const int E = max(max(e0, e1), e2);
      const FxC q0 = fx_lower(k0.c, E - e0), q1 = fx_lower(k1.c, E - e1), q2 = fx_lower(k2.c, E - e2);
      if (role == 0) copy_wait();
      int m = 0;
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const FxC va = rows[(role * 9 + a) * nt + tid], vv = rows[(role * 9 + 3 + a) * nt + tid];
        fx64 hr = fx_mul(q0.rh, va.rh), hi = fx_mul(q0.rh, va.ih), xr = fx_mad_to(q0.rh, va.rl, (fx64)1 << 29),
             xi = fx_mad_to(q0.rh, va.il, (fx64)1 << 29);
        fx_mad(xr, q0.rl, va.rh);
        fx_mad(xi, q0.rl, va.ih);
        if (role == 1) {  // (vhat's coefficient of A v is real)
          fx_mad(hr, -q0.ih, va.ih);
          fx_mad(hi, q0.ih, va.rh);
          fx_mad(xr, -q0.ih, va.il);
          fx_mad(xi, q0.ih, va.rl);
          fx_mad(xr, -q0.il, va.ih);
          fx_mad(xi, q0.il, va.rh);
        }
        fx_cmad(q1, -q1.ih, -q1.il, vv, hr, hi, xr, xi);
        if (prev) fx_cmad(q2, -q2.ih, -q2.il, rows[(role * 9 + 6 + a) * nt + tid], hr, hi, xr, xi);
        hr += xr >> 30;
        hi += xi >> 30;
        x[role][a][0] = hr;
        x[role][a][1] = hi;
        m = fx_top(fx_top(m, hr), hi);
      }
      tops[grp][role][sp][lane] = m;
      en[role] = E;
    }
    group_sync(grp);
    FxC nv[2][3];  // new limbs of vhat and what
    int em[2];     // largest exponent of the chunk's sites
#pragma unroll
    for (int role = 0; role < 2; ++role) {
      const int m = max(max(tops[grp][role][0][lane], tops[grp][role][1][lane]),
                        max(tops[grp][role][2][lane], tops[grp][role][3][lane]));
      int r = fx_norm_shift(m);
      const int e = en[role] + r + 1;
      em[role] = __reduce_max_sync(0xffffffffu, live ? e : kFxNone);
      // sites within three bits of the largest exponent of the previous column take that one: nearly all
      // sites of a vector then share it, and the next pair stencil's hops need no shift
      const int up = eref[role] - e;
      if (up > 0 && up <= 3) r += up;
      en[role] += r + 1;
      const int rr = max(r, 0), rl = max(-r, 0);
      const fx64 half = rr > 0 ? (fx64)1 << (rr - 1) : 0;
      FxC* P = (role ? fx.w : fx.v)[(j + 1) & 1] + base;  // in place of column j-1
      const int k = en[role] - 1022 - 59;
      const bool normal = k > -1000 && k < 900;
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const fx64 qr = ((x[role][a][0] + half) >> rr) << rl, qi = ((x[role][a][1] + half) >> rr) << rl;
        FxC y;
        fx_split(qr, y.rh, y.rl);
        fx_split(qi, y.ih, y.il);
        nv[role][a] = y;
        if (live) {
          P[(size_t)a * g.vol] = y;
          if (role == 0 && (STORE || XACC)) {
            zd d = mk((double)qr, (double)qi);
            if (normal) {  // q is 0 or between 1 and 2^59: the exponent field moves
              d.re = __hiloint2double(__double2hiint(d.re) + (qr ? k * (1 << 20) : 0), __double2loint(d.re));
              d.im = __hiloint2double(__double2hiint(d.im) + (qi ? k * (1 << 20) : 0), __double2loint(d.im));
            } else {
              d = mk(fx_scalb(d.re, k), fx_scalb(d.im, k));
            }
            const size_t at = (size_t)(sp * 3 + a) * g.vol + s;
            if (STORE) stc<double>(vh, ((size_t)rhs * lz.vcols + j) * n + at, d);  // column j + 1
            if (XACC) {
              double2* xa = lz.xacc + (size_t)rhs * n;
              stc<double>(xa, at, ldc<double>(xa, at) + xc * d);
            }
          }
        }
      }
      if (live && sp == 0) (role ? fx.ew : fx.ev)[(j + 1) & 1][es] = en[role];
    }
    if (lane == 0 && sp < 2) atomicMax(&fx_step(fx, rhs)->emax[sp][(j + 1) & 1], sp ? em[1] : em[0]);
    if (ch + ngrp < c1) {  // (this thread has read its rows)
      const size_t nx = (size_t)rhs * g.vol + min((ch + ngrp) * 32 + lane, g.vol - 1);
      fetch(ch + ngrp, false);
      fetch(ch + ngrp, true);
      fetch_e(nx, false);
      fetch_e(nx, true);
    }
    // what^H vhat, |vhat|^2, |what|^2 of this spin
    fx64 h[4] = {0, 0, 0, 0}, xx[4] = {0, 0, 0, 0};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const FxC u = nv[0][a], y = nv[1][a];
      const int nh = -y.ih, nl = -y.il;
      fx_mad(h[0], y.rh, u.rh);
      fx_mad(h[0], y.ih, u.ih);
      fx_mad(xx[0], y.rh, u.rl);
      fx_mad(xx[0], y.rl, u.rh);
      fx_mad(xx[0], y.ih, u.il);
      fx_mad(xx[0], y.il, u.ih);
      fx_mad(h[1], y.rh, u.ih);
      fx_mad(h[1], nh, u.rh);
      fx_mad(xx[1], y.rh, u.il);
      fx_mad(xx[1], y.rl, u.ih);
      fx_mad(xx[1], nh, u.rl);
      fx_mad(xx[1], nl, u.rh);
      fx_mad(h[2], u.rh, u.rh);
      fx_mad(h[2], u.ih, u.ih);
      fx_mad(xx[2], u.rh, u.rl);
      fx_mad(xx[2], u.ih, u.il);
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
      const int e = !live ? kFxNone : v < 2 ? en[0] + en[1] : v == 2 ? 2 * en[0] : 2 * en[1];
      const int em = __reduce_max_sync(0xffffffffu, e);
      const fx64 t = warp_sum(live ? fx_align(d, em - e + 5) : 0);
      if (lane == 0) {
        parts.u[(size_t)v * nchunk + ch] = t;
        parts.ue[(size_t)v * nchunk + ch] = em + 5;
      }
    }
    // (the next chunk's tops are written before its first barrier, which every warp reaches only after
    // reading this chunk's dots; its dots are written after that barrier)
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

cudaError_t launch_fx_begin(const Geom& g, const Links& U, double m_w, const LzDev& lz, const FxVecs& fx, const void* vh,
                            const void* w1, cudaStream_t st) {
  return launch_plain(k_fx_begin, dim3((g.vol + 63) / 64, lz.nrhs), dim3(64), st, g, lz, fx, (const double2*)vh,
                      (const double2*)w1, hop_coef<double>(m_w, 0.0).ks, U.fxf);
}

cudaError_t launch_fx_settle(const Geom& g, const Links& U, double m_w, const LzDev& lz, const FxVecs& fx,
                             cudaStream_t st) {
  return launch_plain(k_fx_settle, dim3(1, lz.nrhs), dim3(kFxSettle), st, lz, fx, (g.vol + 31) >> 5,
                      hop_coef<double>(m_w, 0.0).ks, U.fxf);
}

// Early launch behind the previous kernel of the stream, with dynamic shared memory.
template <typename... KArgs, typename... Args>
static cudaError_t launch_early(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args... args) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  {  // once per kernel and device and size
    static std::mutex mu;
    static std::map<std::pair<const void*, int>, size_t> allowed;
    std::lock_guard<std::mutex> lk(mu);
    size_t& a = allowed[{(const void*)kern, dev}];
    if (a < smem) {
      if ((e = cudaFuncSetAttribute((const void*)kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem))) return e;
      a = smem;
    }
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, args...);
}

cudaError_t launch_fx_pair(const Geom& g, const Links& U, double m_w, double mu, const LzDev& lz, const FxVecs& fx,
                           cudaStream_t st, int variant) {
  const FxCoef cp = fx_coef(m_w, mu), cm = fx_coef(m_w, -mu);
  const bool split = variant == 1 || variant == 4 || variant == 5;
  const dim3 grid((g.vol + 31) / 32 + 1, lz.nrhs);
  const FxPairArgs args{{cp, cm},
                        {{fx.v[0], fx.v[1]}, {fx.w[0], fx.w[1]}},
                        {{fx.ev[0], fx.ev[1]}, {fx.ew[0], fx.ew[1]}},
                        {fx.av, fx.aw},
                        {fx.eav, fx.eaw}};
  return split ? launch_early(k_fx_pair<4>, grid, dim3(32, 8), sizeof(FxPairSmem<4>), st, g, U, args, fx_self(cp.k.ks), lz,
                              fx, cp.k.ks)
               : launch_early(k_fx_pair<1>, grid, dim3(32, 2), sizeof(FxPairSmem<1>), st, g, U, args, fx_self(cp.k.ks), lz,
                              fx, cp.k.ks);
}

cudaError_t launch_fx_update(const Geom& g, const LzDev& lz, const FxVecs& fx, void* vh, cudaStream_t st) {
  int dev = 0, nsm = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  const int nchunk = (g.vol + 31) >> 5;
  const int nb = std::min(nsm, nchunk);
  const int grp = std::min(kFxGroups, (nchunk + nb - 1) / nb);
  using Kern = void (*)(Geom, LzDev, FxVecs, double2*);
  const Kern kern = lz.xacc ? k_fx_update<false, true> : fx.store ? k_fx_update<true, false> : k_fx_update<false, false>;
  return launch_early(kern, dim3(nb, lz.nrhs), dim3(128 * grp), (size_t)128 * grp * kFxRows * 16, st, g, lz, fx,
                      (double2*)vh);
}

}  // namespace ovl
