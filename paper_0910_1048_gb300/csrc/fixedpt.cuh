// The FP64 stencil's hop sums in fixed point on the integer pipe.
//
// GB300 issues two FP64 operations per SM and clock (a DFMA chain probe: 1.7 lanes), so a DFMA holds a scheduler's
// pipe for 64-75 clocks. A 32 x 32 + 64 bit integer multiply-add (mad.wide.s32) takes about 4, so a product of two
// 59-bit fixed-point numbers from three of them costs a fifth to a sixth of one. A hop's link product is a sum of six
// real products with a common scale, which fixed point holds exactly, so the stencil's FP64 work is left only
// where values leave a site: one conversion and one fused multiply-add per output component.
//
// A number is x = (h 2^30 + l) 2^-59 S: h a signed, l a 30-bit limb, S a power of two.
//  - Spinors: S is 2^(e+1) for e the exponent of the site's largest component (block floating point:
//    one S for the 24 reals of a neighbour), |h| <= 2^29, 0 <= l < 2^30. A component is cut at
//    2^-59 S; FP64 arithmetic on the same site rounds every partial sum at about 2^-54 S.
//  - Links: (h 2^30 + l) 2^-58 S, S one power of two for the field, at least its largest component and its
//    largest row or column sum of moduli of components over sqrt(6) (1 for SU(3)), l balanced in
//    [-2^29, 2^29), so that the dropped l l products have mean zero.
//  - Projected half spinors are limb-wise sums: |h| <= 2^30, l in (-2^30, 2^31).
//  - Products: H = sum h_u h, X = sum (h_u l + l_u h) over a row's six components, |H| < 2^59.4 and
//    |X| < 2^62.5; the l_u l terms, below 2^-59 of full scale, are dropped.
//  - A hop's 12 reals T = H + (X >> 30) are in units of 2^-57 of the neighbour's scale. The site's
//    accumulators are in units of 2^-57 2^(E-1022), E at least every hop's exponent; a hop whose
//    exponent is smaller is shifted (rounded). Six hops and two with factors below 4 stay below 2^62.7.
// The error of a hop sum is about 2^-55 of the neighbours' common scale (the cuts of eight hops and the
// dropped products), against about 2^-52 of their largest component for the FP64 chains it replaces.
// Measured on GB300 (independent chains, operands that change): mad.wide.s32 3.7 to 4.6 clocks per warp and
// scheduler, logic operations and shifts 2, mul.hi 3.6. So a hop's 216 products are 800 to 1000 clocks a warp of the
// about 1300 it takes. Against the FP64 hops D_W at 12^4 takes 22.9 us instead of 65.5, eight sources at 16^4
// 261 instead of 801 (255 without the zeros' signs and the neighbours' sizes, see below); its error against 64 bits
// is 1.4e-16 instead of 1.8e-16.
//
// That is an error relative to the largest terms around a site. FP64 arithmetic keeps a component's 53 bits however
// much smaller than the others it is, so the sums are used only where every component has terms of that size:
//  - Fields whose links mix the colours. Where colours decouple (unit or diagonal links, SU(2) blocks), a colour
//    1e-10 of the others came out with an error of 2e-7. FxField::ok = 0 also without a common scale: a
//    non-finite field, a link whose largest component is below a quarter of the field's scale, a scale far
//    from 1; a link with an entry below 2^-20 of its largest component, or more than half of the links with
//    one, or with their real or imaginary parts all, below 2^-6.
//  - Sites whose neighbours together fill every spin to 2^-6 of the largest component, or leave it zero
//    (FxSizes), or where a spin's sums come out large (fx_large, the split shape): a hop joins two spins only, so a
//    small spin beside a large one can reach the site alone.
//    Gaussian fields fill all of them; a site beside one site of widely different spins is refused, and so are
//    sites next to an infinity, a NaN or only components below 2^-959 (E < 64).
// Others take the FP64 hops. Integer sums do not depend on their order, so every shape of the stencil gives the
// same hop sums up to the rounding above.
#pragma once

#include "wilson.cuh"

namespace ovl {

typedef long long fx64;

struct alignas(16) FxC {  // a complex link entry: limbs of its real and imaginary part
  int rh, rl, ih, il;
};

// Hop coefficients of the fixed-point stencil: the time hops' factors e^{+-mu} as 2^-57 fractions (below 4) of
// a power of two, 2^0 for |mu| < 1.38.
struct FxCoef {
  HopCoef<double> k;
  int fh, fl, fe;  // forward: (fh 2^30 + fl) 2^-57 2^fe
  int bh, bl, be;  // backward
  int ft, bt;      // exponents of the factors (2^ft <= factor < 2^(ft+1)), for FxSizes
  int unit;        // 1: both factors are 1 (mu = 0)
  int ok;          // 0: a factor is outside the fixed-point range (FP64 path)
};

inline FxCoef fx_coef(double m_w, double mu) {
  FxCoef c;
  c.k = hop_coef<double>(m_w, mu);
  c.unit = mu == 0.0;
  c.ok = std::fabs(mu) <= 16.0;
  auto split = [&](double f, int& h, int& l, int& e, int& x) {
    const double m = std::frexp(c.ok ? f : 1.0, &x);
    e = x > 2 ? x - 2 : 0;
    const fx64 q = std::llrint(std::ldexp(m, 57 + x - e));
    h = (int)(q >> 30);
    l = (int)(q & ((1 << 30) - 1));
    --x;
  };
  split(std::exp(mu), c.fh, c.fl, c.fe, c.ft);
  split(std::exp(-mu), c.bh, c.bl, c.be, c.bt);
  return c;
}

// Shifts with the amount clamped to the word (PTX semantics).
OVL_HD unsigned long long fx_shr(unsigned long long v, int n) {
#if defined(__CUDA_ARCH__)
  unsigned long long r;
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(n));
  return r;
#else
  return n > 63 ? 0ull : v >> n;
#endif
}
OVL_HD fx64 fx_sar(fx64 v, int n) {
#if defined(__CUDA_ARCH__)
  fx64 r;
  asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(n));
  return r;
#else
  return v >> (n > 63 ? 63 : n);
#endif
}
// acc + a b in one instruction. (Written out, with the negated factor formed once per link entry: as plain C products the
// Lanczos step at 12^4 took 49.3 us instead of 45.7.)
OVL_HD void fx_mad(fx64& acc, int a, int b) {
#if defined(__CUDA_ARCH__)
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(acc) : "r"(a), "r"(b));
#else
  acc += (fx64)a * b;
#endif
}
// a b + c (c kept)
OVL_HD fx64 fx_mad_to(int a, int b, fx64 c) {
#if defined(__CUDA_ARCH__)
  fx64 r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
#else
  return c + (fx64)a * b;
#endif
}
OVL_HD fx64 fx_mul(int a, int b) {
#if defined(__CUDA_ARCH__)
  fx64 r;
  asm("mul.wide.s32 %0, %1, %2;" : "=l"(r) : "r"(a), "r"(b));
  return r;
#else
  return (fx64)a * b;
#endif
}
OVL_HD void fx_words(double x, int& hi, unsigned& lo) {
#if defined(__CUDA_ARCH__)
  hi = __double2hiint(x);
  lo = (unsigned)__double2loint(x);
#else
  unsigned long long b;
  std::memcpy(&b, &x, 8);
  hi = (int)(b >> 32);
  lo = (unsigned)b;
#endif
}
OVL_HD double fx_pow2(int biased) {  // 2^(biased - 1023), 0 < biased < 2047
#if defined(__CUDA_ARCH__)
  return __hiloint2double(biased << 20, 0);
#else
  return std::ldexp(1.0, biased - 1023);
#endif
}

// Limbs of x in units of 2^-59 2^(e-1022), e >= 64 at least x's biased exponent (smaller values are
// shifted out). A negative value is the one's complement of its 59-bit magnitude: one unit off, and two
// instructions less per component. Zeros of either sign, and subnormals (biased exponent 0), give 0: their sign is
// left out, so that components that are exactly zero add nothing.
OVL_HD void fx_limbs(int hi, unsigned lo, int e, int& h, int& l) {
  const int d = e - (int)(((unsigned)hi >> 20) & 0x7ffu);
  const unsigned s = (unsigned)hi >= 0x80100000u ? ~0u : 0u;
  const unsigned mh = (((unsigned)hi << 6 | lo >> 26) & 0x03ffffffu) ^ s ^ 0x04000000u;
  const fx64 v = (fx64)((unsigned long long)mh << 32 | ((lo << 6) ^ s));
  h = (int)fx_sar(v, d + 30);
  l = (int)((unsigned)fx_sar(v, d) & 0x3fffffffu);
}

struct FxHalf {  // projected half spinor: limbs of [2 spins][3 colours] complex
  int rh[2][3], rl[2][3], ih[2][3], il[2][3];
};

struct FxAcc {  // accumulators of a site: sums of hops in units of 2^-57 2^(E-1022), E their biased exponent
  fx64 re[4][3], im[4][3];
};

OVL_HD void fx_clear(FxAcc& a) {
#pragma unroll
  for (int i = 0; i < 12; ++i) a.re[i / 3][i % 3] = a.im[i / 3][i % 3] = 0;
}

struct FxSpin {  // limbs of a site's 12 complex components relative to one exponent
  int rh[4][3], rl[4][3], ih[4][3], il[4][3];
};

// High word of the largest modulus of spin i's components.
OVL_HD int fx_spin_word(const Spin<double>& p, int i) {
  int m = 0;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    int w;
    unsigned z;
    fx_words(p.c[i][a].re, w, z);
    m = m > (w & 0x7fffffff) ? m : (w & 0x7fffffff);
    fx_words(p.c[i][a].im, w, z);
    m = m > (w & 0x7fffffff) ? m : (w & 0x7fffffff);
  }
  return m;
}
// Of the site's (its biased exponent is the word >> 20).
OVL_HD int fx_top_word(const Spin<double>& p) {
  int m = 0;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int w = fx_spin_word(p, i);
    m = m > w ? m : w;
  }
  return m;
}

// Largest component of each spin over the neighbours of a site, times the hops' factors: the upper halves of the
// moduli's high words (exponent and four bits of the mantissa), two spins to a word.
struct FxSizes {
  unsigned m[2] = {0, 0};
};
OVL_HD unsigned fx_max2(unsigned a, unsigned b) {  // of both halves
#if defined(__CUDA_ARCH__)
  unsigned r;
  asm("max.u16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
  return r;
#else
  const unsigned h = a >> 16 > b >> 16 ? a : b, l = (a & 0xffffu) > (b & 0xffffu) ? a : b;
  return (h & 0xffff0000u) | (l & 0xffffu);
#endif
}
OVL_HD unsigned fx_sizes2(int a, int b) {  // from two high words of moduli
#if defined(__CUDA_ARCH__)
  return __byte_perm((unsigned)a, (unsigned)b, 0x7632);
#else
  return ((unsigned)b & 0xffff0000u) | (unsigned)a >> 16;
#endif
}
OVL_HD int fx_raise(int w, int e) {  // a high word times 2^e, where not zero
  const int r = w + e * (1 << 20);
  return w ? (r > 1 << 16 ? r : 1 << 16) : 0;
}
constexpr int kFxEven = 6;  // bits

// Whether all of them are zero or within 2^-kFxEven of the largest.
OVL_HD bool fx_even(const FxSizes& z) {
  const int a = (int)(z.m[0] & 0xffffu), b = (int)(z.m[0] >> 16), c = (int)(z.m[1] & 0xffffu), d = (int)(z.m[1] >> 16);
  const int t = a > b ? a : b, u = c > d ? c : d, least = (t > u ? t : u) - (kFxEven << 4);
  return (a == 0 || a >= least) && (b == 0 || b >= least) && (c == 0 || c >= least) && (d == 0 || d >= least);
}

OVL_HD void fx_spin(const Spin<double>& p, int e, FxSpin& o) {
#pragma unroll
  for (int i = 0; i < 12; ++i) {
    int w;
    unsigned z;
    fx_words(p.c[i / 3][i % 3].re, w, z);
    fx_limbs(w, z, e, o.rh[i / 3][i % 3], o.rl[i / 3][i % 3]);
    fx_words(p.c[i / 3][i % 3].im, w, z);
    fx_limbs(w, z, e, o.ih[i / 3][i % 3], o.il[i / 3][i % 3]);
  }
}

// h_s = p_s + rot p_q with rot = 1 (ROT 0), i (1), -1 (2), -i (3); CONJ: its complex conjugate.
template <int ROT, bool CONJ>
OVL_HD void fx_row(const FxSpin& p, int s, int q, FxHalf& h) {
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    int rh, rl, ih, il;  // rot p_q
    if (ROT == 0) rh = p.rh[q][a], rl = p.rl[q][a], ih = p.ih[q][a], il = p.il[q][a];
    if (ROT == 1) rh = -p.ih[q][a], rl = -p.il[q][a], ih = p.rh[q][a], il = p.rl[q][a];
    if (ROT == 2) rh = -p.rh[q][a], rl = -p.rl[q][a], ih = -p.ih[q][a], il = -p.il[q][a];
    if (ROT == 3) rh = p.ih[q][a], rl = p.il[q][a], ih = -p.rh[q][a], il = -p.rl[q][a];
    h.rh[s][a] = p.rh[s][a] + rh;
    h.rl[s][a] = p.rl[s][a] + rl;
    h.ih[s][a] = CONJ ? -(p.ih[s][a] + ih) : p.ih[s][a] + ih;
    h.il[s][a] = CONJ ? -(p.il[s][a] + il) : p.il[s][a] + il;
  }
}

// Half spinor of (1 - g_mu) p (MINUS) or (1 + g_mu) p (see project()).
template <int MU, bool MINUS, bool CONJ>
OVL_HD void fx_project(const FxSpin& p, FxHalf& h) {
  constexpr int r0 = MU == 0 ? (MINUS ? 1 : 3) : MU == 1 ? (MINUS ? 0 : 2) : MU == 2 ? (MINUS ? 1 : 3) : (MINUS ? 2 : 0);
  constexpr int r1 = MU == 0 ? (MINUS ? 1 : 3) : MU == 1 ? (MINUS ? 2 : 0) : MU == 2 ? (MINUS ? 3 : 1) : (MINUS ? 2 : 0);
  fx_row<r0, CONJ>(p, 0, MU < 2 ? 3 : 2, h);
  fx_row<r1, CONJ>(p, 1, MU < 2 ? 2 : 3, h);
}

// a + rot (re, im), rot = 1 (ROT 0), i (1), -1 (2), -i (3)
template <int ROT>
OVL_HD void fx_add_rot(fx64& re, fx64& im, fx64 tr, fx64 ti) {
  re += ROT == 0 ? tr : ROT == 1 ? -ti : ROT == 2 ? -tr : ti;
  im += ROT == 0 ? ti : ROT == 1 ? tr : ROT == 2 ? -ti : -tr;
}

// acc += (t, -/+ N t) for the half spinor t of a hop (see reconstruct_add).
template <int MU, bool FWD>
OVL_HD void fx_reconstruct(FxAcc& acc, const fx64 (&tr)[2][3], const fx64 (&ti)[2][3]) {
  constexpr int i2 = MU < 2 ? 1 : 0, i3 = MU < 2 ? 0 : 1;
  constexpr int r2 = MU == 0 ? (FWD ? 3 : 1) : MU == 1 ? (FWD ? 2 : 0) : MU == 2 ? (FWD ? 3 : 1) : (FWD ? 2 : 0);
  constexpr int r3 = MU == 0 ? (FWD ? 3 : 1) : MU == 1 ? (FWD ? 0 : 2) : MU == 2 ? (FWD ? 1 : 3) : (FWD ? 2 : 0);
#pragma unroll
  for (int a = 0; a < 3; ++a) {  // the backward hop's t is conjugated
    fx_add_rot<0>(acc.re[0][a], acc.im[0][a], tr[0][a], FWD ? ti[0][a] : -ti[0][a]);
    fx_add_rot<0>(acc.re[1][a], acc.im[1][a], tr[1][a], FWD ? ti[1][a] : -ti[1][a]);
    fx_add_rot<r2>(acc.re[2][a], acc.im[2][a], tr[i2][a], FWD ? ti[i2][a] : -ti[i2][a]);
    fx_add_rot<r3>(acc.re[3][a], acc.im[3][a], tr[i3][a], FWD ? ti[i3][a] : -ti[i3][a]);
  }
}

// T (|T| < 2^59.4) times the factor (h 2^30 + l) 2^-57.
OVL_HD fx64 fx_scale(fx64 t, int h, int l) {
  const int th = (int)(t >> 30), tl = (int)((unsigned)t & 0x3fffffffu);
  fx64 x = fx_mad_to(th, l, (fx64)1 << 26);
  fx_mad(x, tl, h);
  return (fx_mul(th, h) << 3) + (x >> 27);
}

// Half spinor of hop k = 2 mu (forward, U) or 2 mu + 1 (backward, U^H) from the neighbour's limbs.
// g5in: the input is gamma5 p (the lower spins change sign, which exchanges the two projectors). The
// direction is a run-time value (uniform over a warp) so that the hops share one copy of the conversion
// and the product: unrolled over the eight hops the kernel was 100 KB of code and took minutes to compile.
OVL_HD void fx_half(int k, const FxSpin& q, bool g5in, FxHalf& h) {
  // the backward hop multiplies by U^H = conj(U^T): conj(U^T conj(h)) conjugated at the end
  switch (g5in ? k + 8 : k) {
    case 0: fx_project<0, true, false>(q, h); break;
    case 1: fx_project<0, false, true>(q, h); break;
    case 2: fx_project<1, true, false>(q, h); break;
    case 3: fx_project<1, false, true>(q, h); break;
    case 4: fx_project<2, true, false>(q, h); break;
    case 5: fx_project<2, false, true>(q, h); break;
    case 6: fx_project<3, true, false>(q, h); break;
    case 7: fx_project<3, false, true>(q, h); break;
    case 8: fx_project<0, false, false>(q, h); break;
    case 9: fx_project<0, true, true>(q, h); break;
    case 10: fx_project<1, false, false>(q, h); break;
    case 11: fx_project<1, true, true>(q, h); break;
    case 12: fx_project<2, false, false>(q, h); break;
    case 13: fx_project<2, true, true>(q, h); break;
    case 14: fx_project<3, false, false>(q, h); break;
    default: fx_project<3, true, true>(q, h); break;
  }
}

// Exponent of hop k's contribution for a neighbour of exponent e.
OVL_HD int fx_hop_exponent(int k, int e, const FxCoef& c) { return k < 6 ? e : e + ((k & 1) ? c.be : c.fe); }

// Adds hop k of the half spinor h to the accumulators, d = E - (the hop's exponent) >= 0, `shift` whether any
// lane of the warp has d > 0. link(a, b): entry U[a][b], or U[b][a] for a backward hop. flip: the hop
// crosses an antiperiodic boundary.
template <class Link>
OVL_HD void fx_hop(int k, int d, bool shift, const FxHalf& h, Link link, const FxCoef& c, bool flip, FxAcc& acc) {
  const bool fwd = !(k & 1);
  fx64 tr[2][3], ti[2][3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    fx64 hr[2], hi[2], xr[2], xi[2];
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const FxC u = link(a, b);
      const int nh = -u.ih, nl = -u.il;
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        if (b == 0) {
          hr[r] = fx_mul(u.rh, h.rh[r][b]);
          hi[r] = fx_mul(u.rh, h.ih[r][b]);
          xr[r] = fx_mad_to(u.rh, h.rl[r][b], (fx64)1 << 29);  // (rounds the shift of X)
          xi[r] = fx_mad_to(u.rh, h.il[r][b], (fx64)1 << 29);
        } else {
          fx_mad(hr[r], u.rh, h.rh[r][b]);
          fx_mad(hi[r], u.rh, h.ih[r][b]);
          fx_mad(xr[r], u.rh, h.rl[r][b]);
          fx_mad(xi[r], u.rh, h.il[r][b]);
        }
        fx_mad(xr[r], u.rl, h.rh[r][b]);
        fx_mad(xi[r], u.rl, h.ih[r][b]);
        fx_mad(hr[r], nh, h.ih[r][b]);
        fx_mad(hi[r], u.ih, h.rh[r][b]);
        fx_mad(xr[r], nh, h.il[r][b]);
        fx_mad(xi[r], u.ih, h.rl[r][b]);
        fx_mad(xr[r], nl, h.ih[r][b]);
        fx_mad(xi[r], u.il, h.rh[r][b]);
      }
    }
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      tr[r][a] = hr[r] + (xr[r] >> 30);
      ti[r][a] = hi[r] + (xi[r] >> 30);
    }
  }
  if (k >= 6) {
    if (!c.unit) {
      const int fh = fwd ? c.fh : c.bh, fl = fwd ? c.fl : c.bl;
#pragma unroll
      for (int i = 0; i < 6; ++i) {
        tr[i / 3][i % 3] = fx_scale(tr[i / 3][i % 3], fh, fl);
        ti[i / 3][i % 3] = fx_scale(ti[i / 3][i % 3], fh, fl);
      }
    }
    if (flip) {
#pragma unroll
      for (int i = 0; i < 6; ++i) {
        tr[i / 3][i % 3] = -tr[i / 3][i % 3];
        ti[i / 3][i % 3] = -ti[i / 3][i % 3];
      }
    }
  }
  if (shift) {
    const int n = d < 62 ? d : 62;
    const fx64 half = n > 0 ? (fx64)1 << (n - 1) : 0;
#pragma unroll
    for (int i = 0; i < 6; ++i) {
      tr[i / 3][i % 3] = fx_sar(tr[i / 3][i % 3] + half, n);
      ti[i / 3][i % 3] = fx_sar(ti[i / 3][i % 3] + half, n);
    }
  }
  switch (k) {
    case 0: fx_reconstruct<0, true>(acc, tr, ti); break;
    case 1: fx_reconstruct<0, false>(acc, tr, ti); break;
    case 2: fx_reconstruct<1, true>(acc, tr, ti); break;
    case 3: fx_reconstruct<1, false>(acc, tr, ti); break;
    case 4: fx_reconstruct<2, true>(acc, tr, ti); break;
    case 5: fx_reconstruct<2, false>(acc, tr, ti); break;
    case 6: fx_reconstruct<3, true>(acc, tr, ti); break;
    default: fx_reconstruct<3, false>(acc, tr, ti); break;
  }
}

// Field-wide scale of the fixed-point links, kept in device memory beside them (a later ovl_set_links
// rewrites both in place, so captured graphs stay valid).
struct FxField {
  int ok;    // the links share a scale and mix the colours (see above)
  int uexp;  // the scale is 2^uexp
  unsigned long long nlo, hi;  // bits of the smallest of the links' largest components (complemented, so that all
                               // start from zero) and of the largest of the links' scales (fx_link_range)
  unsigned weak;              // links that mix the colours weakly
};

// |x| rounded up to 21 bits, from x's high word. (Without the FP64 pipe: with about 130 FP64 operations a link,
// set_links on a field of 102400 sites took 188 us instead of 117.)
OVL_HD float fx_abs_up(int hi) {
  const int a = hi & 0x7fffffff, e = (a >> 20) - 896;
  const int b = e < 1 ? 0x00800000 : e > 254 ? 0x7f800000 : (e << 23 | (a & 0xfffff) << 3) + 8;
#if defined(__CUDA_ARCH__)
  return __int_as_float(b);
#else
  float f;
  std::memcpy(&f, &b, 4);
  return f;
#endif
}

// Bits below the largest component of a link at which its smallest entry (its larger component) may lie: for any
// link, and for one that is not weak; there also its largest real and its largest imaginary part. Of random SU(3)
// links one in 7 10^10 falls below the first and one in 250 below the second, so a field of 64^4 sites is refused by
// chance once in a thousand times; links exp(i eps H) are mostly weak below eps = 0.04.
constexpr int kFxMixAny = 20, kFxMixMost = 6;

// Largest component of a link (0 if the link leaves a colour out), the scale it needs: the largest of that
// and its row and column sums of |re| + |im| over sqrt(6) (rounded up, but 1 for SU(3) to rounding), and whether it
// mixes the colours weakly.
OVL_HD void fx_link_range(const Mat3<double>& u, double& top, double& need, bool& weak) {
  float row[3] = {0, 0, 0}, col[3] = {0, 0, 0};
  unsigned long long m = 0;
  int least = 0x7fffffff, re = 0, im = 0;
#pragma unroll
  for (int i = 0; i < 9; ++i) {
    int hr, hi;
    unsigned lr, li;
    fx_words(u.m[i / 3][i % 3].re, hr, lr);
    fx_words(u.m[i / 3][i % 3].im, hi, li);
    hr &= 0x7fffffff;
    hi &= 0x7fffffff;
    const unsigned long long wr = (unsigned long long)(unsigned)hr << 32 | lr;
    const unsigned long long wi = (unsigned long long)(unsigned)hi << 32 | li;
    m = m > wr ? m : wr;
    m = m > wi ? m : wi;
    const int entry = hr > hi ? hr : hi;
    least = least < entry ? least : entry;
    re = re > hr ? re : hr;
    im = im > hi ? im : hi;
    const float a = fx_abs_up(hr) + fx_abs_up(hi);
    row[i / 3] += a;
    col[i % 3] += a;
  }
  const int most = (int)(m >> 32);
  const int part = re < im ? re : im;
  weak = (least < part ? least : part) < most - (kFxMixMost << 20);
  float sum = row[0];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    sum = row[i] > sum ? row[i] : sum;
    sum = col[i] > sum ? col[i] : sum;
  }
  const bool finite = m < 0x7ffull << 52;
#if defined(__CUDA_ARCH__)
  top = __longlong_as_double((long long)m);
#else
  std::memcpy(&top, &m, 8);
#endif
  if (!finite) top = 0.0;
  need = sum * 0.408247f;  // 1 / 2.4495, just above sqrt(6), and 21 bits
  need = top > need ? top : need;
  if (!finite) need = 1e308 * 10;  // infinity: the field is not usable
  if (least < most - (kFxMixAny << 20)) top = 0.0;
}
OVL_HD void fx_link_range(const Mat3<double>& u, double& top, double& need) {
  bool weak;
  fx_link_range(u, top, need, weak);
}

// Whether a field of n links, `weak` of them weakly mixing, mixes the colours.
OVL_HD bool fx_field_mixes(unsigned weak, size_t n) { return 2 * (size_t)weak <= n; }

// Scale exponent of a field with these ranges; false: the FP64 hops.
OVL_HD bool fx_field_scale(double lo, double hi, int* uexp) {
  *uexp = 0;
  if (!(hi > 0.0) || !(hi < 1e100) || !(lo >= 0.25 * hi)) return false;
  std::frexp(hi * (1.0 - 1e-6), uexp);  // a scale of 1 (+ rounding) is 2^0
  return *uexp >= -8 && *uexp <= 8;
}

// x 2^(58 - uexp) rounded to nearest, ties to even, for |x| up to about 2^uexp; subnormal numbers give 0. (By shifts: the
// conversion and the power of two are FP64 instructions, two lanes per SM and clock, and with both for every
// component set_links on 32^4 sites took 2.3 ms.)
OVL_HD fx64 fx_link_fixed(double x, int uexp) {
  int hi;
  unsigned lo;
  fx_words(x, hi, lo);
  const int ex = (hi >> 20) & 0x7ff, sh = ex - 1017 - uexp;
  if (ex == 0 || sh < -54) return 0;
  const fx64 m = (fx64)((unsigned long long)((hi & 0xfffff) | 0x100000) << 32 | lo);
  fx64 q;
  if (sh >= 0) {
    q = m << (sh < 8 ? sh : 8);  // (above 6 the field does not fit this scale)
  } else {
    q = (m + ((fx64)1 << (-sh - 1)) - 1 + (m >> -sh & 1)) >> -sh;
  }
  return hi < 0 ? -q : q;
}

OVL_HD FxC fx_link_entry(cplx<double> u, int uexp) {
  const fx64 qr = fx_link_fixed(u.re, uexp), qi = fx_link_fixed(u.im, uexp);
  FxC r;
  r.rh = (int)((qr + (1 << 29)) >> 30);
  r.rl = (int)(qr - ((fx64)r.rh << 30));
  r.ih = (int)((qi + (1 << 29)) >> 30);
  r.il = (int)(qi - ((fx64)r.ih << 30));
  return r;
}

// The coordinates of a site in 16-bit fields (extents are at most 4096).
OVL_HD unsigned long long fx_coords(const Geom& g, int s) {
  const int x = s % g.lx;
  int r = s / g.lx;
  const int y = r % g.ly;
  r /= g.ly;
  const int z = r % g.lz, t = r / g.lz;
  return (unsigned long long)(t << 16 | z) << 32 | (unsigned)(y << 16 | x);
}

// Neighbour of site s for hop k, and whether the hop crosses the time boundary.
OVL_HD int fx_neighbour(const Geom& g, int s, unsigned long long xyzt, int k, bool* wraps) {
  const int mu = k >> 1;
  const int st = mu == 0 ? 1 : mu == 1 ? g.sy : mu == 2 ? g.sz : g.st;
  const int len = mu == 0 ? g.lx : mu == 1 ? g.ly : mu == 2 ? g.lz : g.lt;
  const int x = (int)(fx_shr(xyzt, 16 * mu) & 0xffff);
  const bool edge = x == ((k & 1) ? 0 : len - 1);
  *wraps = mu == 3 && edge;
  const int step = edge ? (1 - len) * st : st;
  return (k & 1) ? s - step : s + step;
}

// Hops k0 .. k1-1 of site s, psi in FP64 loaded through `ld` and converted on the way, to limbs relative to the
// largest exponent E met so far (+1), so that no hop is shifted afterwards; the neighbours' sizes in z. Returns
// whether the accumulators hold the hop sum: no infinity or NaN among the neighbours, and not only components
// too small for the common exponent (all zero is fine: the sum is zero). For all eight hops together fx_even(z)
// has to hold too.
template <class Load>
OVL_HD bool fx_hops(const Geom& g, const FxC* U, int s, int k0, int k1, const FxCoef& c, Load ld, bool g5in, FxAcc& acc,
                    int& E, FxSizes& z) {
  const unsigned long long xyzt = fx_coords(g, s);
  int top = 0;
  E = 0;
#pragma unroll 1
  for (int k = k0; k < k1; ++k) {
    bool wraps;
    const int nb = fx_neighbour(g, s, xyzt, k, &wraps);
    FxHalf h;
    {
      Spin<double> p;
      ld(nb, p);
      int m[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) m[i] = fx_spin_word(p, i);
      const int t = m[0] > m[1] ? m[0] : m[1], u = m[2] > m[3] ? m[2] : m[3], w = t > u ? t : u, eb = w >> 20;
      top = top > w ? top : w;
      const int ft = k < 6 ? 0 : (k & 1) ? c.bt : c.ft;
      if (ft != 0) {
#pragma unroll
        for (int i = 0; i < 4; ++i) m[i] = fx_raise(m[i], ft);
      }
      z.m[0] = fx_max2(z.m[0], fx_sizes2(m[0], m[1]));
      z.m[1] = fx_max2(z.m[1], fx_sizes2(m[2], m[3]));
      const int fe = fx_hop_exponent(k, 0, c), eh = (eb > 64 ? eb : 64) + fe;
      if (eh > E) {  // first hop, or a larger neighbour than any before
        if (E != 0) {
#pragma unroll
          for (int i = 0; i < 12; ++i) {
            acc.re[i / 3][i % 3] = fx_sar(acc.re[i / 3][i % 3], eh + 1 - E);
            acc.im[i / 3][i % 3] = fx_sar(acc.im[i / 3][i % 3], eh + 1 - E);
          }
        }
        E = eh + 1;
      }
      FxSpin q;
      fx_spin(p, E - fe, q);
      fx_half(k, q, g5in, h);
    }
    const FxC* u = U + (size_t)(k >> 1) * 9 * g.vol + ((k & 1) ? nb : s);
    const size_t sa = (k & 1) ? (size_t)g.vol : (size_t)3 * g.vol, sb = (k & 1) ? (size_t)3 * g.vol : (size_t)g.vol;
    fx_hop(k, 0, false, h, [&](int a, int b) { return u[a * sa + b * sb]; }, c, wraps && g.t_bc < 0, acc);
  }
  if (top == 0) {  // zeros, or subnormal numbers
    unsigned any = 0;
#pragma unroll 1
    for (int k = k0; k < k1; ++k) {
      bool wraps;
      Spin<double> p;
      ld(fx_neighbour(g, s, xyzt, k, &wraps), p);
#pragma unroll
      for (int i = 0; i < 12; ++i) {
        int hr, hi;
        unsigned lr, li;
        fx_words(p.c[i / 3][i % 3].re, hr, lr);
        fx_words(p.c[i / 3][i % 3].im, hi, li);
        any |= ((unsigned)(hr | hi) & 0x7fffffffu) | lr | li;
      }
    }
    return any == 0;
  }
  return E < 2000 && top >= 64 << 20;  // (E is above 2047 beside an infinity or a NaN)
}
// Whether a spin's sums over all eight hops are at least 2^53 units, 2^-3 of the neighbours' largest component or more: some
// of its terms are then of that component's size, whatever the neighbours' spins are.
OVL_HD bool fx_large(const fx64 (&re)[3], const fx64 (&im)[3]) {
  int m = 0;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const int r = (int)(re[a] >> 32), i = (int)(im[a] >> 32);
    m = m > (r ^ (r >> 31)) ? m : (r ^ (r >> 31));
    m = m > (i ^ (i >> 31)) ? m : (i ^ (i >> 31));
  }
  return m >= 1 << 21;
}

// All eight hops.
template <class Load>
OVL_HD bool fx_hops(const Geom& g, const FxC* U, int s, int k0, int k1, const FxCoef& c, Load ld, bool g5in, FxAcc& acc,
                    int& E) {
  FxSizes z;
  return fx_hops(g, U, s, k0, k1, c, ld, g5in, acc, E, z) && fx_even(z);
}

// FP64 value of one unit of the accumulators times the hop coefficient ks and the links' scale.
OVL_HD double fx_unit(int E, const FxCoef& c, int uexp) { return c.k.ks * fx_pow2(E - 56 + uexp); }

}  // namespace ovl
