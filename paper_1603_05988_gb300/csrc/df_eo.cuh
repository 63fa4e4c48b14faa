// Double-float (hi + lo FP32, dfloat.cuh) red-black stencil, two columns per thread in packed FP32x2 instructions and
// one spin row per thread as in eo_core.cuh: the outer residuals of the mixed solvers.
//
// Every sum is a TwoSum and every product of hi parts a TwoProd, their errors and the cross terms gathered in lo:
// 12 packed instructions for a real product added to a sum, ~4200 for a site, row and column pair.  They run on the
// FP32 pipe, which bounds the kernels; FP64 instructions (two lanes per clock and SM, sixty-four times fewer) are kept
// out of the loops down to the conversions, which are done on the integer pipe (split_f64).
#pragma once

#include "dfloat.cuh"
#include "eo_core.cuh"

namespace dtr {

struct d2 {  // a real number per column
  float2 hi, lo;
};
struct z2 {  // a complex one
  d2 re, im;
};
__device__ __forceinline__ d2 dzero() { return d2{f2(0.f), f2(0.f)}; }
// u + s l for s a power of two (or 0) per column: the product is exact, so this is a TwoSum on hi
__device__ __forceinline__ d2 axs(d2 u, d2 l, float2 s) {
  const float2 t = __ffma2_rn(s, l.hi, u.hi);
  const float2 nb = sub2(u.hi, t);
  const float2 e = __fadd2_rn(sub2(u.hi, __fadd2_rn(t, nb)), __ffma2_rn(s, l.hi, nb));
  return d2{t, __fadd2_rn(__ffma2_rn(s, l.lo, u.lo), e)};
}
// the same for an l without lo part
__device__ __forceinline__ d2 axs1(d2 u, float2 l, float2 s) {
  const float2 t = __ffma2_rn(s, l, u.hi);
  const float2 nb = sub2(u.hi, t);
  const float2 e = __fadd2_rn(sub2(u.hi, __fadd2_rn(t, nb)), __ffma2_rn(s, l, nb));
  return d2{t, __fadd2_rn(u.lo, e)};
}
__device__ __forceinline__ z2 axs(z2 u, z2 l, float2 s) { return z2{axs(u.re, l.re, s), axs(u.im, l.im, s)}; }
// u + i s l, n = -s
__device__ __forceinline__ z2 axis(z2 u, z2 l, float2 s, float2 n) { return z2{axs(u.re, l.im, n), axs(u.im, l.re, s)}; }
// hi + lo with |lo| at most half an ulp of hi
__device__ __forceinline__ d2 renorm(d2 a) {
  const float2 t = __fadd2_rn(a.hi, a.lo);
  const float2 nb = sub2(a.hi, t);
  return d2{t, __fadd2_rn(sub2(a.hi, __fadd2_rn(t, nb)), __fadd2_rn(a.lo, nb))};
}
// a link entry's real or imaginary part, hi + lo, with its sign for this product
struct dm {
  float2 hi, nhi, lo;
};
__device__ __forceinline__ dm dmul(float hi, float lo) { return dm{f2(hi), f2(-hi), f2(lo)}; }
__device__ __forceinline__ dm dneg(float hi, float lo) { return dm{f2(-hi), f2(hi), f2(-lo)}; }
__device__ __forceinline__ d2 prod(const dm &m, d2 h) {
  const float2 p = __fmul2_rn(m.hi, h.hi);
  const float2 ne = __ffma2_rn(m.nhi, h.hi, p);  // minus the rounding error of p
  return d2{p, sub2(__ffma2_rn(m.hi, h.lo, __fmul2_rn(m.lo, h.hi)), ne)};
}
__device__ __forceinline__ d2 mac(const dm &m, d2 h, d2 s) {
  const float2 p = __fmul2_rn(m.hi, h.hi);
  const float2 ne = __ffma2_rn(m.nhi, h.hi, p);
  const float2 t = __fadd2_rn(s.hi, p);
  const float2 nb = sub2(s.hi, t);
  const float2 e = __fadd2_rn(sub2(s.hi, __fadd2_rn(t, nb)), __fadd2_rn(p, nb));
  const float2 lo = __ffma2_rn(m.hi, h.lo, __ffma2_rn(m.lo, h.hi, s.lo));
  return d2{t, __fadd2_rn(sub2(lo, ne), e)};
}

// FP64 value times 2^(ks + 896) as hi + lo by integer operations: hi its leading 24 bits (truncated), lo the other 29
// rounded to 24, so hi + lo is the value to 2^-48.  Below FP32's normal range it is 0, above (and for infinities and
// NaN) infinite.  |ks + 896| <= 890.
__device__ __forceinline__ void split_f64(double d, int ks, float &hi, float &lo) {
  const unsigned H = (unsigned)__double2hiint(d), L = (unsigned)__double2loint(d), sign = H & 0x80000000u;
  const int t = (int)(H & 0x7fffffffu) + ks * (1 << 20);  // exponent rebased to FP32's, upper 20 fraction bits
  const int ex = t >> 20;
  const float big = __uint_as_float(sign | 0x7f800000u);
  hi = ex < 1 ? 0.f : ex > 254 ? big : __uint_as_float(sign | __funnelshift_l(L, (unsigned)t, 3));
  const float unit = ex > 52 && ex < 255 ? __uint_as_float(sign | ((unsigned)(ex - 52) << 23)) : 0.f;
  lo = (float)(L & 0x1fffffffu) * unit;
}
// column shift ks of split_f64 for a factor that is a power of two
__device__ __forceinline__ int split_shift(double pow2) { return ((__double2hiint(pow2) >> 20) & 0x7ff) - 1023 - 896; }

// loaders of a pair-layout field (or of its hi and lo parts) at half-lattice site h
struct DfLoad1 {
  const float4 *f;
  struct Raw {
    float4 u[3], l[3];
  };
  template <class LN> __device__ __forceinline__ Raw load(const LN &ln, int h, int cl) const {
    const float4 *q = f + (int64_t)h * 12 * ln.P + ln.jp;
    Raw w;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      w.u[k] = q[ln.cu + k * ln.P];
      w.l[k] = q[cl + k * ln.P];
    }
    return w;
  }
  // u + s l or u + i s l
  __device__ __forceinline__ static z2 half(const Raw &w, int k, bool imag, float2 s, float2 n) {
    const c2 u = Pair2<float>::widen(w.u[k]), l = Pair2<float>::widen(w.l[k]);
    const d2 ur{u.re, f2(0.f)}, ui{u.im, f2(0.f)};
    return imag ? z2{axs1(ur, l.im, n), axs1(ui, l.re, s)} : z2{axs1(ur, l.re, s), axs1(ui, l.im, s)};
  }
};
struct DfLoad2 {
  DfLoad1 hi, lo;
  struct Raw {
    DfLoad1::Raw hi, lo;
  };
  template <class LN> __device__ __forceinline__ Raw load(const LN &ln, int h, int cl) const {
    return Raw{hi.load(ln, h, cl), lo.load(ln, h, cl)};
  }
  __device__ __forceinline__ static z2 half(const Raw &w, int k, bool imag, float2 s, float2 n) {
    const c2 uh = Pair2<float>::widen(w.hi.u[k]), lh = Pair2<float>::widen(w.hi.l[k]);
    const c2 ul = Pair2<float>::widen(w.lo.u[k]), ll = Pair2<float>::widen(w.lo.l[k]);
    const z2 u{d2{uh.re, ul.re}, d2{uh.im, ul.im}}, l{d2{lh.re, ll.re}, d2{lh.im, ll.im}};
    return imag ? axis(u, l, s, n) : axs(u, l, s);
  }
};

template <int MU, bool FWD, class LN, class LD>
__device__ __forceinline__ void hop_df_dir(const LN &ln, const float4 *__restrict__ U, const LD &in, int hn, z2 (&Su)[3],
                                           z2 (&L)[3]) {
  const typename LD::Raw raw = in.load(ln, hn, MU < 2 ? ln.clx : ln.clz);
  const float2 one = f2(1.f), mone = f2(-1.f);
  const float2 s = FWD ? (MU == 0 ? one : MU == 3 ? mone : ln.sg) : (MU == 0 ? mone : MU == 3 ? one : ln.ng);
  const float2 n = FWD ? (MU == 0 ? mone : MU == 3 ? one : ln.ng) : (MU == 0 ? one : MU == 3 ? mone : ln.sg);
  z2 h[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) h[a] = LD::half(raw, a, MU == 0 || MU == 2, s, n);
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    z2 w;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const float4 m = __ldg(U + (FWD ? 3 * a + c : 3 * c + a));  // Re hi, Re lo, Im hi, Im lo
      const dm r = dmul(m.x, m.y);
      // forward m h, backward conj(m) h
      const dm i = dmul(m.z, m.w), ni = dm{i.nhi, i.hi, f2(-m.w)};
      if (c == 0) {
        w.re = prod(r, h[0].re);
        w.im = prod(r, h[0].im);
      } else {
        w.re = mac(r, h[c].re, w.re);
        w.im = mac(r, h[c].im, w.im);
      }
      w.re = mac(FWD ? ni : i, h[c].im, w.re);
      w.im = mac(FWD ? i : ni, h[c].re, w.im);
    }
    Su[a] = axs(Su[a], w, one);
    if (MU == 0) L[a] = axis(L[a], w, FWD ? one : mone, FWD ? mone : one);
    if (MU == 1) L[a] = axs(L[a], w, FWD ? ln.ng : ln.sg);
    if (MU == 2) L[a] = axis(L[a], w, FWD ? ln.sg : ln.ng, FWD ? ln.ng : ln.sg);
    if (MU == 3) L[a] = axs(L[a], w, FWD ? one : mone);
  }
}

// this row of (H psi)(s) (see hop_eo); U: links split into hi and lo, [site][mu][3][3]
template <class LN, class LD>
__device__ __forceinline__ void hop_df(const LN &ln, const float4 *__restrict__ U, const LD &in, const Geom &g,
                                       const EoSite &s, z2 (&Su)[3], z2 (&Sl)[3]) {
#pragma unroll
  for (int a = 0; a < 3; ++a) Su[a] = Sl[a] = z2{dzero(), dzero()};
  const int hx = g.L[0] >> 1, odd = s.x & 1, h = s.h;
  const float4 *Us = U + (int64_t)eo_lex(s) * 36;
  {
    const int hf = odd ? (s.x == g.L[0] - 1 ? h - (hx - 1) : h + 1) : h;
    const int hb = odd ? h : (s.x == 0 ? h + (hx - 1) : h - 1);
    hop_df_dir<0, true>(ln, Us, in, hf, Su, Sl);
    hop_df_dir<0, false>(ln, U + (int64_t)(2 * hb + 1 - odd) * 36, in, hb, Su, Sl);
  }
  int st = hx;
  {
    const int hf = s.y == g.L[1] - 1 ? h - (g.L[1] - 1) * st : h + st;
    const int hb = s.y == 0 ? h + (g.L[1] - 1) * st : h - st;
    hop_df_dir<1, true>(ln, Us + 9, in, hf, Su, Sl);
    hop_df_dir<1, false>(ln, U + (int64_t)(2 * hb + odd) * 36 + 9, in, hb, Su, Sl);
  }
  // so far Sl belongs to the partner's row
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    Sl[a].re = d2{LN::other_row(Sl[a].re.hi), LN::other_row(Sl[a].re.lo)};
    Sl[a].im = d2{LN::other_row(Sl[a].im.hi), LN::other_row(Sl[a].im.lo)};
  }
  st *= g.L[1];
  {
    const int hf = s.z == g.L[2] - 1 ? h - (g.L[2] - 1) * st : h + st;
    const int hb = s.z == 0 ? h + (g.L[2] - 1) * st : h - st;
    hop_df_dir<2, true>(ln, Us + 18, in, hf, Su, Sl);
    hop_df_dir<2, false>(ln, U + (int64_t)(2 * hb + odd) * 36 + 18, in, hb, Su, Sl);
  }
  st *= g.L[2];
  {
    const int hf = s.t == g.L[3] - 1 ? h - (g.L[3] - 1) * st : h + st;
    const int hb = s.t == 0 ? h + (g.L[3] - 1) * st : h - st;
    hop_df_dir<3, true>(ln, Us + 27, in, hf, Su, Sl);
    hop_df_dir<3, false>(ln, U + (int64_t)(2 * hb + odd) * 36 + 27, in, hb, Su, Sl);
  }
}

// sum of squares of a field's values in double-float, one lane per column
struct Norm2 {
  d2 s;
  __device__ __forceinline__ Norm2() : s(dzero()) {}
  __device__ __forceinline__ void add1(d2 a) {  // a renormalised
    const float2 p = __fmul2_rn(a.hi, a.hi);
    const float2 e = __ffma2_rn(a.hi, a.hi, make_float2(-p.x, -p.y));
    const float2 t = __fadd2_rn(s.hi, p);
    const float2 nb = sub2(s.hi, t);
    const float2 q = __fadd2_rn(sub2(s.hi, __fadd2_rn(t, nb)), __fadd2_rn(p, nb));
    const float2 al = __fadd2_rn(a.lo, a.lo);
    s = d2{t, __fadd2_rn(__fadd2_rn(__ffma2_rn(al, a.hi, s.lo), e), q)};
  }
  __device__ __forceinline__ void add(z2 v) {
    add1(v.re);
    add1(v.im);
  }
  __device__ __forceinline__ double col(int c) const {
    return c ? (double)s.hi.y + (double)s.lo.y : (double)s.hi.x + (double)s.lo.x;
  }
};

}  // namespace dtr
