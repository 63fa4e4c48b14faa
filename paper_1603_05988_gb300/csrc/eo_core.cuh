// Red-black (even-odd) half-lattice stencil in FP32, two right-hand sides per thread.
//
// With the sites split by the parity of x + y + z + t the operator is
//   A = [[D, -H_eo / 2], [-H_oe / 2, D]],  D = 4 + m0,
// H the sum of the eight hops (each hop changes the parity).  Eliminating the odd sites leaves the Schur
// complement on the even ones,
//   S = D - H_eo H_oe / (4 D),   S x_e = r_e + H_eo r_o / (2 D),   x_o = (r_o + H_oe x_e / 2) / D,
// whose spectrum is so much narrower that BiCGStab takes half the iterations (8^4, eps 0.7, m0 -0.6, to 1e-10:
// 12 instead of 24; eps 0.2, m0 -0.15: 88 instead of 177), on vectors half as long; one application of S is the
// same eight hops per site as one of A.  The residual of the whole system is the Schur residual on the even sites
// and zero on the odd ones, so tolerances carry over unchanged.
//
// Half-lattice index: sites 2h and 2h + 1 (x even and odd, Lx is even) hold one even and one odd site, so both
// sublattices are indexed by h = site >> 1, and the neighbours in y, z, t of the site at h lie at the same h
// offsets as on the whole lattice.
//
// Fields are [h][12][b] complex (b a power of two, 2..64).  A thread works on columns 2 jp and 2 jp + 1 in the two
// lanes of packed FP32x2 instructions (half the issue slots of the scalar form).  Krylov vectors are stored as
// {Re_2jp, Re_2jp+1, Im_2jp, Im_2jp+1} so that a load lands in the lanes without moves.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "dtr_internal.cuh"

namespace dtr {

// two complex numbers, one per column
struct c2 {
  float2 re, im;
};
__device__ __forceinline__ float2 f2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, f2(-1.f), a); }
__device__ __forceinline__ c2 zero2() { return c2{f2(0.f), f2(0.f)}; }
__device__ __forceinline__ c2 scale2(c2 a, float2 s) { return c2{__fmul2_rn(a.re, s), __fmul2_rn(a.im, s)}; }
// a + s b, complex s per column (its negated imaginary part given, so that no lane is negated per element)
struct s2 {
  float2 re, im, nim;
};
__device__ __forceinline__ c2 axpy2(const s2 &s, c2 b, c2 a) {
  return c2{__ffma2_rn(s.re, b.re, __ffma2_rn(s.nim, b.im, a.re)),
            __ffma2_rn(s.re, b.im, __ffma2_rn(s.im, b.re, a.im))};
}
// u + w l for w = 1, i, -1, -i (W = 0..3)
template <int W> __device__ __forceinline__ c2 addw(c2 u, c2 l) {
  if (W == 0) return c2{__fadd2_rn(u.re, l.re), __fadd2_rn(u.im, l.im)};
  if (W == 1) return c2{sub2(u.re, l.im), __fadd2_rn(u.im, l.re)};
  if (W == 2) return c2{sub2(u.re, l.re), sub2(u.im, l.im)};
  return c2{__fadd2_rn(u.re, l.im), sub2(u.im, l.re)};
}

// ---------------------------------------------------------------- storage
// Two complex values of adjacent columns: FP32 (16 bytes), FP16 or BF16 (8 bytes).
template <typename S> struct Pair2;
template <> struct Pair2<float> {
  typedef float4 T;
  __device__ __forceinline__ static c2 widen(float4 v) { return c2{make_float2(v.x, v.y), make_float2(v.z, v.w)}; }
  __device__ __forceinline__ static float4 narrow(c2 v) { return make_float4(v.re.x, v.re.y, v.im.x, v.im.y); }
};
struct __align__(8) h2pair { __half2 re, im; };
struct __align__(8) b2pair { __nv_bfloat162 re, im; };
template <> struct Pair2<__half> {
  typedef h2pair T;
  __device__ __forceinline__ static c2 widen(h2pair v) { return c2{__half22float2(v.re), __half22float2(v.im)}; }
  __device__ __forceinline__ static h2pair narrow(c2 v) {
    return h2pair{__float22half2_rn(v.re), __float22half2_rn(v.im)};
  }
};
template <> struct Pair2<__nv_bfloat16> {
  typedef b2pair T;
  __device__ __forceinline__ static c2 widen(b2pair v) { return c2{__bfloat1622float2(v.re), __bfloat1622float2(v.im)}; }
  __device__ __forceinline__ static b2pair narrow(c2 v) {
    return b2pair{__float22bfloat162_rn(v.re), __float22bfloat162_rn(v.im)};
  }
};

// Loaders: value of component c at half-lattice site h (columns 2 jp, 2 jp + 1); P = b / 2.
template <typename S> struct PairLoad {
  const typename Pair2<S>::T *f;
  int P, jp;
  __device__ __forceinline__ void get(int h, const int (&c)[12], c2 (&o)[12]) const {
    const typename Pair2<S>::T *q = f + (int64_t)h * 12 * P + jp;
    typename Pair2<S>::T v[12];
#pragma unroll
    for (int k = 0; k < 12; ++k) v[k] = q[c[k]];
#pragma unroll
    for (int k = 0; k < 12; ++k) o[k] = Pair2<S>::widen(v[k]);
  }
};
// r - a v on the fly
template <typename S> struct PairAxpyLoad {
  const typename Pair2<S>::T *r;
  const typename Pair2<S>::T *v;
  int P, jp;
  s2 ma;  // -a
  __device__ __forceinline__ void get(int h, const int (&c)[12], c2 (&o)[12]) const {
    const int64_t q = (int64_t)h * 12 * P + jp;
    typename Pair2<S>::T rr[12], vv[12];
#pragma unroll
    for (int k = 0; k < 12; ++k) {
      rr[k] = r[q + c[k]];
      vv[k] = v[q + c[k]];
    }
#pragma unroll
    for (int k = 0; k < 12; ++k) o[k] = axpy2(ma, Pair2<S>::widen(vv[k]), Pair2<S>::widen(rr[k]));
  }
};
// FP32 field stored as interleaved complex columns, [h][12][b] float2
struct CplxLoad {
  const float2 *__restrict__ f;
  int P, jp;
  __device__ __forceinline__ void get(int h, const int (&c)[12], c2 (&o)[12]) const {
    const float4 *q = (const float4 *)f + (int64_t)h * 12 * P + jp;
    float4 v[12];
#pragma unroll
    for (int k = 0; k < 12; ++k) v[k] = q[c[k]];
#pragma unroll
    for (int k = 0; k < 12; ++k) o[k] = c2{make_float2(v[k].x, v[k].z), make_float2(v[k].y, v[k].w)};
  }
};

// ---------------------------------------------------------------- stencil
// Su += w, Sl += +-B^H w for w = U h (FWD) or U^H h, h = u -+ B l the half spinor of the neighbour at hn.
template <int MU, bool FWD, class LD>
__device__ __forceinline__ void hop_eo_dir(const float2 *__restrict__ Ul, const LD &in, int hn, const int (&c)[12],
                                           c2 (&Su)[2][3], c2 (&Sl)[2][3]) {
  c2 f[12];
  in.get(hn, c, f);
  float2 m[9];
#pragma unroll
  for (int k = 0; k < 9; ++k) m[k] = __ldg(Ul + k);
  // B l = (-i l1, -i l0), (-l1, l0), (-i l0, i l1), (l0, l1) for x, y, z, t; h = u - B l forward, u + B l backward
  constexpr int W0 = (MU == 0) ? 1 : (MU == 1) ? 0 : (MU == 2) ? 1 : 2;  // power of i in -B, upper row
  constexpr int W1 = (MU == 0) ? 1 : (MU == 1) ? 2 : (MU == 2) ? 3 : 2;  // lower row
  constexpr int F = FWD ? 0 : 2;
  constexpr int r0 = (MU == 0 || MU == 1) ? 1 : 0;                        // spin of l that enters the upper row
  c2 h[2][3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    h[0][a] = addw<(W0 + F) & 3>(f[a], f[6 + 3 * r0 + a]);
    h[1][a] = addw<(W1 + F) & 3>(f[3 + a], f[6 + 3 * (1 - r0) + a]);
  }
  // B^H w = (i w1, i w0), (w1, -w0), (i w0, -i w1), (w0, w1); + forward, - backward
  constexpr int V0 = (MU == 0) ? 1 : (MU == 1) ? 0 : (MU == 2) ? 1 : 0;
  constexpr int V1 = (MU == 0) ? 1 : (MU == 1) ? 2 : (MU == 2) ? 3 : 0;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    c2 w[2];
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      // the products with a minus sign are summed apart and subtracted once
      float2 pos, neg, sum;
      if (FWD) {  // sum_c U[a][c] h_c
        const float2 m0 = m[3 * a], m1 = m[3 * a + 1], m2 = m[3 * a + 2];
        pos = __ffma2_rn(f2(m2.x), h[s][2].re, __ffma2_rn(f2(m1.x), h[s][1].re, __fmul2_rn(f2(m0.x), h[s][0].re)));
        neg = __ffma2_rn(f2(m2.y), h[s][2].im, __ffma2_rn(f2(m1.y), h[s][1].im, __fmul2_rn(f2(m0.y), h[s][0].im)));
        sum = __ffma2_rn(f2(m2.x), h[s][2].im, __ffma2_rn(f2(m1.x), h[s][1].im, __fmul2_rn(f2(m0.x), h[s][0].im)));
        sum = __ffma2_rn(f2(m2.y), h[s][2].re, __ffma2_rn(f2(m1.y), h[s][1].re, __ffma2_rn(f2(m0.y), h[s][0].re, sum)));
        w[s] = c2{sub2(pos, neg), sum};
      } else {  // sum_c conj(U[c][a]) h_c
        const float2 m0 = m[a], m1 = m[3 + a], m2 = m[6 + a];
        pos = __ffma2_rn(f2(m2.x), h[s][2].im, __ffma2_rn(f2(m1.x), h[s][1].im, __fmul2_rn(f2(m0.x), h[s][0].im)));
        neg = __ffma2_rn(f2(m2.y), h[s][2].re, __ffma2_rn(f2(m1.y), h[s][1].re, __fmul2_rn(f2(m0.y), h[s][0].re)));
        sum = __ffma2_rn(f2(m2.x), h[s][2].re, __ffma2_rn(f2(m1.x), h[s][1].re, __fmul2_rn(f2(m0.x), h[s][0].re)));
        sum = __ffma2_rn(f2(m2.y), h[s][2].im, __ffma2_rn(f2(m1.y), h[s][1].im, __ffma2_rn(f2(m0.y), h[s][0].im, sum)));
        w[s] = c2{sum, sub2(pos, neg)};
      }
    }
    Su[0][a] = addw<0>(Su[0][a], w[0]);
    Su[1][a] = addw<0>(Su[1][a], w[1]);
    Sl[0][a] = addw<(V0 + F) & 3>(Sl[0][a], w[r0]);
    Sl[1][a] = addw<(V1 + F) & 3>(Sl[1][a], w[1 - r0]);
  }
}

// half-lattice geometry of one site
struct EoSite {
  int h;      // half-lattice index
  int x, y, z, t;
};
// the site of parity q at half-lattice index h
__device__ __forceinline__ EoSite eo_site(const Geom &g, int h, int q) {
  int c[4];
  site_coords(g, 2 * h, c);
  return EoSite{h, c[0] + ((c[1] + c[2] + c[3] + q) & 1), c[1], c[2], c[3]};
}
__device__ __forceinline__ int eo_lex(const EoSite &s) { return 2 * s.h + (s.x & 1); }

// (H psi)(s) without its signs on the lower spins: upper part Su, lower part -Sl.
template <class LD>
__device__ __forceinline__ void hop_eo(const float2 *__restrict__ U, const LD &in, const Geom &g, const EoSite &s,
                                       c2 (&Su)[2][3], c2 (&Sl)[2][3]) {
#pragma unroll
  for (int r = 0; r < 2; ++r)
#pragma unroll
    for (int a = 0; a < 3; ++a) Su[r][a] = Sl[r][a] = zero2();
  const int P = in.P;
  const int c[12] = {0, P, 2 * P, 3 * P, 4 * P, 5 * P, 6 * P, 7 * P, 8 * P, 9 * P, 10 * P, 11 * P};
  const int hx = g.L[0] >> 1, odd = s.x & 1, h = s.h;
  const int lex = eo_lex(s);
  const float2 *Us = U + (int64_t)lex * 36;
  {
    // x: the pair (2h, 2h + 1) holds one of the two neighbours
    const int hf = odd ? (s.x == g.L[0] - 1 ? h - (hx - 1) : h + 1) : h;
    const int hb = odd ? h : (s.x == 0 ? h + (hx - 1) : h - 1);
    hop_eo_dir<0, true>(Us, in, hf, c, Su, Sl);
    hop_eo_dir<0, false>(U + (int64_t)(2 * hb + 1 - odd) * 36, in, hb, c, Su, Sl);
  }
  int st = hx;
  {
    const int hf = s.y == g.L[1] - 1 ? h - (g.L[1] - 1) * st : h + st;
    const int hb = s.y == 0 ? h + (g.L[1] - 1) * st : h - st;
    hop_eo_dir<1, true>(Us + 9, in, hf, c, Su, Sl);
    hop_eo_dir<1, false>(U + (int64_t)(2 * hb + odd) * 36 + 9, in, hb, c, Su, Sl);
  }
  st *= g.L[1];
  {
    const int hf = s.z == g.L[2] - 1 ? h - (g.L[2] - 1) * st : h + st;
    const int hb = s.z == 0 ? h + (g.L[2] - 1) * st : h - st;
    hop_eo_dir<2, true>(Us + 18, in, hf, c, Su, Sl);
    hop_eo_dir<2, false>(U + (int64_t)(2 * hb + odd) * 36 + 18, in, hb, c, Su, Sl);
  }
  st *= g.L[2];
  {
    const int hf = s.t == g.L[3] - 1 ? h - (g.L[3] - 1) * st : h + st;
    const int hb = s.t == 0 ? h + (g.L[3] - 1) * st : h - st;
    hop_eo_dir<3, true>(Us + 27, in, hf, c, Su, Sl);
    hop_eo_dir<3, false>(U + (int64_t)(2 * hb + odd) * 36 + 27, in, hb, c, Su, Sl);
  }
}

}  // namespace dtr
