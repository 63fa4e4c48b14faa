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
// Fields are [h][12][b] complex (b a power of two, 2..64).  A work item is one site, one column pair 2 jp, 2 jp + 1
// and one spin row r (0 or 1): the columns sit in the two lanes of packed FP32x2 instructions (half the issue slots
// of the scalar form), and the two threads of a site and pair (lanes of one warp) each do one row of the half spinors.
// A row needs 6 of a neighbour's 12 components, none of them twice, so the split costs no field loads; it halves a
// thread's registers, which buys the warps that hide the load latency, and doubles the threads of a small lattice.
// Only the lower-spin sums of the x and y hops cross rows: they are exchanged once per site by shuffles.
// Krylov vectors are stored as {Re_2jp, Re_2jp+1, Im_2jp, Im_2jp+1} so that a load lands in the lanes without moves.
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
// u + s l and u + i s l, s real (+-1), n = -s
__device__ __forceinline__ c2 adds(c2 u, c2 l, float2 s) {
  return c2{__ffma2_rn(s, l.re, u.re), __ffma2_rn(s, l.im, u.im)};
}
__device__ __forceinline__ c2 addi(c2 u, c2 l, float2 s, float2 n) {
  return c2{__ffma2_rn(n, l.im, u.re), __ffma2_rn(s, l.re, u.im)};
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

// What a thread keeps for its work items: column pair, spin row and the offsets of its 6 components.  ROWBIT: the
// bit of the thread index that is the spin row.  4 (a half warp per row) for fields of 16 bytes per pair, whose loads
// go by quarter warps; 0 for the 8-byte ones (16^3 x 32 x 32, hop of A in us: FP32 140 against 148 with bit 0, FP16
// 129 against 136 with bit 4).
template <int ROWBIT> struct EoLane {
  int P;                    // column pairs, b / 2
  int jp;                   // this thread's
  int r;                    // spin row
  float2 sg, ng;            // +1, -1 for row 0; -1, +1 for row 1
  int cu, clx, clz;         // components: u_r, and l of the row's partner in x, y (1 - r) and z, t (r), times P
  __device__ __forceinline__ EoLane(int b, int tid) : P(b >> 1) {
    r = (tid >> ROWBIT) & 1;
    jp = (int)pair_of_item(tid) & (P - 1);
    sg = f2(r ? -1.f : 1.f);
    ng = f2(r ? 1.f : -1.f);
    cu = 3 * r * P;
    clx = (9 - 3 * r) * P;
    clz = (6 + 3 * r) * P;
  }
  // (site, column pair) that thread item `it` works on: 16 of them a warp
  __host__ __device__ __forceinline__ static constexpr int64_t pair_of_item(int64_t it) {
    return ROWBIT ? (it >> 5) * 16 + (it & 15) : it >> 1;
  }
  // v of the thread with the other spin row
  __device__ __forceinline__ static float2 other_row(float2 v) {
    return make_float2(__shfl_xor_sync(0xffffffffu, v.x, 1 << ROWBIT), __shfl_xor_sync(0xffffffffu, v.y, 1 << ROWBIT));
  }
};
template <typename S> constexpr int row_bit() { return sizeof(typename Pair2<S>::T) == 16 ? 4 : 0; }

// Loaders: load(h, cl) fetches components c + a P (a = 0, 1, 2) of u and l at half-lattice site h, value() turns them
// into FP32 pairs (apart, so that the next hop's loads are in flight while this one is computed).
template <typename S> struct PairLoad {
  typedef typename Pair2<S>::T ST;
  struct Raw {
    ST u[3], l[3];
  };
  const ST *f;
  template <class LN> __device__ __forceinline__ Raw load(const LN &ln, int h, int cl) const {
    const ST *q = f + (int64_t)h * 12 * ln.P + ln.jp;
    Raw w;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      w.u[k] = q[ln.cu + k * ln.P];
      w.l[k] = q[cl + k * ln.P];
    }
    return w;
  }
  __device__ __forceinline__ void value(const Raw &w, c2 (&u)[3], c2 (&l)[3]) const {
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      u[k] = Pair2<S>::widen(w.u[k]);
      l[k] = Pair2<S>::widen(w.l[k]);
    }
  }
};
// r - a v on the fly
template <typename S> struct PairAxpyLoad {
  typedef typename Pair2<S>::T ST;
  struct Raw {
    typename PairLoad<S>::Raw r, v;
  };
  const ST *r;
  const ST *v;
  s2 ma;  // -a
  template <class LN> __device__ __forceinline__ Raw load(const LN &ln, int h, int cl) const {
    return Raw{PairLoad<S>{r}.load(ln, h, cl), PairLoad<S>{v}.load(ln, h, cl)};
  }
  __device__ __forceinline__ void value(const Raw &w, c2 (&u)[3], c2 (&l)[3]) const {
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      u[k] = axpy2(ma, Pair2<S>::widen(w.v.u[k]), Pair2<S>::widen(w.r.u[k]));
      l[k] = axpy2(ma, Pair2<S>::widen(w.v.l[k]), Pair2<S>::widen(w.r.l[k]));
    }
  }
};
// ---------------------------------------------------------------- stencil
// One hop for one spin row: Su += w, L += +-B^H w, w = U h (FWD) or U^H h, h = u - B l (FWD) or u + B l the row of
// the neighbour's half spinor (raw: its loaded components).
template <int MU, bool FWD, class LN, class LD>
__device__ __forceinline__ void hop_eo_dir(const LN &ln, const float2 *__restrict__ Ul, const LD &in,
                                           const typename LD::Raw &raw, c2 (&Su)[3], c2 (&L)[3]) {
  c2 h[3], l[3];
  in.value(raw, h, l);
  float2 m[9];
  {
    const float4 *q = (const float4 *)Ul;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float4 v = __ldg(q + k);
      m[2 * k] = make_float2(v.x, v.y);
      m[2 * k + 1] = make_float2(v.z, v.w);
    }
    m[8] = __ldg(Ul + 8);
  }
  // -B = (i, i), (1, -1), (i, -i), (-1, -1) on the partner row for x, y, z, t, B^H its conjugate transpose's inverse
  // order: (i, i) on l's rows, (-1, 1), (i, -i), (1, 1) as seen from the row that holds w
  const float2 one = f2(1.f), mone = f2(-1.f);
  const float2 s = FWD ? (MU == 0 ? one : MU == 3 ? mone : ln.sg) : (MU == 0 ? mone : MU == 3 ? one : ln.ng);
  const float2 n = FWD ? (MU == 0 ? mone : MU == 3 ? one : ln.ng) : (MU == 0 ? one : MU == 3 ? mone : ln.sg);
#pragma unroll
  for (int a = 0; a < 3; ++a) h[a] = (MU == 0 || MU == 2) ? addi(h[a], l[a], s, n) : adds(h[a], l[a], s);
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    // the products with a minus sign are summed apart and subtracted once
    float2 pos, neg, sum;
    c2 w;
    if (FWD) {  // sum_c U[a][c] h_c
      const float2 m0 = m[3 * a], m1 = m[3 * a + 1], m2 = m[3 * a + 2];
      pos = __ffma2_rn(f2(m2.x), h[2].re, __ffma2_rn(f2(m1.x), h[1].re, __fmul2_rn(f2(m0.x), h[0].re)));
      neg = __ffma2_rn(f2(m2.y), h[2].im, __ffma2_rn(f2(m1.y), h[1].im, __fmul2_rn(f2(m0.y), h[0].im)));
      sum = __ffma2_rn(f2(m2.x), h[2].im, __ffma2_rn(f2(m1.x), h[1].im, __fmul2_rn(f2(m0.x), h[0].im)));
      sum = __ffma2_rn(f2(m2.y), h[2].re, __ffma2_rn(f2(m1.y), h[1].re, __ffma2_rn(f2(m0.y), h[0].re, sum)));
      w = c2{sub2(pos, neg), sum};
    } else {  // sum_c conj(U[c][a]) h_c
      const float2 m0 = m[a], m1 = m[3 + a], m2 = m[6 + a];
      pos = __ffma2_rn(f2(m2.x), h[2].im, __ffma2_rn(f2(m1.x), h[1].im, __fmul2_rn(f2(m0.x), h[0].im)));
      neg = __ffma2_rn(f2(m2.y), h[2].re, __ffma2_rn(f2(m1.y), h[1].re, __fmul2_rn(f2(m0.y), h[0].re)));
      sum = __ffma2_rn(f2(m2.x), h[2].re, __ffma2_rn(f2(m1.x), h[1].re, __fmul2_rn(f2(m0.x), h[0].re)));
      sum = __ffma2_rn(f2(m2.y), h[2].im, __ffma2_rn(f2(m1.y), h[1].im, __ffma2_rn(f2(m0.y), h[0].im, sum)));
      w = c2{sum, sub2(pos, neg)};
    }
    Su[a] = adds(Su[a], w, one);
    if (MU == 0) L[a] = addi(L[a], w, FWD ? one : mone, FWD ? mone : one);
    if (MU == 1) L[a] = adds(L[a], w, FWD ? ln.ng : ln.sg);
    if (MU == 2) L[a] = addi(L[a], w, FWD ? ln.sg : ln.ng, FWD ? ln.ng : ln.sg);
    if (MU == 3) L[a] = adds(L[a], w, FWD ? one : mone);
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

// This row of (H psi)(s): upper spin Su, and Sl, minus the lower spin.  All lanes of a warp take part.
// AHEAD: hops whose field loads are issued before they are needed (0 or 1).
template <int AHEAD, class LN, class LD>
__device__ __forceinline__ void hop_eo(const LN &ln, const float2 *__restrict__ U, const LD &in, const Geom &g,
                                       const EoSite &s, c2 (&Su)[3], c2 (&Sl)[3]) {
#pragma unroll
  for (int a = 0; a < 3; ++a) Su[a] = Sl[a] = zero2();
  const int hx = g.L[0] >> 1, odd = s.x & 1, h = s.h;
  constexpr int K = kLink32;
  const float2 *Us = U + (int64_t)eo_lex(s) * (4 * K);
  int hf[4], hb[4];
  // x: the pair (2h, 2h + 1) holds one of the two neighbours
  hf[0] = odd ? (s.x == g.L[0] - 1 ? h - (hx - 1) : h + 1) : h;
  hb[0] = odd ? h : (s.x == 0 ? h + (hx - 1) : h - 1);
  const int sy = hx, sz = sy * g.L[1], st = sz * g.L[2];
  hf[1] = s.y == g.L[1] - 1 ? h - (g.L[1] - 1) * sy : h + sy;
  hb[1] = s.y == 0 ? h + (g.L[1] - 1) * sy : h - sy;
  hf[2] = s.z == g.L[2] - 1 ? h - (g.L[2] - 1) * sz : h + sz;
  hb[2] = s.z == 0 ? h + (g.L[2] - 1) * sz : h - sz;
  hf[3] = s.t == g.L[3] - 1 ? h - (g.L[3] - 1) * st : h + st;
  hb[3] = s.t == 0 ? h + (g.L[3] - 1) * st : h - st;
#define DTR_BLINK(mu, o) (U + (int64_t)(2 * hb[mu] + (o)) * (4 * K) + (mu) * K)
  typename LD::Raw r0, r1;
  r0 = in.load(ln, hf[0], ln.clx);
  if (AHEAD) r1 = in.load(ln, hb[0], ln.clx);
  hop_eo_dir<0, true>(ln, Us, in, r0, Su, Sl);
  (AHEAD ? r0 : r1) = in.load(ln, AHEAD ? hf[1] : hb[0], ln.clx);
  hop_eo_dir<0, false>(ln, DTR_BLINK(0, 1 - odd), in, r1, Su, Sl);
  (AHEAD ? r1 : r0) = in.load(ln, AHEAD ? hb[1] : hf[1], ln.clx);
  hop_eo_dir<1, true>(ln, Us + K, in, r0, Su, Sl);
  (AHEAD ? r0 : r1) = in.load(ln, AHEAD ? hf[2] : hb[1], AHEAD ? ln.clz : ln.clx);
  hop_eo_dir<1, false>(ln, DTR_BLINK(1, odd), in, r1, Su, Sl);
  (AHEAD ? r1 : r0) = in.load(ln, AHEAD ? hb[2] : hf[2], ln.clz);
  // so far Sl belongs to the partner's row
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    Sl[a].re = LN::other_row(Sl[a].re);
    Sl[a].im = LN::other_row(Sl[a].im);
  }
  hop_eo_dir<2, true>(ln, Us + 2 * K, in, r0, Su, Sl);
  (AHEAD ? r0 : r1) = in.load(ln, AHEAD ? hf[3] : hb[2], ln.clz);
  hop_eo_dir<2, false>(ln, DTR_BLINK(2, odd), in, r1, Su, Sl);
  (AHEAD ? r1 : r0) = in.load(ln, AHEAD ? hb[3] : hf[3], ln.clz);
  hop_eo_dir<3, true>(ln, Us + 3 * K, in, r0, Su, Sl);
  if (!AHEAD) r1 = in.load(ln, hb[3], ln.clz);
  hop_eo_dir<3, false>(ln, DTR_BLINK(3, odd), in, r1, Su, Sl);
#undef DTR_BLINK
}

// Work items [0, n) of one phase over the grid: full sweeps of the whole grid (neighbouring items run at the same
// time, so the stencil's neighbours meet in L2), and the remainder spread evenly over the blocks (a last sweep of the
// first blocks alone would leave the other SMs idle: 8^4 x 16 on 19 blocks is 3.4 sweeps).  The remainder goes by
// GRAIN items, a whole number of sites.  Runs whole warps, so items up to the next multiple of 32 are visited too.
template <int T, int GRAIN> struct Sweep {
  int64_t full, lo, hi;
  __device__ __forceinline__ explicit Sweep(int64_t n) {
    const int64_t G = gridDim.x, round = G * T;
    full = n / round * round;
    const int64_t ch = ((n - full + GRAIN - 1) / GRAIN + G - 1) / G * GRAIN;
    lo = full + blockIdx.x * ch;
    hi = min(n, lo + ch);
  }
  template <class F> __device__ __forceinline__ void run(const F &body) const {
    for (int64_t it = (int64_t)blockIdx.x * T + threadIdx.x; it < full; it += (int64_t)gridDim.x * T) body(it);
    const int64_t it = lo + threadIdx.x;
    if ((it & ~(int64_t)31) < hi) body(it);
  }
};

}  // namespace dtr
