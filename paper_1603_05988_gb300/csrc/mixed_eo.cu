// Defect correction of the mixed solvers on the red-black Schur complement (eo_core.cuh): the outer residuals in
// double-float arithmetic, the inner problem on the even sites, and the correction on both sublattices.
//
// The iterate x and the right-hand side z are FP64.  The residual is kept in double-float, times a power of two
// `base` per column that brings |z| to the square root of the unknowns (so no entry leaves FP32's range), and the
// inner right-hand sides are the residual times another power of two `fac`: both scalings are exact.
#include "mixed_eo.cuh"

#include "df_eo.cuh"
#include "krylov_fin.cuh"

namespace dtr {

static size_t al(size_t x) { return (x + 255) / 256 * 256; }
static int log2i(int b) {
  int l = 0;
  while ((1 << l) < b) ++l;
  return l;
}
static size_t half_bytes(int64_t V, int b) { return al((size_t)(V / 2) * 12 * eo_width(b) * sizeof(float2)); }

size_t eo_scratch_bytes(int64_t V, int b) { return 12 * half_bytes(V, b); }

EoBufs eo_carve(char *w, int64_t V, int b) {
  const size_t half = half_bytes(V, b);
  EoBufs B;
  B.rhi = (float4 *)w;
  B.rlo = (float4 *)(w + 2 * half);
  B.e = (float4 *)(w + 4 * half);
  B.r = w + 6 * half;
  B.rhat = w + 7 * half;
  B.p = w + 8 * half;
  B.v = w + 9 * half;
  B.t = w + 10 * half;
  B.w = w + 11 * half;
  B.xhi = (float4 *)B.r;
  B.xlo = (float4 *)B.p;
  return B;
}

typedef EoLane<4> LN;

// what the kernels below need of a block
struct Blk {
  Geom g;
  int b, P, logp;
  int64_t half;  // float4 elements of one sublattice
};
static Blk blk_of(const EoSolve &S) {
  const int P = eo_width(S.b) / 2;
  return Blk{S.g, S.b, P, log2i(P), (int64_t)(S.g.V / 2) * 12 * P};
}

// body(h, valid) for the work items of all half-lattice sites, in whole warps (the stencil's lanes exchange values)
template <class F> __device__ __forceinline__ void for_eo_items(const Blk &k, const F &body) {
  const int64_t npair = (int64_t)(k.g.V >> 1) << k.logp;
  for (int64_t it = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; (it & ~(int64_t)31) < 2 * npair;
       it += (int64_t)gridDim.x * blockDim.x) {
    const int64_t pr = LN::pair_of_item(it);
    body(pr < npair ? (int)(pr >> k.logp) : 0, pr < npair);
  }
}
// the same over the sites of both sublattices in one range: body(parity, h, valid)
template <class F> __device__ __forceinline__ void for_all_items(const Blk &k, const F &body) {
  const int64_t npair = (int64_t)(k.g.V >> 1) << k.logp, row = (2 * npair + 31) & ~(int64_t)31;  // whole warps
  for (int64_t it = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; it < 2 * row;
       it += (int64_t)gridDim.x * blockDim.x) {
    const int parity = it >= row;
    const int64_t pr = LN::pair_of_item(parity ? it - row : it);
    body(parity, pr < npair ? (int)(pr >> k.logp) : 0, pr < npair);
  }
}
// offset of this thread's component c (0..2 upper, 3..5 lower spin) in units of a component
__device__ __forceinline__ int comp_of(const LN &ln, int c) { return (c < 3 ? 0 : 6) + 3 * ln.r + c % 3; }

// Grid sums of one value per column from threads that hold those of their pair (acc[0], acc[1]): true in the last
// block, where col_total gives column j's.
__device__ __forceinline__ int pair_width(int P) { return P <= 16 ? P : 64; }
__device__ __forceinline__ bool pair_reduce(const double (&acc)[2], int P, const Reduce &red, double2 *tot) {
  const double2 v[2] = {make_double2(acc[0], 0.0), make_double2(acc[1], 0.0)};
  return block_reduce<2>(v, pair_width(P), red.partial, red.counter, tot);
}
__device__ __forceinline__ double col_total(const double2 *tot, int P, int j) {
  const int jp = j >> 1, q = (j & 1) * pair_width(P);
  // a thread's pair is threadIdx.x & (P - 1) up to P = 16; with P = 32 the row bit sits in between
  return P <= 16 ? tot[q + jp].x : tot[q + (jp & 15) + 2 * (jp & 16)].x + tot[q + (jp & 15) + 2 * (jp & 16) + 16].x;
}

// 2^floor(log2 v), within 2^+-800
__device__ __forceinline__ double pow2_below(double v) {
  int e = ((__double2hiint(v) >> 20) & 0x7ff) - 1023;
  e = min(800, max(-800, e));
  return __hiloint2double((e + 1023) << 20, 0);
}
// 1 / v for a power of two, on the integer pipe (an FP64 division is ~40 instructions at two lanes a clock)
__device__ __forceinline__ double pow2_inv(double v) {
  return __hiloint2double((2046 << 20) - (__double2hiint(v) & 0x7ff00000), 0);
}
__device__ __forceinline__ int pow2_exp(double v) { return ((__double2hiint(v) >> 20) & 0x7ff) - 1023; }
// f 2^-e in FP64, exact (integer pipe: a widening by instruction and a fused multiply are two FP64 instructions; the
// rest behind a call, see f64_to_f32)
__device__ __noinline__ double unscale_slow(float f, int e) { return scalbn((double)f, -e); }
__device__ __forceinline__ double unscale(float f, int e) {
  const unsigned b = __float_as_uint(f), m = b & 0x7fffffffu;
  const int x = (int)(m >> 23) + 896 - e;  // exponent field of the result
  if (m == 0u) return 0.0;
  if (m - 0x00800000u >= 0x7f000000u || x < 1 || x > 2046) return unscale_slow(f, e);
  return __hiloint2double((int)((b & 0x80000000u) | ((m >> 3) & 0x000fffffu) | ((unsigned)x << 20)), (int)(b << 29));
}
__device__ __forceinline__ void set_fac(Scal *sc, int j, double hs) {
  sc->fac[j] = sc->active[j] ? pow2_below(hs / (sqrt(sc->rtrue2[j]) * sc->base[j])) : 0.0;
}
// a residual norm (of the scaled residual) is known for every column
__device__ __forceinline__ void finish_resid(Scal *sc, const double2 *tot, int b, int P, int restart, double hs,
                                             int *mark, int marked) {
  const int j = threadIdx.x;
  if (j < b) {
    const double inv = pow2_inv(sc->base[j]);
    fin_resid(sc, j, make_double2(col_total(tot, P, j) * inv * inv, sc->bnorm2[j]), restart);
    set_fac(sc, j, hs);
  }
  __syncthreads();
  if (j == 0) {
    count_active(sc, b);
    if (mark) *mark = marked;
  }
}

// |z|^2 and the column scale; if x is zero also the residual's norm (r = z, split below)
__global__ void __launch_bounds__(kBlock) k_eo_znorm(const double2 *__restrict__ z, int64_t n, int b, Scal *sc,
                                                     Reduce red, double hs, double unit, const int *x_nonzero) {
  __shared__ double2 tot[64];
  double2 acc[1] = {make_double2(0.0, 0.0)};
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  for (; e + 3 * stride < n; e += 4 * stride) {
    double2 v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) v[u] = z[e + u * stride];
#pragma unroll
    for (int u = 0; u < 4; ++u) acc[0].x = fma(v[u].x, v[u].x, fma(v[u].y, v[u].y, acc[0].x));
  }
  for (; e < n; e += stride) acc[0].x = fma(z[e].x, z[e].x, fma(z[e].y, z[e].y, acc[0].x));
  if (block_reduce<1>(acc, b, red.partial, red.counter, tot)) {
    const int j = threadIdx.x;
    if (j < b) {
      const double z2 = tot[j].x;
      sc->bnorm2[j] = z2;
      sc->base[j] = z2 > 0.0 && z2 < 1e300 ? pow2_below(unit / sqrt(z2)) : 1.0;
      if (!x_nonzero || *(volatile const int *)x_nonzero == 0) {
        fin_resid(sc, j, make_double2(z2, z2), 1);
        set_fac(sc, j, hs);
      }
    }
    __syncthreads();
    if (j == 0) count_active(sc, b);
  }
}

// two columns' values of a whole-lattice FP64 field, scaled and split
__device__ __forceinline__ z2 split_pair(const double2 *f, bool two, int k0, int k1) {
  const double2 u = f[0];
  double2 v = make_double2(0.0, 0.0);
  if (two) v = f[1];
  z2 o;
  split_f64(u.x, k0, o.re.hi.x, o.re.lo.x);
  split_f64(u.y, k0, o.im.hi.x, o.im.lo.x);
  split_f64(v.x, k1, o.re.hi.y, o.re.lo.y);
  split_f64(v.y, k1, o.im.hi.y, o.im.lo.y);
  return o;
}
__device__ __forceinline__ float4 hi_of(z2 v) { return make_float4(v.re.hi.x, v.re.hi.y, v.im.hi.x, v.im.hi.y); }
__device__ __forceinline__ float4 lo_of(z2 v) { return make_float4(v.re.lo.x, v.re.lo.y, v.im.lo.x, v.im.lo.y); }
__device__ __forceinline__ z2 join(float4 h, float4 l) {
  const c2 a = Pair2<float>::widen(h), b = Pair2<float>::widen(l);
  return z2{d2{a.re, b.re}, d2{a.im, b.im}};
}

// f (FP64, [site][12][b]) times base, split into hi and lo in red-black order.  With a flag pointer also |f|^2 per
// column: where |x| / |z| exceeds kDfCertRatio the double-float residual's error (~1e-13 |x| / |z|) would no longer be
// negligible next to a 1e-10 tolerance, and *fp64_cert selects the FP64 residual instead.
constexpr double kDfCertRatio = 30.0;
__global__ void __launch_bounds__(kBlock) k_eo_split(const double2 *__restrict__ f, float4 *__restrict__ hi,
                                                     float4 *__restrict__ lo, Blk k, const Scal *sc, Reduce red,
                                                     int *fp64_cert, const int *run_flag, int run_if) {
  __shared__ double2 tot[2 * 64];
  __shared__ int any;
  if (run_flag && *(volatile const int *)run_flag != run_if) return;  // not selected (uniform over the grid)
  const LN ln(2 * k.P, threadIdx.x);
  const bool two = k.b > 1;
  const int k0 = split_shift(sc->base[2 * ln.jp]), k1 = two ? split_shift(sc->base[2 * ln.jp + 1]) : 0;
  double acc[2] = {0.0, 0.0};
  for_all_items(k, [&](int parity, int site, bool valid) {
    if (!valid) return;
    float4 *h = hi + parity * k.half, *l = lo + parity * k.half;
    const EoSite s = eo_site(k.g, site, parity);
    const double2 *src = f + (int64_t)eo_lex(s) * 12 * k.b + 2 * ln.jp;
    const int64_t q = (int64_t)site * 12 * k.P + ln.jp;
    float2 n = f2(0.f);
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      const int m = comp_of(ln, c);
      const z2 v = split_pair(src + m * k.b, two, k0, k1);
      h[q + m * k.P] = hi_of(v);
      l[q + m * k.P] = lo_of(v);
      n = __ffma2_rn(v.re.hi, v.re.hi, __ffma2_rn(v.im.hi, v.im.hi, n));
    }
    acc[0] += (double)n.x;
    acc[1] += (double)n.y;
  });
  if (!fp64_cert) return;
  if (pair_reduce(acc, k.P, red, tot)) {
    if (threadIdx.x == 0) any = 0;
    __syncthreads();
    if (threadIdx.x < k.b) {
      const int j = threadIdx.x;
      const double lim = kDfCertRatio * kDfCertRatio * sc->bnorm2[j] * sc->base[j] * sc->base[j];
      if (lim > 0.0 && col_total(tot, k.P, j) > lim) atomicOr(&any, 1);
    }
    __syncthreads();
    if (threadIdx.x == 0) *fp64_cert = any;
  }
}

// inner problem: r = rhat = p = fac (r_e + H r_o / (2 D)), e = 0 on the even sites, from the hi parts of the residual alone
// (truncated, not rounded, to 24 bits: the next outer residual takes that up with the rest); the inner scalars, with
// rho = |r|^2 and the norm that the tolerance refers to that of the whole residual
template <typename S>
__global__ void __launch_bounds__(kBlock, 2) k_eo_init(const float2 *__restrict__ U, const float4 *__restrict__ res,
                                                    typename Pair2<S>::T *__restrict__ r,
                                                    typename Pair2<S>::T *__restrict__ rhat,
                                                    typename Pair2<S>::T *__restrict__ p, float4 *__restrict__ e,
                                                    Blk k, float wscale, const Scal *__restrict__ outer, Scal *inner,
                                                    double tol2, int maxiter, Reduce red) {
  typedef Pair2<S> PS;
  __shared__ double2 tot[2 * 64];
  const LN ln(2 * k.P, threadIdx.x);
  const PairLoad<float> odd{res + k.half};
  const float2 fac = make_float2((float)outer->fac[2 * ln.jp], k.b > 1 ? (float)outer->fac[2 * ln.jp + 1] : 0.f);
  const float2 wp = f2(wscale), wm = f2(-wscale);
  float2 nrm = f2(0.f);
  for_eo_items(k, [&](int h, bool valid) {
    const EoSite s = eo_site(k.g, h, 0);
    c2 H[2][3];
    hop_eo<0>(ln, U, odd, k.g, s, H[0], H[1]);
    if (!valid) return;
    const int64_t q = (int64_t)h * 12 * k.P + ln.jp;
    float4 own[6];
#pragma unroll
    for (int c = 0; c < 6; ++c) own[c] = res[q + comp_of(ln, c) * k.P];
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      const c2 hk = H[c / 3][c % 3], o = Pair2<float>::widen(own[c]);
      const float2 f = c < 3 ? wp : wm;
      const int64_t i = q + comp_of(ln, c) * k.P;
      const typename PS::T st =
          PS::narrow(scale2(c2{__ffma2_rn(f, hk.re, o.re), __ffma2_rn(f, hk.im, o.im)}, fac));
      r[i] = st;
      rhat[i] = st;
      p[i] = st;
      e[i] = make_float4(0.f, 0.f, 0.f, 0.f);
      const c2 w = PS::widen(st);
      nrm = __ffma2_rn(w.re, w.re, __ffma2_rn(w.im, w.im, nrm));
    }
  });
  const double acc[2] = {(double)nrm.x, (double)nrm.y};
  if (pair_reduce(acc, k.P, red, tot)) {
    const int j = threadIdx.x;
    if (j < 2 * k.P) {
      const double rho = col_total(tot, k.P, j);
      const int act = j < k.b ? outer->active[j] : 0;
      const double f = act ? outer->fac[j] * outer->base[j] : 0.0;
      inner->active[j] = act;
      inner->rho[j] = make_double2(rho, 0.0);
      inner->bnorm2[j] = act ? outer->rtrue2[j] * f * f : 0.0;
      inner->rnorm2[j] = rho;
      inner->iters[j] = 0;
      inner->flags[j] = 0;
      inner->alpha[j] = inner->omega[j] = inner->beta[j] = make_double2(0.0, 0.0);
      if (j == 0) {
        int n = 0;
        for (int q = 0; q < k.b; ++q) n += outer->active[q];
        inner->n_active = n;
        inner->tol2 = tol2;
        inner->maxiter = maxiter;
      }
    }
  }
}

// e_o = (fac r_o + H e_e / 2) / D, x += e / (base fac) on both sublattices (one thread per site pair 2h, 2h + 1,
// column pair and spin row); folds the inner counters.  With gs: chooses the residual that ends this cycle (gs->sel):
// the double-float update if some active column is predicted (its last residual times the inner solve's achieved
// reduction) to stay more than 10x above tol, else the true residual, which then also certifies convergence.
__global__ void __launch_bounds__(kBlock, 2) k_eo_accum(const float2 *__restrict__ U, const float4 *__restrict__ res,
                                                     float4 *e, double2 *__restrict__ x, Blk k, float dinv,
                                                     Scal *outer, const Scal *__restrict__ inner, GridSync *gs) {
  if (gs && blockIdx.x == 0) {  // one column per thread of block 0
    const int q = threadIdx.x;
    int far = 0;
    if (q < k.b && outer->active[q]) {
      const double red2 = inner->bnorm2[q] > 0.0 ? inner->rnorm2[q] / inner->bnorm2[q] : 1.0;
      far = outer->rtrue2[q] * red2 > 100.0 * outer->tol2 * outer->bnorm2[q];
    }
    far = __syncthreads_or(far);
    if (q == 0) gs->sel = far ? 1 : 0;
  }
  const LN ln(2 * k.P, threadIdx.x);
  const PairLoad<float> even{e};
  const int j0 = 2 * ln.jp;
  const bool a0 = outer->active[j0] != 0, a1 = k.b > 1 && outer->active[j0 + 1] != 0;
  const int s0 = a0 ? pow2_exp(outer->fac[j0] * outer->base[j0]) : 0;
  const int s1 = a1 ? pow2_exp(outer->fac[j0 + 1] * outer->base[j0 + 1]) : 0;
  const float2 di = make_float2(a0 ? dinv * (float)outer->fac[j0] : 0.f, a1 ? dinv * (float)outer->fac[j0 + 1] : 0.f);
  const float2 dh = f2(0.5f * dinv), dmh = f2(-0.5f * dinv);
  for_eo_items(k, [&](int h, bool valid) {
    const EoSite s = eo_site(k.g, h, 1);
    c2 H[2][3], eo[6], ee[6];
    hop_eo<0>(ln, U, even, k.g, s, H[0], H[1]);
    if (!valid) return;
    const int64_t q = (int64_t)h * 12 * k.P + ln.jp;
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      eo[c] = Pair2<float>::widen(res[k.half + q + comp_of(ln, c) * k.P]);
      ee[c] = Pair2<float>::widen(e[q + comp_of(ln, c) * k.P]);
    }
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      const c2 hk = H[c / 3][c % 3];
      const float2 f = c < 3 ? dh : dmh;
      eo[c] = c2{__ffma2_rn(f, hk.re, __fmul2_rn(di, eo[c].re)), __ffma2_rn(f, hk.im, __fmul2_rn(di, eo[c].im))};
      e[k.half + q + comp_of(ln, c) * k.P] = Pair2<float>::narrow(eo[c]);
    }
    if (!a0 && !a1) return;
    const int lex = eo_lex(s);
#pragma unroll
    for (int side = 0; side < 2; ++side) {  // the odd site, then the even one of the pair 2h, 2h + 1
      double2 *xs = x + (int64_t)(side ? lex ^ 1 : lex) * 12 * k.b + j0;
      double2 v[6][2];
#pragma unroll
      for (int c = 0; c < 6; ++c) {
        const double2 *xp = xs + comp_of(ln, c) * k.b;
        v[c][0] = xp[0];
        if (k.b > 1) v[c][1] = xp[1];
      }
#pragma unroll
      for (int c = 0; c < 6; ++c) {
        const c2 d = side ? ee[c] : eo[c];
        double2 *xp = xs + comp_of(ln, c) * k.b;
        if (a0) xp[0] = make_double2(v[c][0].x + unscale(d.re.x, s0), v[c][0].y + unscale(d.im.x, s0));
        if (a1) xp[1] = make_double2(v[c][1].x + unscale(d.re.y, s1), v[c][1].y + unscale(d.im.y, s1));
      }
    }
  });
  if (blockIdx.x == 0 && threadIdx.x < k.b) {
    outer->iters[threadIdx.x] += inner->iters[threadIdx.x];
    outer->flags[threadIdx.x] |= inner->flags[threadIdx.x] & ~kFlagBreakdown;
  }
}

// Residual after a cycle without a stencil on x: x grew by e / (base fac), so r -= A e / fac, A e in double-float
// (links split into hi and lo, e exact in FP32): relative error ~2^-46 of |A| |e|, so r stays the true residual of x
// to ~1e-14 kappa |z| over all cycles; a true residual confirms convergence before it is reported.
// FP32 arithmetic and load latency bound it: two blocks to an SM (128 registers, ~150 B spilled) 13.4 ms against 14.7 ms
// for one (232 registers) at 32^3 x 64 x 16, each of the two that run in a solve; a loop over directions that needs no
// spills took 16.3 ms.
__global__ void __launch_bounds__(kBlock, 2) k_eo_update(const float4 *__restrict__ Udf, const float4 *__restrict__ e,
                                                         float4 *__restrict__ rhi, float4 *__restrict__ rlo, Blk k,
                                                         float dhi, float dlo, Scal *sc, Reduce red, double hs,
                                                         const int *run_flag, int run_if, int *mark) {
  __shared__ double2 tot[2 * 64];
  if (run_flag && *(volatile const int *)run_flag != run_if) return;  // not selected (uniform over the grid)
  const LN ln(2 * k.P, threadIdx.x);
  const int j0 = 2 * ln.jp;
  const float2 mg = make_float2(sc->active[j0] ? -(float)pow2_inv(sc->fac[j0]) : 0.f,
                                k.b > 1 && sc->active[j0 + 1] ? -(float)pow2_inv(sc->fac[j0 + 1]) : 0.f);
  const dm D = dmul(dhi, dlo);
  Norm2 nrm;
  for_all_items(k, [&](int parity, int site, bool valid) {
    const DfLoad1 in{e + (1 - parity) * k.half};
    const float4 *self = e + parity * k.half;
    float4 *h = rhi + parity * k.half, *l = rlo + parity * k.half;
    const EoSite s = eo_site(k.g, site, parity);
    z2 H[2][3];
    hop_df(ln, Udf, in, k.g, s, H[0], H[1]);
    if (!valid) return;
    const int64_t q = (int64_t)site * 12 * k.P + ln.jp;
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      const int64_t i = q + comp_of(ln, c) * k.P;
      const c2 v = Pair2<float>::widen(self[i]);
      z2 o{prod(D, d2{v.re, f2(0.f)}), prod(D, d2{v.im, f2(0.f)})};
      o = axs(o, H[c / 3][c % 3], f2(c < 3 ? -0.5f : 0.5f));
      z2 r = axs(join(h[i], l[i]), o, mg);
      r = z2{renorm(r.re), renorm(r.im)};
      h[i] = hi_of(r);
      l[i] = lo_of(r);
      nrm.add(r);
    }
  });
  const double acc[2] = {nrm.col(0), nrm.col(1)};
  if (pair_reduce(acc, k.P, red, tot)) finish_resid(sc, tot, k.b, k.P, 1, hs, mark, 1);
}

// True residual r = base (z - A x) with A x in double-float on the split x: each component carries an error of about
// 2^-46 times the sum of the stencil terms' magnitudes (~9 |x|), i.e. ~1e-13 |x| / |z| relative to z, a hundredth of a
// 1e-10 tolerance while |x| / |z| stays below ~10.  One block to an SM: 15.1 ms at 32^3 x 64 x 16 where it runs (once a
// solve), two blocks 16.5 ms.
__global__ void __launch_bounds__(kBlock, 1) k_eo_resid_df(const float4 *__restrict__ Udf,
                                                           const float4 *__restrict__ xhi,
                                                           const float4 *__restrict__ xlo,
                                                           const double2 *__restrict__ z, float4 *__restrict__ rhi,
                                                           float4 *__restrict__ rlo, Blk k, float dhi, float dlo,
                                                           Scal *sc, Reduce red, int restart, double hs,
                                                           const int *run_flag, int run_if, int *mark,
                                                           const int *fp64_cert) {
  __shared__ double2 tot[2 * 64];
  if (run_flag && *(volatile const int *)run_flag != run_if) return;  // not selected (uniform over the grid)
  if (*(volatile const int *)fp64_cert) return;                        // the FP64 residual runs instead
  const LN ln(2 * k.P, threadIdx.x);
  const bool two = k.b > 1;
  const int k0 = split_shift(sc->base[2 * ln.jp]), k1 = two ? split_shift(sc->base[2 * ln.jp + 1]) : 0;
  const dm D = dmul(dhi, dlo);
  Norm2 nrm;
  for_all_items(k, [&](int parity, int site, bool valid) {
    const int64_t nb = (1 - parity) * k.half, own = parity * k.half;
    const DfLoad2 in{DfLoad1{xhi + nb}, DfLoad1{xlo + nb}};
    const EoSite s = eo_site(k.g, site, parity);
    z2 H[2][3];
    hop_df(ln, Udf, in, k.g, s, H[0], H[1]);
    if (!valid) return;
    const int64_t q = own + (int64_t)site * 12 * k.P + ln.jp;
    const double2 *zs = z + (int64_t)eo_lex(s) * 12 * k.b + 2 * ln.jp;
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      const int m = comp_of(ln, c);
      const int64_t i = q + m * k.P;
      const z2 v = join(xhi[i], xlo[i]);
      z2 o{prod(D, v.re), prod(D, v.im)};
      o = axs(o, H[c / 3][c % 3], f2(c < 3 ? -0.5f : 0.5f));
      z2 r = axs(split_pair(zs + m * k.b, two, k0, k1), o, f2(-1.f));
      r = z2{renorm(r.re), renorm(r.im)};
      rhi[i] = hi_of(r);
      rlo[i] = lo_of(r);
      nrm.add(r);
    }
  });
  const double acc[2] = {nrm.col(0), nrm.col(1)};
  if (pair_reduce(acc, k.P, red, tot)) finish_resid(sc, tot, k.b, k.P, restart, hs, mark, 0);
}

// the same in FP64 (run where *fp64_cert is 1): one thread per site and column
__global__ void __launch_bounds__(kBlock) k_eo_resid64(const double2 *__restrict__ U, const double2 *__restrict__ x,
                                                       const double2 *__restrict__ z, float4 *__restrict__ rhi,
                                                       float4 *__restrict__ rlo, Blk k, int logb, double diag,
                                                       Scal *sc, Reduce red, int restart, double hs,
                                                       const int *run_flag, int run_if, int *mark,
                                                       const int *fp64_cert) {
  __shared__ double2 tot[64];
  if (run_flag && *(volatile const int *)run_flag != run_if) return;  // not selected (uniform over the grid)
  if (*(volatile const int *)fp64_cert != 1) return;
  const int b = k.b, j = threadIdx.x & (b - 1);
  const int ks = split_shift(sc->base[j]);
  double2 acc[1] = {make_double2(0.0, 0.0)};
  const int64_t n = (int64_t)k.g.V << logb;
  for (int64_t it = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; it < n; it += (int64_t)gridDim.x * blockDim.x) {
    const int s = (int)(it >> logb);
    double2 o[12], self[12];
    dslash_site<1, double>(U, x, k.g, b, s, j, diag, o, self);
    const int64_t base = (int64_t)s * 12 * b + j;
    const int64_t q = (site_parity(k.g, s) ? k.half : 0) + (int64_t)(s >> 1) * 12 * k.P + (j >> 1);
#pragma unroll
    for (int c = 0; c < 12; ++c) {
      const double2 r = csub(z[base + c * b], o[c]);
      float *h = (float *)(rhi + q + c * k.P) + (j & 1), *l = (float *)(rlo + q + c * k.P) + (j & 1);
      split_f64(r.x, ks, h[0], l[0]);
      split_f64(r.y, ks, h[2], l[2]);
      if (b == 1) h[1] = h[3] = l[1] = l[3] = 0.f;
      acc[0].x = fma(r.x, r.x, fma(r.y, r.y, acc[0].x));
    }
  }
  if (block_reduce<1>(acc, b, red.partial, red.counter, tot)) {
    if (j == (int)threadIdx.x) {
      fin_resid(sc, j, make_double2(tot[j].x, sc->bnorm2[j]), restart);
      set_fac(sc, j, hs);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      count_active(sc, b);
      if (mark) *mark = 0;
    }
  }
}

// --------------------------------------------------------------- launchers
// A solve that runs on its lane's share of the SMs keeps its other kernels there too, two blocks to an SM: blocks beyond
// that only queue behind the persistent kernels of the other lanes, which fill their SMs (8^4, 8 lanes of 19 CTAs).
static unsigned share(const EoSolve &S, unsigned g, int per_sm) {
  const unsigned most = (unsigned)((S.grid > 0 ? S.grid : device_sms()) * per_sm);
  return g < most ? g : most;
}
static unsigned item_grid(const EoSolve &S) {
  return share(S, reduce_grid((int64_t)S.g.V * (eo_width(S.b) / 2), device_sms()), 2);
}
static unsigned one_per_sm(const EoSolve &S) { return share(S, item_grid(S), 1); }

void eo_true_resid(const EoSolve &S, int restart, const int *run_flag, int run_if, cudaStream_t st) {
  const Blk k = blk_of(S);
  const double D = 4.0 + S.m0;
  const float dh = (float)D, dl = (float)(D - (double)dh);
  int *cert = &S.gs->fp64_cert, *mark = &S.gs->last_upd;
  k_eo_split<<<item_grid(S), kBlock, 0, st>>>(S.x, S.B.xhi, S.B.xlo, k, S.outer, S.red, cert, run_flag, run_if);
  k_eo_resid_df<<<one_per_sm(S), kBlock, 0, st>>>((const float4 *)S.gauge->Udf, S.B.xhi, S.B.xlo, S.z, S.B.rhi, S.B.rlo,
                                                  k, dh, dl, S.outer, S.red, restart, S.hs, run_flag, run_if, mark,
                                                  cert);
  k_eo_resid64<<<share(S, reduce_grid((int64_t)S.g.V * S.b, device_sms()), 2), kBlock, 0, st>>>(
      S.gauge->U64, S.x, S.z, S.B.rhi, S.B.rlo, k, log2i(S.b), D, S.outer, S.red, restart, S.hs, run_flag, run_if, mark,
      cert);
  count_launches(3);
}

void eo_first_resid(const EoSolve &S, int x_is_zero, cudaStream_t st) {
  const Blk k = blk_of(S);
  const int64_t n = (int64_t)S.g.V * 12 * S.b;
  const int *nz = x_is_zero ? nullptr : &S.gs->x_nonzero;
  k_eo_znorm<<<share(S, reduce_grid(n, device_sms()), 2), kBlock, 0, st>>>(S.z, n, S.b, S.outer, S.red, S.hs, sqrt(12.0 * S.g.V), nz);
  k_eo_split<<<item_grid(S), kBlock, 0, st>>>(S.z, S.B.rhi, S.B.rlo, k, S.outer, S.red, nullptr, nz, 0);
  count_launches(2);
  if (nz) eo_true_resid(S, 1, nz, 1, st);
}

template <typename T>
static int inner_t(const EoSolve &S, double inner_tol2, int maxiter, int grid, cudaStream_t st) {
  typedef typename Pair2<T>::T ST;
  const Blk k = blk_of(S);
  EoArgs<T> ea;
  ea.U = S.gauge->U32;
  ea.x = S.B.e;
  ea.r = (ST *)S.B.r; ea.rhat = (ST *)S.B.rhat; ea.p = (ST *)S.B.p; ea.v = (ST *)S.B.v; ea.t = (ST *)S.B.t;
  ea.w = (float4 *)S.B.w;
  ea.g = S.g; ea.b = 2 * k.P; ea.logp = k.logp;
  ea.diag = (float)(4.0 + S.m0);
  ea.wscale = (float)(0.5 / (4.0 + S.m0));
  ea.sc = S.inner; ea.partial = S.red.partial; ea.gs = S.gs;
  ea.max_iters = maxiter + 1;
  ea.grid = grid;
  k_eo_init<T><<<item_grid(S), kBlock, 0, st>>>(ea.U, S.B.rhi, ea.r, ea.rhat, ea.p, S.B.e, k, ea.wscale, S.outer,
                                                S.inner, inner_tol2, maxiter, S.red);
  count_launches(1);
  DTR_LAUNCH_CHECK("inner init");
  DTR_CUDA(cudaMemsetAsync(S.gs, 0, kGridSyncLaunchBytes, st));
  return launch_persistent_eo<T>(ea, st);
}

int eo_inner(const EoSolve &S, double inner_tol2, int maxiter, int store, int grid, cudaStream_t st, int *kernels) {
  *kernels = 2;
  if (store == 1) return inner_t<__half>(S, inner_tol2, maxiter, grid, st);
  if (store == 2) return inner_t<__nv_bfloat16>(S, inner_tol2, maxiter, grid, st);
  return inner_t<float>(S, inner_tol2, maxiter, grid, st);
}

void eo_accum(const EoSolve &S, int choose, cudaStream_t st) {
  k_eo_accum<<<item_grid(S), kBlock, 0, st>>>(S.gauge->U32, S.B.rhi, S.B.e, S.x, blk_of(S), (float)(1.0 / (4.0 + S.m0)),
                                              S.outer, S.inner, choose ? S.gs : nullptr);
  count_launches(1);
}

void eo_update(const EoSolve &S, cudaStream_t st) {
  const double D = 4.0 + S.m0;
  const float dh = (float)D;
  k_eo_update<<<item_grid(S), kBlock, 0, st>>>((const float4 *)S.gauge->Udf, S.B.e, S.B.rhi, S.B.rlo, blk_of(S), dh,
                                                (float)(D - (double)dh), S.outer, S.red, S.hs, &S.gs->sel, 1,
                                                &S.gs->last_upd);
  count_launches(1);
}

}  // namespace dtr
