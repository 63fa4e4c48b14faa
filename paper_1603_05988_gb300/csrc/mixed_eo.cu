// One defect-correction cycle of the mixed solvers on the red-black Schur complement (eo_core.cuh): the scaled
// residual, the inner problem on the even sites, and the correction on both sublattices afterwards.
#include "mixed_eo.cuh"

namespace dtr {

static size_t al(size_t x) { return (x + 255) / 256 * 256; }
static int log2i(int b) {
  int l = 0;
  while ((1 << l) < b) ++l;
  return l;
}

size_t eo_scratch_bytes(int64_t V, int b) {
  const size_t half = al((size_t)(V / 2) * 12 * eo_width(b) * sizeof(float2));
  return 10 * half;
}

EoBufs eo_carve(char *w, int64_t V, int b) {
  const size_t half = al((size_t)(V / 2) * 12 * eo_width(b) * sizeof(float2));
  EoBufs B;
  B.rf = (float2 *)w;
  B.e = (float2 *)(w + 2 * half);
  B.r = w + 4 * half;
  B.rhat = w + 5 * half;
  B.p = w + 6 * half;
  B.v = w + 7 * half;
  B.t = w + 8 * half;
  B.w = w + 9 * half;
  return B;
}

// body(h, valid) for the work items of all half-lattice sites, in whole warps (the stencil's lanes exchange values)
template <class F> __device__ __forceinline__ void for_eo_items(const Geom &g, int logp, const F &body) {
  const int64_t npair = (int64_t)(g.V >> 1) << logp;
  for (int64_t it = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; (it & ~(int64_t)31) < 2 * npair;
       it += (int64_t)gridDim.x * blockDim.x) {
    const int64_t pr = EoLane<4>::pair_of_item(it);
    body(pr < npair ? (int)(pr >> logp) : 0, pr < npair);
  }
}

// rf = hs * scale * r64 in red-black order (zero in inactive and padding columns)
__global__ void __launch_bounds__(kBlock) k_eo_scale(const double2 *__restrict__ r64, float2 *__restrict__ rf, Geom g,
                                                     int b, int logb, int64_t half, int bi,
                                                     const Scal *__restrict__ outer, double hs) {
  const int j = threadIdx.x & (b - 1);
  const double sc = outer->active[j] ? outer->scale[j] * hs : 0.0;
  const int64_t n = (int64_t)g.V * 12 << logb;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const double2 v = r64[i];
    const int k = (int)(i >> logb);
    const int s = k / 12, c = k - 12 * s;
    float2 *q = rf + (site_parity(g, s) ? half : 0) + ((int64_t)(s >> 1) * 12 + c) * bi + j;
    q[0] = make_float2((float)(v.x * sc), (float)(v.y * sc));
    if (bi > b) q[1] = make_float2(0.f, 0.f);
  }
}

// r = rhat = p = rf_e + H rf_o / (2 D), e = 0 on the even sites; the inner scalars, with rho = |r|^2 and the norm
// that the tolerance refers to that of the whole residual (hs2)
template <typename S>
__global__ void __launch_bounds__(kBlock) k_eo_init(const float2 *__restrict__ U, const float2 *__restrict__ rf,
                                                    int64_t half, typename Pair2<S>::T *__restrict__ r,
                                                    typename Pair2<S>::T *__restrict__ rhat,
                                                    typename Pair2<S>::T *__restrict__ p, float2 *__restrict__ e,
                                                    Geom g, int b, int P, int logp, float wscale,
                                                    const Scal *__restrict__ outer, Scal *inner, double tol2,
                                                    int maxiter, double hs2, Reduce red) {
  __shared__ double2 tot[2 * 64];
  const EoLane<4> ln(2 * P, threadIdx.x);
  const CplxLoad odd{rf + half}, even{rf};
  const float2 wp = f2(wscale), wm = f2(-wscale);
  float2 nrm = f2(0.f);
  double2 acc[2] = {make_double2(0.0, 0.0), make_double2(0.0, 0.0)};
  for_eo_items(g, logp, [&](int h, bool valid) {
    const EoSite s = eo_site(g, h, 0);
    c2 H[2][3], own[2][3];
    hop_eo<0>(ln, U, odd, g, s, H[0], H[1]);
    even.get(ln, h, ln.clz, own[0], own[1]);
    if (!valid) return;
    const int64_t q = (int64_t)h * 12 * P + ln.jp;
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      const c2 hk = H[k / 3][k % 3], o = own[k / 3][k % 3];
      const float2 f = k < 3 ? wp : wm;
      const int64_t i = q + (k < 3 ? ln.cu : ln.clz) + (k % 3) * P;
      const typename Pair2<S>::T st = Pair2<S>::narrow(c2{__ffma2_rn(f, hk.re, o.re), __ffma2_rn(f, hk.im, o.im)});
      r[i] = st;
      rhat[i] = st;
      p[i] = st;
      ((float4 *)e)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
      const c2 w = Pair2<S>::widen(st);
      nrm = __ffma2_rn(w.re, w.re, __ffma2_rn(w.im, w.im, nrm));
    }
  });
  acc[0].x = (double)nrm.x;
  acc[1].x = (double)nrm.y;
  // a thread's column pair is threadIdx.x & (P - 1) up to P = 16; with P = 32 the row bit sits in between
  const int w = P <= 16 ? P : 64;
  if (block_reduce<2>(acc, w, red.partial, red.counter, tot)) {
    const int j = threadIdx.x;
    if (j < 2 * P) {
      const int jp = j >> 1, q = (j & 1) * w;
      const double rho = P <= 16 ? tot[q + jp].x : tot[q + (jp & 15) + 2 * (jp & 16)].x + tot[q + (jp & 15) + 2 * (jp & 16) + 16].x;
      const int act = j < b ? outer->active[j] : 0;
      inner->active[j] = act;
      inner->rho[j] = make_double2(rho, 0.0);
      inner->bnorm2[j] = hs2;
      inner->rnorm2[j] = rho;
      inner->iters[j] = 0;
      inner->flags[j] = 0;
      inner->alpha[j] = inner->omega[j] = inner->beta[j] = make_double2(0.0, 0.0);
      if (j == 0) {
        int n = 0;
        for (int q = 0; q < b; ++q) n += outer->active[q];
        inner->n_active = n;
        inner->tol2 = tol2;
        inner->maxiter = maxiter;
      }
    }
  }
}

// e_o = (rf_o + H e_e / 2) / D, x64 += e / (hs * scale) on both sublattices (one thread per site pair 2h, 2h + 1 and
// column pair); counters and the choice of the next residual as in k_mixed_accum
__global__ void __launch_bounds__(kBlock) k_eo_accum(const float2 *__restrict__ U, const float2 *__restrict__ rf,
                                                     float2 *e, int64_t half, double2 *__restrict__ x, Geom g, int b,
                                                     int P, int logp, float dinv, Scal *outer,
                                                     const Scal *__restrict__ inner, double hs, GridSync *gs,
                                                     int allow_update) {
  if (gs && blockIdx.x == 0) {  // one column per thread of block 0
    const int q = threadIdx.x;
    int far = 0;
    if (q < b && outer->active[q]) {
      const double red2 = inner->bnorm2[q] > 0.0 ? inner->rnorm2[q] / inner->bnorm2[q] : 1.0;
      far = outer->rtrue2[q] * red2 > 100.0 * outer->tol2 * outer->bnorm2[q];
    }
    far = __syncthreads_or(far);
    if (q == 0) gs->sel = (allow_update && far) ? 1 : 0;
  }
  const EoLane<4> ln(2 * P, threadIdx.x);
  const CplxLoad even{e}, res{rf + half};
  const bool a0 = outer->active[2 * ln.jp] != 0, a1 = b > 1 && outer->active[2 * ln.jp + 1] != 0;
  const double inv0 = a0 ? 1.0 / (outer->scale[2 * ln.jp] * hs) : 0.0;
  const double inv1 = a1 ? 1.0 / (outer->scale[2 * ln.jp + 1] * hs) : 0.0;
  const float2 di = f2(dinv), dh = f2(0.5f * dinv), dmh = f2(-0.5f * dinv);
  for_eo_items(g, logp, [&](int h, bool valid) {
    const EoSite s = eo_site(g, h, 1);
    c2 H[2][3], eo[2][3], ee[2][3];
    hop_eo<0>(ln, U, even, g, s, H[0], H[1]);
    res.get(ln, h, ln.clz, eo[0], eo[1]);
    even.get(ln, h, ln.clz, ee[0], ee[1]);
    if (!valid) return;
    const int64_t q = (int64_t)h * 12 * P + ln.jp;
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      const c2 hk = H[k / 3][k % 3];
      c2 &o = eo[k / 3][k % 3];
      const float2 f = k < 3 ? dh : dmh;
      o = c2{__ffma2_rn(f, hk.re, __fmul2_rn(di, o.re)), __ffma2_rn(f, hk.im, __fmul2_rn(di, o.im))};
      ((float4 *)(e + half))[q + (k < 3 ? ln.cu : ln.clz) + (k % 3) * P] = to_cols(o);
    }
    if (!a0 && !a1) return;
    const int lex = eo_lex(s);
#pragma unroll
    for (int side = 0; side < 2; ++side) {  // the odd site, then the even one of the pair 2h, 2h + 1
      double2 *xs = x + (int64_t)(side ? lex ^ 1 : lex) * 12 * b + 2 * ln.jp;
      double2 v[6][2];
#pragma unroll
      for (int k = 0; k < 6; ++k) {
        const double2 *xp = xs + ((k < 3 ? 0 : 6) + 3 * ln.r + k % 3) * b;
        v[k][0] = xp[0];
        if (b > 1) v[k][1] = xp[1];
      }
#pragma unroll
      for (int k = 0; k < 6; ++k) {
        const c2 d = side ? ee[k / 3][k % 3] : eo[k / 3][k % 3];
        double2 *xp = xs + ((k < 3 ? 0 : 6) + 3 * ln.r + k % 3) * b;
        xp[0] = make_double2(fma((double)d.re.x, inv0, v[k][0].x), fma((double)d.im.x, inv0, v[k][0].y));
        if (b > 1) xp[1] = make_double2(fma((double)d.re.y, inv1, v[k][1].x), fma((double)d.im.y, inv1, v[k][1].y));
      }
    }
  });
  if (blockIdx.x == 0 && threadIdx.x < b) {
    outer->iters[threadIdx.x] += inner->iters[threadIdx.x];
    outer->flags[threadIdx.x] |= inner->flags[threadIdx.x] & ~kFlagBreakdown;
  }
}

template <typename S>
static int inner_t(const dtr_gauge_s *gauge, const EoBufs &B, const Geom &g, int b, double m0, const Scal *outer,
                   Scal *inner, const Reduce &red, GridSync *gs, double inner_tol2, int maxiter, double hs, int grid,
                   cudaStream_t st) {
  typedef typename Pair2<S>::T ST;
  const int bi = eo_width(b), P = bi / 2;
  const int64_t half = (int64_t)(g.V / 2) * 12 * bi;
  EoArgs<S> ea;
  ea.U = gauge->U32;
  ea.x = B.e;
  ea.r = (ST *)B.r; ea.rhat = (ST *)B.rhat; ea.p = (ST *)B.p; ea.v = (ST *)B.v; ea.t = (ST *)B.t; ea.w = (float4 *)B.w;
  ea.g = g; ea.b = bi; ea.logp = log2i(P);
  ea.diag = (float)(4.0 + m0);
  ea.wscale = (float)(0.5 / (4.0 + m0));
  ea.sc = inner; ea.partial = red.partial; ea.gs = gs;
  ea.max_iters = maxiter + 1;
  ea.grid = grid;
  k_eo_init<S><<<reduce_grid((int64_t)g.V * P, device_sms()), kBlock, 0, st>>>(
      gauge->U32, B.rf, half, ea.r, ea.rhat, ea.p, B.e, g, b, P, ea.logp, ea.wscale, outer, inner, inner_tol2, maxiter,
      hs * hs, red);
  count_launches(1);
  DTR_LAUNCH_CHECK("inner init");
  DTR_CUDA(cudaMemsetAsync(gs, 0, kGridSyncLaunchBytes, st));
  return launch_persistent_eo<S>(ea, st);
}

int eo_inner(const dtr_gauge_s *gauge, const EoBufs &B, const Geom &g, int b, double m0, const double2 *r64,
             const Scal *outer, Scal *inner, const Reduce &red, GridSync *gs, double inner_tol2, int maxiter,
             double hs, int store, int grid, cudaStream_t st, int *kernels) {
  const int bi = eo_width(b);
  const int64_t n = (int64_t)g.V * 12 * b;
  k_eo_scale<<<reduce_grid(n, device_sms()), kBlock, 0, st>>>(r64, B.rf, g, b, log2i(b),
                                                              (int64_t)(g.V / 2) * 12 * bi, bi, outer, hs);
  count_launches(1);
  *kernels = 3;
  if (store == 1)
    return inner_t<__half>(gauge, B, g, b, m0, outer, inner, red, gs, inner_tol2, maxiter, hs, grid, st);
  if (store == 2)
    return inner_t<__nv_bfloat16>(gauge, B, g, b, m0, outer, inner, red, gs, inner_tol2, maxiter, hs, grid, st);
  return inner_t<float>(gauge, B, g, b, m0, outer, inner, red, gs, inner_tol2, maxiter, hs, grid, st);
}

void eo_accum(const dtr_gauge_s *gauge, const EoBufs &B, const Geom &g, int b, double m0, double2 *x, Scal *outer,
              const Scal *inner, double hs, GridSync *gs, int allow_update, cudaStream_t st) {
  const int bi = eo_width(b), P = bi / 2;
  k_eo_accum<<<reduce_grid((int64_t)g.V * P, device_sms()), kBlock, 0, st>>>(
      gauge->U32, B.rf, B.e, (int64_t)(g.V / 2) * 12 * bi, x, g, b, P, log2i(P), (float)(1.0 / (4.0 + m0)), outer,
      inner, hs, gs, allow_update);
  count_launches(1);
}

}  // namespace dtr
