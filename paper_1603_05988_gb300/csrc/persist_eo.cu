// Persistent batched BiCGStab on the red-black Schur complement (eo_core.cuh): the inner solve of the mixed
// solvers for one block of right-hand sides in ONE cooperative launch.
//
// Per iteration, five phases separated by grid barriers (all vectors on the even sites but w):
//   A  w = H_oe p / (2 D)                              on the odd sites
//   B  v = D p - H_eo w / 2        rhat^H v            -> alpha
//   C  w = H_oe s / (2 D)          s = r - alpha v, formed at the neighbours
//   D  t = D s - H_eo w / 2        t^H s, t^H t, rhat^H s, rhat^H t, s^H s -> omega, beta, convergence
//   E  x += alpha p + omega s, r = s - omega t, p = r + beta (p - omega v)
// The reductions are all-reduce barriers, as in persist.cu: per-block partials, and every block sums all partials in
// one fixed order and runs the scalar algebra on its own copy of the column scalars.
//
// What bounds it (GB300, us per phase of one iteration): 32^3 x 64 x 16, FP16 storage: A 1060, B 1337, C 1600, D 1506
// (FP32 pipe 72% and load pipe 67% busy; the hops' HBM floor is 330), E 1112 (7.2 TB/s), barriers 25 to 130 each;
// 16^3 x 32 x 32, FP32: A 140, B 181, C 187, D 201, E 194.  One thread per site and column pair instead of two took
// 1057, 1930, 1820, 2110, 1258 and 124, 261, 196, 289, 218 (its loads after a store, in B and D, waited one by one).
// 8^4 x 16: A 3.3, B 4.3, C 5.1, D 5.7, E 2.9, barriers 1.6 to 5.3: latency.
#include <type_traits>

#include "eo_core.cuh"
#include "grid_barrier.cuh"
#include "krylov_fin.cuh"
#include "persist_eo.cuh"

namespace dtr {

// Sums over the block of F values per column, each thread holding them for the column pair and spin row of its
// EoLane: butterfly over the lanes of one column pair, then a fixed order over the warps; written to
// part[block * F b + q b + j].
template <class LN, int F, int T>
__device__ __forceinline__ void block_sums2(float2 (&v)[F], int b, float *__restrict__ part, float *shw) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int bw = b < 32 ? b : 32;   // columns that one warp holds
#pragma unroll
  for (int q = 0; q < F; ++q) {
    const float2 o = LN::other_row(v[q]);
    v[q].x += o.x;
    v[q].y += o.y;
  }
  // lanes of one pair are b / 2 items apart, an item being 2 lanes (row bit 0) or 1 (row bit 4) wide
  constexpr int kItem = LN::pair_of_item(2) == 1 ? 2 : 1;
  for (int off = 8; 2 * off >= b; off >>= 1) {
#pragma unroll
    for (int q = 0; q < F; ++q) {
      v[q].x += __shfl_xor_sync(0xffffffffu, v[q].x, off * kItem);
      v[q].y += __shfl_xor_sync(0xffffffffu, v[q].y, off * kItem);
    }
  }
  const int col = 2 * (lane / kItem);
  if (col < bw && lane % kItem == 0) {
#pragma unroll
    for (int q = 0; q < F; ++q) *(float2 *)&shw[(w * F + q) * bw + col] = v[q];
  }
  __syncthreads();
  const int n = F * b, cw = b > 32 ? 2 : 1;  // warps that share a set of columns
  for (int k = threadIdx.x; k < n; k += T) {
    const int q = k / b, j = k & (b - 1);
    const float *src = shw + q * bw + (j & (bw - 1));
    float s[4] = {0.f, 0.f, 0.f, 0.f};
    for (int ww = j >> 5; ww < T / 32; ww += 4 * cw)
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (ww + u * cw < T / 32) s[u] += src[(ww + u * cw) * F * bw];
    part[(int64_t)blockIdx.x * n + k] = (s[0] + s[1]) + (s[2] + s[3]);
  }
}

// tot[k] = sum over blocks of part[block * n + k], k < n = F b, in one fixed order (slices of contiguous blocks,
// four values per load).
template <int T> __device__ __forceinline__ void grid_sums2(int n, const float *__restrict__ part, float4 *sh,
                                                            float *tot) {
  const int t = threadIdx.x, G = gridDim.x, Q = n >> 2;
  int S = T / Q;
  if (S > 16) S = 16;
  const int ch = (G + S - 1) / S;
  const int q = t % Q, sl = t / Q;
  __syncthreads();  // the partial sums above have read sh's memory
  if (sl < S) {
    const int lo = sl * ch, hi = min(G, lo + ch);
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
    const float4 *src = (const float4 *)part + q;
    for (int k0 = lo; k0 < hi; k0 += 8) {
      float4 v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u)
        v[u] = k0 + u < hi ? __ldcg(src + (int64_t)(k0 + u) * Q) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        a.x += v[u].x;
        a.y += v[u].y;
        a.z += v[u].z;
        a.w += v[u].w;
      }
    }
    sh[sl * Q + q] = a;
  }
  __syncthreads();
  for (int k = t; k < n; k += T) {
    float s = ((const float *)sh)[k];
    for (int u = 1; u < S; ++u) s += ((const float *)sh)[u * n + k];
    tot[k] = s;
  }
  __syncthreads();
}

// column pair scalars as packed operands
__device__ __forceinline__ s2 pair_of(const double2 *v, int jp, float sign) {
  const double2 a = v[2 * jp], c = v[2 * jp + 1];
  s2 s;
  s.re = make_float2(sign * (float)a.x, sign * (float)c.x);
  s.im = make_float2(sign * (float)a.y, sign * (float)c.y);
  s.nim = make_float2(-s.im.x, -s.im.y);
  return s;
}
// acc (re, im) += conj(a) b
__device__ __forceinline__ void cdot2(float2 &re, float2 &im, c2 a, c2 b) {
  re = __ffma2_rn(a.re, b.re, __ffma2_rn(a.im, b.im, re));
  im = __ffma2_rn(a.re, b.im, im);
  im = sub2(im, __fmul2_rn(a.im, b.re));
}
__device__ __forceinline__ void norm2(float2 &s, c2 a) { s = __ffma2_rn(a.re, a.re, __ffma2_rn(a.im, a.im, s)); }

template <typename S, int T> __global__ void __launch_bounds__(T, 1) k_bicgstab_eo(EoArgs<S> a) {
  typedef typename Pair2<S>::T ST;
  typedef Pair2<S> PS;
  // components loaded before the first is used (a store in between would order the loads one by one)
  constexpr int NB = sizeof(ST) == 8 ? 6 : 3;
  constexpr int kShw = T / 32 * 8 * 32 * 4, kSh = T * 16;
  __shared__ __align__(16) unsigned char smem[kShw > kSh ? kShw : kSh];
  __shared__ float tot[8 * 64];
  __shared__ Scal ss;  // this block's copy of the per-column scalars
  float *shw = (float *)smem;
  float4 *sh = (float4 *)smem;
  const int b = a.b;
  typedef EoLane<row_bit<S>()> LA;   // lanes of the phases that gather Krylov vectors
  typedef EoLane<row_bit<float>()> LN;  // and of those that gather w
  const LN ln(b, threadIdx.x);
  const int P = ln.P, jp = ln.jp;
  const int64_t nh = a.g.V >> 1;
  const int64_t npair = nh << a.logp, nel = npair * 12;
  const Sweep<T, 64> pairs(2 * npair), elems(nel);  // two threads (spin rows) for a site and column pair
  const unsigned int G = gridDim.x;
  float *part[2] = {(float *)a.partial, (float *)a.partial + (int64_t)8 * 64 * G};
  unsigned int nbar = 0, nred = 0;
  if (threadIdx.x == 0) atomicMax(&a.gs->nt0, ~global_ns());
  {
    const int *src = (const int *)a.sc;
    int *dst = (int *)&ss;
    for (int i = threadIdx.x; i < (int)(sizeof(Scal) / sizeof(int)); i += T) dst[i] = __ldcg(src + i);
  }
  __syncthreads();
  const float2 dg = f2(a.diag), mh = f2(-0.5f), ph = f2(0.5f);
  const float2 wp = f2(a.wscale), wm = f2(-a.wscale);
  const PairLoad<S> ldp{a.p};
  const PairLoad<float> ldw{a.w};
  // offset of this thread's component k (upper spin 0..2, lower spin 3..5) from its site
  const int own[6] = {ln.cu, ln.cu + P, ln.cu + 2 * P, ln.clz, ln.clz + P, ln.clz + 2 * P};
  // w at an odd site from the hops of the loader's field
  auto odd_phase = [&](const auto &ld, const LA &la, auto ahead) {
    pairs.run([&](int64_t it) {
      const int64_t pr = LA::pair_of_item(it);
      const bool valid = pr < npair;
      const EoSite s = eo_site(a.g, valid ? (int)(pr >> a.logp) : 0, 1);
      c2 Su[3], Sl[3];
      hop_eo<decltype(ahead)::value>(la, a.U, ld, a.g, s, Su, Sl);
      float4 *w = a.w + (int64_t)s.h * 12 * P + la.jp;
      if (valid) {
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          w[la.cu + k * P] = Pair2<float>::narrow(scale2(Su[k], wp));
          w[la.clz + k * P] = Pair2<float>::narrow(scale2(Sl[k], wm));
        }
      }
    });
  };

  for (int iter = 0; iter < a.max_iters; ++iter) {
    if (blockIdx.x == 0 && threadIdx.x == 0) a.gs->iters = iter + 1;
    odd_phase(ldp, LA(b, threadIdx.x), std::integral_constant<int, 0>());  // A
    if (!grid_arrive_wait(a.gs, ++nbar * G, kSpinBudget)) break;
    {
      float2 d[2] = {f2(0.f), f2(0.f)};
      pairs.run([&](int64_t it) {  // B
        const int64_t pr = LN::pair_of_item(it);
        const bool valid = pr < npair;
        const EoSite s = eo_site(a.g, valid ? (int)(pr >> a.logp) : 0, 0);
        c2 Su[3], Sl[3];
        hop_eo<0>(ln, a.U, ldw, a.g, s, Su, Sl);
        const int64_t q = (int64_t)s.h * 12 * P + jp;
        if (valid) {
#pragma unroll
          for (int k0 = 0; k0 < 6; k0 += NB) {
            ST pr[NB], hr[NB];
#pragma unroll
            for (int k = 0; k < NB; ++k) {
              pr[k] = a.p[q + own[k0 + k]];
              hr[k] = a.rhat[q + own[k0 + k]];
            }
#pragma unroll
            for (int k = 0; k < NB; ++k) {
              const int c = k0 + k;
              const c2 p = PS::widen(pr[k]), hk = c < 3 ? Su[c] : Sl[c - 3];
              const float2 f = c < 3 ? mh : ph;
              const c2 v{__ffma2_rn(f, hk.re, __fmul2_rn(dg, p.re)), __ffma2_rn(f, hk.im, __fmul2_rn(dg, p.im))};
              a.v[q + own[c]] = PS::narrow(v);
              cdot2(d[0], d[1], PS::widen(hr[k]), v);
            }
          }
        }
      });
      float *pb = part[nred++ & 1];
      block_sums2<LN, 2, T>(d, b, pb, shw);
      if (!grid_arrive_wait(a.gs, ++nbar * G, kSpinBudget)) break;
      grid_sums2<T>(2 * b, pb, sh, tot);
      if (threadIdx.x < b) fin_alpha(&ss, threadIdx.x, make_double2(tot[threadIdx.x], tot[b + threadIdx.x]));
      __syncthreads();
    }
    {
      const LA la(b, threadIdx.x);
      const PairAxpyLoad<S> ld{a.r, a.v, pair_of(ss.alpha, la.jp, -1.f)};
      // the one phase with two fields to load a hop ahead; FP32 storage has no registers left for it (spills of 1 KB:
      // 262 instead of 187 us at 16^3 x 32 x 32), FP16 gains (1691 -> 1602 us at 32^3 x 64 x 16)
      odd_phase(ld, la, std::integral_constant<int, sizeof(ST) == 8 ? 1 : 0>());  // C
    }
    if (!grid_arrive_wait(a.gs, ++nbar * G, kSpinBudget)) break;
    int n_active = 0;
    {
      const s2 mal = pair_of(ss.alpha, jp, -1.f);
      float2 d[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) d[k] = f2(0.f);
      pairs.run([&](int64_t it) {  // D
        const int64_t pr = LN::pair_of_item(it);
        const bool valid = pr < npair;
        const EoSite st = eo_site(a.g, valid ? (int)(pr >> a.logp) : 0, 0);
        c2 Su[3], Sl[3];
        hop_eo<0>(ln, a.U, ldw, a.g, st, Su, Sl);
        const int64_t q = (int64_t)st.h * 12 * P + jp;
        if (valid) {
#pragma unroll
          for (int k0 = 0; k0 < 6; k0 += NB) {
            ST rr[NB], vr[NB], hr[NB];
#pragma unroll
            for (int k = 0; k < NB; ++k) {
              rr[k] = a.r[q + own[k0 + k]];
              vr[k] = a.v[q + own[k0 + k]];
              hr[k] = a.rhat[q + own[k0 + k]];
            }
#pragma unroll
            for (int k = 0; k < NB; ++k) {
              const int c = k0 + k;
              const c2 s = axpy2(mal, PS::widen(vr[k]), PS::widen(rr[k]));
              const c2 hk = c < 3 ? Su[c] : Sl[c - 3];
              const float2 f = c < 3 ? mh : ph;
              const c2 t{__ffma2_rn(f, hk.re, __fmul2_rn(dg, s.re)), __ffma2_rn(f, hk.im, __fmul2_rn(dg, s.im))};
              a.t[q + own[c]] = PS::narrow(t);
              const c2 rh = PS::widen(hr[k]);
              cdot2(d[0], d[1], t, s);    // t^H s
              norm2(d[2], t);             // t^H t
              cdot2(d[3], d[4], rh, s);   // rhat^H s
              cdot2(d[5], d[6], rh, t);   // rhat^H t
              norm2(d[7], s);             // s^H s
            }
          }
        }
      });
      float *pb = part[nred++ & 1];
      block_sums2<LN, 8, T>(d, b, pb, shw);
      if (!grid_arrive_wait(a.gs, ++nbar * G, kSpinBudget)) break;
      grid_sums2<T>(8 * b, pb, sh, tot);
      if (threadIdx.x < b) {
        const float *x = tot + threadIdx.x;
        fin_omega_beta(&ss, threadIdx.x, make_double2(x[0], x[b]), make_double2(x[2 * b], 0.0),
                       make_double2(x[3 * b], x[4 * b]), make_double2(x[5 * b], x[6 * b]),
                       make_double2(x[7 * b], 0.0));
      }
      n_active = __syncthreads_count(threadIdx.x < b && ss.active[threadIdx.x]);
      if (threadIdx.x == 0) ss.n_active = n_active;
    }
    {  // E
      const int je = threadIdx.x & (P - 1);  // column pair of this thread's elements
      const s2 al = pair_of(ss.alpha, je, 1.f), om = pair_of(ss.omega, je, 1.f), be = pair_of(ss.beta, je, 1.f);
      const s2 mal = pair_of(ss.alpha, je, -1.f), mom = pair_of(ss.omega, je, -1.f);
      const bool act0 = ss.active[2 * je] != 0, act1 = ss.active[2 * je + 1] != 0;
      const bool stop = n_active == 0;
      elems.run([&](int64_t q) {
        if (q >= nel) return;
        const c2 vv = PS::widen(a.v[q]), pp = PS::widen(a.p[q]);
        const c2 s = axpy2(mal, vv, PS::widen(a.r[q]));
        const c2 tt = PS::widen(a.t[q]);
        a.x[q] = Pair2<float>::narrow(axpy2(om, s, axpy2(al, pp, Pair2<float>::widen(a.x[q]))));
        if (!stop) {
          const c2 rn = axpy2(mom, tt, s);
          a.r[q] = PS::narrow(rn);
          c2 pn = axpy2(be, axpy2(mom, vv, pp), rn);
          if (!act0) pn.re.x = pp.re.x, pn.im.x = pp.im.x;
          if (!act1) pn.re.y = pp.re.y, pn.im.y = pp.im.y;
          a.p[q] = PS::narrow(pn);
        }
      });
      if (stop) break;  // kernel exit orders x for the next kernel
      if (!grid_arrive_wait(a.gs, ++nbar * G, kSpinBudget)) break;  // p is read at neighbours next
    }
  }
  // block 0 publishes the per-column scalars (identical in every block)
  __syncthreads();
  if (blockIdx.x == 0) {
    const int *src = (const int *)&ss;
    int *dst = (int *)a.sc;
    for (int i = threadIdx.x; i < (int)(sizeof(Scal) / sizeof(int)); i += T) dst[i] = src[i];
  }
  if (threadIdx.x == 0) atomicMax(&a.gs->t1, global_ns());
}

constexpr int kEoThreads = 512;

template <typename S> int launch_persistent_eo(const EoArgs<S> &ea, cudaStream_t st) {
  static int max_grid = 0;
  auto *kern = k_bicgstab_eo<S, kEoThreads>;
  if (!max_grid) {
    int nb = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kern, kEoThreads, 0);
    if (e != cudaSuccess) return cuda_fail(e, "persistent solver occupancy");
    if (nb < 1) return fail(DTR_ECUDA, "persistent solver cannot be resident");
    max_grid = nb * device_sms();
    if (max_grid > kPersistMaxGrid) max_grid = kPersistMaxGrid;
  }
  const int grid = (ea.grid > 0 && ea.grid < max_grid) ? ea.grid : max_grid;
  EoArgs<S> copy = ea;
  void *args[] = {&copy};
  DTR_CUDA(cudaLaunchCooperativeKernel((const void *)kern, dim3(grid), dim3(kEoThreads), args, 0, st));
  count_launches(1);
  if (persist_profile().on) return persist_account(ea.gs, (double)ea.g.V * ea.b, st);
  return DTR_OK;
}
template int launch_persistent_eo<float>(const EoArgs<float> &, cudaStream_t);
template int launch_persistent_eo<__half>(const EoArgs<__half> &, cudaStream_t);
template int launch_persistent_eo<__nv_bfloat16>(const EoArgs<__nv_bfloat16> &, cudaStream_t);

}  // namespace dtr
