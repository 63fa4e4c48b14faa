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
// What bounds it: at 32^3 x 64 the FP32 pipe and issue in A to D and HBM in E; at 8^4 the barriers and L2 round
// trips.  Two columns per thread in packed FP32x2 instructions.
#include <mutex>

#include "eo_core.cuh"
#include "grid_barrier.cuh"
#include "krylov_fin.cuh"
#include "persist_eo.cuh"

namespace dtr {

// Sums over the block of F values per column, each thread holding them for its two columns 2 jp, 2 jp + 1
// (jp = threadIdx.x & (b/2 - 1)): butterfly over the lanes of one column pair, then a fixed order over the warps;
// written to part[block * F b + q b + j].
template <int F, int T>
__device__ __forceinline__ void block_sums2(float2 (&v)[F], int b, float *__restrict__ part, float *shw) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, P = b >> 1;
  for (int off = 16; off >= P; off >>= 1) {
#pragma unroll
    for (int q = 0; q < F; ++q) {
      v[q].x += __shfl_xor_sync(0xffffffffu, v[q].x, off);
      v[q].y += __shfl_xor_sync(0xffffffffu, v[q].y, off);
    }
  }
  if (lane < P) {
#pragma unroll
    for (int q = 0; q < F; ++q) *(float2 *)&shw[(w * F + q) * b + 2 * lane] = v[q];
  }
  __syncthreads();
  const int n = F * b;
  for (int k = threadIdx.x; k < n; k += T) {
    float s[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int ww = 0; ww < T / 32; ww += 4)
#pragma unroll
      for (int u = 0; u < 4; ++u) s[u] += shw[(ww + u) * n + k];
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

// Work items [0, n) of one phase over the grid: full sweeps of the whole grid (neighbouring items run at the same
// time, so the stencil's neighbours meet in L2), and the remainder in whole warps spread evenly over the blocks
// (a last sweep of the first blocks alone would leave the other SMs idle: 8^4 x 16 on 19 blocks is 2.2 sweeps).
template <int T> struct Sweep {
  int64_t n, full, lo, hi;
  __device__ __forceinline__ explicit Sweep(int64_t n_) : n(n_) {
    const int64_t G = gridDim.x, round = G * T;
    full = n / round * round;
    const int64_t warps = (n - full + 31) / 32, ch = (warps + G - 1) / G * 32;
    lo = full + blockIdx.x * ch;
    hi = min(n, lo + ch);
  }
  template <class F> __device__ __forceinline__ void run(const F &body) const {
    for (int64_t it = (int64_t)blockIdx.x * T + threadIdx.x; it < full; it += (int64_t)gridDim.x * T) body(it);
    const int64_t it = lo + threadIdx.x;
    if (it < hi) body(it);
  }
};

template <typename S, int T> __global__ void __launch_bounds__(T, 1) k_bicgstab_eo(EoArgs<S> a) {
  typedef typename Pair2<S>::T ST;
  constexpr int kShw = T / 32 * 8 * 64 * 4, kSh = T * 16;
  __shared__ __align__(16) unsigned char smem[kShw > kSh ? kShw : kSh];
  __shared__ float tot[8 * 64];
  __shared__ Scal ss;  // this block's copy of the per-column scalars
  float *shw = (float *)smem;
  float4 *sh = (float4 *)smem;
  const int b = a.b, P = b >> 1, logp = a.logp;
  const int jp = threadIdx.x & (P - 1);
  const int64_t items = (int64_t)(a.g.V >> 1) << logp;
  const Sweep<T> sites(items), elems(items * 12);
  const unsigned int G = gridDim.x;
  float *part[2] = {(float *)a.partial, (float *)a.partial + (int64_t)8 * 64 * G};
  unsigned int nbar = 0, nred = 0;
  if (threadIdx.x == 0) {
    unsigned long long ns;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(ns));
    atomicMax(&a.gs->nt0, ~ns);
  }
  {
    const int *src = (const int *)a.sc;
    int *dst = (int *)&ss;
    for (int i = threadIdx.x; i < (int)(sizeof(Scal) / sizeof(int)); i += T) dst[i] = __ldcg(src + i);
  }
  __syncthreads();
  const float2 dg = f2(a.diag), mh = f2(-0.5f), ph = f2(0.5f);
  const float2 wp = f2(a.wscale), wm = f2(-a.wscale);
  const PairLoad<S> ldp{a.p, P, jp}, ldw{a.w, P, jp};

  for (int iter = 0; iter < a.max_iters; ++iter) {
    if (blockIdx.x == 0 && threadIdx.x == 0) a.gs->iters = iter + 1;
    sites.run([&](int64_t it) {  // A
      const EoSite s = eo_site(a.g, (int)(it >> logp), 1);
      c2 Su[2][3], Sl[2][3];
      hop_eo(a.U, ldp, a.g, s, Su, Sl);
      ST *w = a.w + (int64_t)s.h * 12 * P + jp;
#pragma unroll
      for (int k = 0; k < 6; ++k) {
        w[k * P] = Pair2<S>::narrow(scale2(Su[k / 3][k % 3], wp));
        w[(k + 6) * P] = Pair2<S>::narrow(scale2(Sl[k / 3][k % 3], wm));
      }
    });
    if (!grid_arrive_wait(a.gs, ++nbar * G, kSpinBudget)) break;
    {
      float2 d[2] = {f2(0.f), f2(0.f)};
      sites.run([&](int64_t it) {  // B
        const EoSite s = eo_site(a.g, (int)(it >> logp), 0);
        c2 Su[2][3], Sl[2][3];
        hop_eo(a.U, ldw, a.g, s, Su, Sl);
        const int64_t q = (int64_t)s.h * 12 * P + jp;
#pragma unroll
        for (int k = 0; k < 12; ++k) {
          const c2 p = Pair2<S>::widen(a.p[q + k * P]);
          const c2 hk = k < 6 ? Su[k / 3][k % 3] : Sl[(k - 6) / 3][k % 3];
          const float2 f = k < 6 ? mh : ph;
          const c2 v{__ffma2_rn(f, hk.re, __fmul2_rn(dg, p.re)), __ffma2_rn(f, hk.im, __fmul2_rn(dg, p.im))};
          a.v[q + k * P] = Pair2<S>::narrow(v);
          cdot2(d[0], d[1], Pair2<S>::widen(a.rhat[q + k * P]), v);
        }
      });
      float *pb = part[nred++ & 1];
      block_sums2<2, T>(d, b, pb, shw);
      if (!grid_arrive_wait(a.gs, ++nbar * G, kSpinBudget)) break;
      grid_sums2<T>(2 * b, pb, sh, tot);
      if (threadIdx.x < b) fin_alpha(&ss, threadIdx.x, make_double2(tot[threadIdx.x], tot[b + threadIdx.x]));
      __syncthreads();
    }
    const s2 mal = pair_of(ss.alpha, jp, -1.f);
    sites.run([&](int64_t it) {  // C
      const EoSite s = eo_site(a.g, (int)(it >> logp), 1);
      const PairAxpyLoad<S> ld{a.r, a.v, P, jp, mal};
      c2 Su[2][3], Sl[2][3];
      hop_eo(a.U, ld, a.g, s, Su, Sl);
      ST *w = a.w + (int64_t)s.h * 12 * P + jp;
#pragma unroll
      for (int k = 0; k < 6; ++k) {
        w[k * P] = Pair2<S>::narrow(scale2(Su[k / 3][k % 3], wp));
        w[(k + 6) * P] = Pair2<S>::narrow(scale2(Sl[k / 3][k % 3], wm));
      }
    });
    if (!grid_arrive_wait(a.gs, ++nbar * G, kSpinBudget)) break;
    int n_active = 0;
    {
      float2 d[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) d[k] = f2(0.f);
      sites.run([&](int64_t it) {  // D
        const EoSite st = eo_site(a.g, (int)(it >> logp), 0);
        c2 Su[2][3], Sl[2][3];
        hop_eo(a.U, ldw, a.g, st, Su, Sl);
        const int64_t q = (int64_t)st.h * 12 * P + jp;
#pragma unroll
        for (int k = 0; k < 12; ++k) {
          const c2 s = axpy2(mal, Pair2<S>::widen(a.v[q + k * P]), Pair2<S>::widen(a.r[q + k * P]));
          const c2 hk = k < 6 ? Su[k / 3][k % 3] : Sl[(k - 6) / 3][k % 3];
          const float2 f = k < 6 ? mh : ph;
          const c2 t{__ffma2_rn(f, hk.re, __fmul2_rn(dg, s.re)), __ffma2_rn(f, hk.im, __fmul2_rn(dg, s.im))};
          a.t[q + k * P] = Pair2<S>::narrow(t);
          const c2 rh = Pair2<S>::widen(a.rhat[q + k * P]);
          cdot2(d[0], d[1], t, s);    // t^H s
          norm2(d[2], t);             // t^H t
          cdot2(d[3], d[4], rh, s);   // rhat^H s
          cdot2(d[5], d[6], rh, t);   // rhat^H t
          norm2(d[7], s);             // s^H s
        }
      });
      float *pb = part[nred++ & 1];
      block_sums2<8, T>(d, b, pb, shw);
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
      const s2 al = pair_of(ss.alpha, jp, 1.f), om = pair_of(ss.omega, jp, 1.f);
      const s2 mom = pair_of(ss.omega, jp, -1.f), be = pair_of(ss.beta, jp, 1.f);
      const bool act0 = ss.active[2 * jp] != 0, act1 = ss.active[2 * jp + 1] != 0;
      const bool stop = n_active == 0;
      float4 *X = (float4 *)a.x;
      elems.run([&](int64_t q) {
        const c2 vv = Pair2<S>::widen(a.v[q]), pp = Pair2<S>::widen(a.p[q]);
        const c2 s = axpy2(mal, vv, Pair2<S>::widen(a.r[q]));
        const c2 tt = Pair2<S>::widen(a.t[q]);
        const float4 xo = X[q];
        const c2 x = axpy2(om, s, axpy2(al, pp, c2{make_float2(xo.x, xo.z), make_float2(xo.y, xo.w)}));
        X[q] = make_float4(x.re.x, x.im.x, x.re.y, x.im.y);
        if (!stop) {
          const c2 rn = axpy2(mom, tt, s);
          a.r[q] = Pair2<S>::narrow(rn);
          c2 pn = axpy2(be, axpy2(mom, vv, pp), rn);
          if (!act0) pn.re.x = pp.re.x, pn.im.x = pp.im.x;
          if (!act1) pn.re.y = pp.re.y, pn.im.y = pp.im.y;
          a.p[q] = Pair2<S>::narrow(pn);
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
  if (threadIdx.x == 0) {
    unsigned long long ns;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(ns));
    atomicMax(&a.gs->t1, ns);
  }
}

constexpr int kEoThreads = 384;

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
