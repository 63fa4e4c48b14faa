// Plain FP64 BiCGStab of a block of right-hand sides on the red-black Schur complement (eo_core.cuh), in ONE
// cooperative launch with true-residual restarts.
//
// A cycle: the true residual r = z - A x on the whole lattice and the restart decision; the Schur problem
// r_e + H r_o / (2 D) on the even sites; iterations of
//   A  w = H_oe p / (4 D)                on the odd sites
//   B  v = D p - H_eo w    rhat^H v      -> alpha
//   S  r <- s = r - alpha v
//   C  w = H_oe s / (4 D)
//   D  t = D s - H_eo w    t^H s, t^H t, rhat^H s, rhat^H t, s^H s -> omega, beta, convergence
//   E  x += alpha p + omega s, r = s - omega t, p = r + beta (p - omega v)
// until the Schur residual, which is the residual of the whole system, meets tol; x_o = (z_o + H x_e / 2) / D.
//
// What bounds it: the FP64 pipe, two lanes per clock and SM, so the steps count FP64 instructions and not bytes: s is
// stored (forming it at eight neighbours costs as much as a hop), every product is fused (the whole-lattice stencil
// adds the three products of a U^H row unfused), the factors 1/2 sit in w.  Per iteration and site 1176 FP64
// instructions against 2976 on the whole lattice, and half the iterations.
#include "eo_core.cuh"
#include "grid_barrier.cuh"
#include "krylov_fin.cuh"
#include "persist_eo.cuh"

namespace dtr {

typedef EoLane<4> L64;  // one column per thread: P = b columns, jp the column

// a + conj(m) b
__device__ __forceinline__ double2 cjaxpy(double2 m, double2 b, double2 a) {
  return make_double2(fma(m.x, b.x, fma(m.y, b.y, a.x)), fma(m.x, b.y, fma(-m.y, b.x, a.y)));
}
__device__ __forceinline__ double2 adds(double2 u, double2 l, double s) {
  return make_double2(fma(s, l.x, u.x), fma(s, l.y, u.y));
}
__device__ __forceinline__ double2 addi(double2 u, double2 l, double s) {
  return make_double2(fma(-s, l.y, u.x), fma(s, l.x, u.y));
}

// loaders: element 0 of column j at the neighbour with half-lattice index h and x & 1 == o
struct HalfLoad64 {  // [h][12][b]
  const double2 *f;
  __device__ __forceinline__ const double2 *at(const L64 &ln, int h, int) const {
    return f + (int64_t)h * 12 * ln.P + ln.jp;
  }
};
struct LexLoad64 {  // [site][12][b]
  const double2 *f;
  __device__ __forceinline__ const double2 *at(const L64 &ln, int h, int o) const {
    return f + (int64_t)(2 * h + o) * 12 * ln.P + ln.jp;
  }
};

template <int MU, bool FWD>
__device__ __forceinline__ void hop64_dir(const L64 &ln, const double2 *__restrict__ U, const double2 *f, double sg,
                                          double2 (&Su)[3], double2 (&L)[3]) {
  const int cl = MU < 2 ? ln.clx : ln.clz;
  double2 h[3], l[3], m[9];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    h[k] = f[ln.cu + k * ln.P];
    l[k] = f[cl + k * ln.P];
  }
#pragma unroll
  for (int k = 0; k < 9; ++k) m[k] = __ldg(U + k);
  const double s = (MU == 0 ? 1.0 : MU == 3 ? -1.0 : sg) * (FWD ? 1.0 : -1.0);
#pragma unroll
  for (int a = 0; a < 3; ++a) h[a] = (MU == 0 || MU == 2) ? addi(h[a], l[a], s) : adds(h[a], l[a], s);
  // factor of w in L: i, -sg, i sg, 1 for x, y, z, t, negated backward
  const double t = (MU == 0 || MU == 3 ? 1.0 : MU == 1 ? -sg : sg) * (FWD ? 1.0 : -1.0);
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    double2 w;
    if (FWD) {
      w = cmul(m[3 * a], h[0]);
      w = caxpy(m[3 * a + 1], h[1], w);
      w = caxpy(m[3 * a + 2], h[2], w);
    } else {
      w = cjmul(m[a], h[0]);
      w = cjaxpy(m[3 + a], h[1], w);
      w = cjaxpy(m[6 + a], h[2], w);
    }
    Su[a] = cadd(Su[a], w);
    L[a] = (MU == 0 || MU == 2) ? addi(L[a], w, t) : adds(L[a], w, t);
  }
}

// this row of (H psi)(s): upper spin Su, and Sl, minus the lower spin (all lanes of a warp take part)
template <class LD>
__device__ __forceinline__ void hop64(const L64 &ln, const double2 *__restrict__ U, const LD &in, const Geom &g,
                                      const EoSite &s, double2 (&Su)[3], double2 (&Sl)[3]) {
#pragma unroll
  for (int a = 0; a < 3; ++a) Su[a] = Sl[a] = make_double2(0.0, 0.0);
  const int hx = g.L[0] >> 1, odd = s.x & 1, h = s.h;
  const double sg = ln.r ? -1.0 : 1.0;
  const double2 *Us = U + (int64_t)eo_lex(s) * 36;
  {
    const int hf = odd ? (s.x == g.L[0] - 1 ? h - (hx - 1) : h + 1) : h;
    const int hb = odd ? h : (s.x == 0 ? h + (hx - 1) : h - 1);
    hop64_dir<0, true>(ln, Us, in.at(ln, hf, 1 - odd), sg, Su, Sl);
    hop64_dir<0, false>(ln, U + (int64_t)(2 * hb + 1 - odd) * 36, in.at(ln, hb, 1 - odd), sg, Su, Sl);
  }
  int st = hx;
  {
    const int hf = s.y == g.L[1] - 1 ? h - (g.L[1] - 1) * st : h + st;
    const int hb = s.y == 0 ? h + (g.L[1] - 1) * st : h - st;
    hop64_dir<1, true>(ln, Us + 9, in.at(ln, hf, odd), sg, Su, Sl);
    hop64_dir<1, false>(ln, U + (int64_t)(2 * hb + odd) * 36 + 9, in.at(ln, hb, odd), sg, Su, Sl);
  }
  // so far Sl belongs to the partner's row
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    Sl[a].x = __shfl_xor_sync(0xffffffffu, Sl[a].x, 16);
    Sl[a].y = __shfl_xor_sync(0xffffffffu, Sl[a].y, 16);
  }
  st *= g.L[1];
  {
    const int hf = s.z == g.L[2] - 1 ? h - (g.L[2] - 1) * st : h + st;
    const int hb = s.z == 0 ? h + (g.L[2] - 1) * st : h - st;
    hop64_dir<2, true>(ln, Us + 18, in.at(ln, hf, odd), sg, Su, Sl);
    hop64_dir<2, false>(ln, U + (int64_t)(2 * hb + odd) * 36 + 18, in.at(ln, hb, odd), sg, Su, Sl);
  }
  st *= g.L[2];
  {
    const int hf = s.t == g.L[3] - 1 ? h - (g.L[3] - 1) * st : h + st;
    const int hb = s.t == 0 ? h + (g.L[3] - 1) * st : h - st;
    hop64_dir<3, true>(ln, Us + 27, in.at(ln, hf, odd), sg, Su, Sl);
    hop64_dir<3, false>(ln, U + (int64_t)(2 * hb + odd) * 36 + 27, in.at(ln, hb, odd), sg, Su, Sl);
  }
}

// Sums over the block of F values of this thread's column: part[block * F b + q b + j], in one fixed order.
template <int F, int T>
__device__ __forceinline__ void block_sums64(double (&v)[F], int b, double *__restrict__ part, double *shw) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int bw = b < 16 ? b : 16;  // columns that one warp holds
#pragma unroll
  for (int q = 0; q < F; ++q) v[q] += __shfl_xor_sync(0xffffffffu, v[q], 16);  // the two spin rows
  for (int off = 8; off >= b; off >>= 1) {
#pragma unroll
    for (int q = 0; q < F; ++q) v[q] += __shfl_xor_sync(0xffffffffu, v[q], off);
  }
  if (lane < bw) {
#pragma unroll
    for (int q = 0; q < F; ++q) shw[(w * F + q) * bw + lane] = v[q];
  }
  __syncthreads();
  const int n = F * b, cw = b > 16 ? b >> 4 : 1;  // warps that share a set of columns
  for (int k = threadIdx.x; k < n; k += T) {
    const int q = k / b, j = k & (b - 1);
    double s = 0.0;
    for (int ww = j >> 4; ww < T / 32; ww += cw) s += shw[(ww * F + q) * bw + (j & (bw - 1))];
    part[(int64_t)blockIdx.x * n + k] = s;
  }
}

// tot[k] = sum over blocks of part[block * n + k], k < n, in one fixed order
template <int T>
__device__ __forceinline__ void grid_sums64(int n, const double *__restrict__ part, double2 *sh, double *tot) {
  const int t = threadIdx.x, G = gridDim.x, Q = n >> 1;
  int S = T / Q;
  if (S < 1) S = 1;
  if (S > 16) S = 16;
  const int ch = (G + S - 1) / S;
  __syncthreads();  // the partial sums above have read sh's memory
  for (int k = t; k < S * Q; k += T) {
    const int q = k % Q, sl = k / Q, lo = sl * ch, hi = min(G, lo + ch);
    double2 a = make_double2(0.0, 0.0);
    const double2 *src = (const double2 *)part + q;
    for (int k0 = lo; k0 < hi; k0 += 8) {
      double2 v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = k0 + u < hi ? __ldcg(src + (int64_t)(k0 + u) * Q) : make_double2(0.0, 0.0);
#pragma unroll
      for (int u = 0; u < 8; ++u) a = cadd(a, v[u]);
    }
    sh[k] = a;
  }
  __syncthreads();
  for (int k = t; k < n; k += T) {
    double s = ((const double *)sh)[k];
    for (int u = 1; u < S; ++u) s += ((const double *)sh)[u * n + k];
    tot[k] = s;
  }
  __syncthreads();
}

__device__ __forceinline__ void cdot64(double &re, double &im, double2 a, double2 b) {  // += conj(a) b
  re = fma(a.x, b.x, fma(a.y, b.y, re));
  im = fma(a.x, b.y, fma(-a.y, b.x, im));
}
__device__ __forceinline__ void norm64(double &s, double2 a) { s = fma(a.x, a.x, fma(a.y, a.y, s)); }

template <int T> __global__ void __launch_bounds__(T, 1) k_bicgstab_eo64(Eo64Args a) {
  constexpr int kShw = T / 32 * 8 * 16 * 8, kSh = 8 * 64 / 2 * 16 > T * 16 ? 8 * 64 / 2 * 16 : T * 16;
  __shared__ __align__(16) unsigned char smem[kShw > kSh ? kShw : kSh];
  __shared__ double tot[8 * 64];
  __shared__ Scal ss;          // this block's copy of the per-column scalars
  __shared__ int cyc_act[64];  // columns that this cycle iterates on
  double *shw = (double *)smem;
  double2 *sh = (double2 *)smem;
  const int b = a.b, logb = a.logb;
  const L64 ln(2 * b, threadIdx.x);
  const int P = b, j = ln.jp;
  const int64_t npair = (int64_t)(a.g.V >> 1) << logb;
  const Sweep<T, 128> pairs(2 * npair);
  const unsigned int G = gridDim.x;
  double *part[2] = {(double *)a.partial, (double *)a.partial + (int64_t)8 * 64 * G};
  unsigned int nbar = 0, nred = 0;
  if (threadIdx.x == 0) atomicMax(&a.gs->nt0, ~global_ns());
  {
    const int *src = (const int *)a.sc;
    int *dst = (int *)&ss;
    for (int i = threadIdx.x; i < (int)(sizeof(Scal) / sizeof(int)); i += T) dst[i] = __ldcg(src + i);
  }
  const bool zero0 = *(volatile const int *)&a.gs->x_nonzero == 0;  // the initial guess is zero
  __syncthreads();
  const int own[6] = {ln.cu, ln.cu + P, ln.cu + 2 * P, ln.clz, ln.clz + P, ln.clz + 2 * P};
  const double D = a.diag, wsc = 0.25 / D, isc = 0.5 / D, dinv = 1.0 / D;
  // body(site, offset of this thread's half-lattice elements, valid) for the sites of one parity
  auto for_sites = [&](int parity, auto body) {
    pairs.run([&](int64_t it) {
      const int64_t pr = L64::pair_of_item(it);
      const bool valid = pr < npair;
      const EoSite s = eo_site(a.g, valid ? (int)(pr >> logb) : 0, parity);
      body(s, (int64_t)s.h * 12 * P + j, valid);
    });
  };
  auto barrier = [&]() { return grid_arrive_wait(a.gs, ++nbar * G, kSpinBudget); };
  // w on the odd sites from the hops of an even field
  auto odd_phase = [&](const double2 *f) {
    for_sites(1, [&](const EoSite &s, int64_t q, bool valid) {
      double2 S[2][3];
      hop64(ln, a.U, HalfLoad64{f}, a.g, s, S[0], S[1]);
      if (valid) {
#pragma unroll
        for (int k = 0; k < 6; ++k) a.w[q + own[k]] = cscale(S[k / 3][k % 3], k < 3 ? wsc : -wsc);
      }
    });
  };
  // this thread's row of D f - H w at an even site
  auto schur_row = [&](const EoSite &s, const double2 *f, int64_t q, double2 (&fv)[6], double2 (&o)[6]) {
    double2 S[2][3];
    hop64(ln, a.U, HalfLoad64{a.w}, a.g, s, S[0], S[1]);
#pragma unroll
    for (int k = 0; k < 6; ++k) fv[k] = f[q + own[k]];
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      const double2 h = S[k / 3][k % 3];
      o[k] = k < 3 ? make_double2(fma(D, fv[k].x, -h.x), fma(D, fv[k].y, -h.y))
                   : make_double2(fma(D, fv[k].x, h.x), fma(D, fv[k].y, h.y));
    }
  };
  int done = 0;
  bool ok = true;

  for (int cycle = 0; ok && cycle < a.max_cycles; ++cycle) {
    {  // true residual on both sublattices: (||r||^2, ||z||^2) -> restart decision
      double d[2] = {0.0, 0.0};
      for (int parity = 0; parity < 2; ++parity) {
        double2 *r = parity ? a.ro : a.r;
        for_sites(parity, [&](const EoSite &s, int64_t q, bool valid) {
          const int64_t lex = (int64_t)eo_lex(s) * 12 * P + j;
          double2 S[2][3];
          const bool with_x = cycle > 0 || !zero0;
          if (with_x) hop64(ln, a.U, LexLoad64{a.x}, a.g, s, S[0], S[1]);
          if (!valid) return;
          double2 zz[6], xx[6];
#pragma unroll
          for (int k = 0; k < 6; ++k) {
            zz[k] = a.z[lex + own[k]];
            xx[k] = with_x ? a.x[lex + own[k]] : make_double2(0.0, 0.0);
          }
#pragma unroll
          for (int k = 0; k < 6; ++k) {
            double2 rr = zz[k];
            if (with_x) {
              const double hf = k < 3 ? 0.5 : -0.5;
              rr.x = fma(hf, S[k / 3][k % 3].x, fma(-D, xx[k].x, rr.x));
              rr.y = fma(hf, S[k / 3][k % 3].y, fma(-D, xx[k].y, rr.y));
            }
            r[q + own[k]] = rr;
            norm64(d[0], rr);
            norm64(d[1], zz[k]);
          }
        });
      }
      double *pb = part[nred++ & 1];
      block_sums64<2, T>(d, b, pb, shw);
      if (!(ok = barrier())) break;
      grid_sums64<T>(2 * b, pb, sh, tot);
      if (threadIdx.x < b) {
        fin_resid(&ss, threadIdx.x, make_double2(tot[threadIdx.x], tot[b + threadIdx.x]), 1);
        cyc_act[threadIdx.x] = ss.active[threadIdx.x];
      }
      const int na = __syncthreads_count(threadIdx.x < b && ss.active[threadIdx.x]);
      if (threadIdx.x == 0) ss.n_active = na;
      if (na == 0) break;
    }
    int n_active;
    {  // Schur problem: r = rhat = p = r_e + H r_o / (2 D)
      double d[2] = {0.0, 0.0};
      for_sites(0, [&](const EoSite &s, int64_t q, bool valid) {
        double2 S[2][3];
        hop64(ln, a.U, HalfLoad64{a.ro}, a.g, s, S[0], S[1]);
        if (!valid) return;
#pragma unroll
        for (int k = 0; k < 6; ++k) {
          double2 rr = a.r[q + own[k]];
          rr = adds(rr, S[k / 3][k % 3], k < 3 ? isc : -isc);
          a.r[q + own[k]] = rr;
          a.rhat[q + own[k]] = rr;
          a.p[q + own[k]] = rr;
          norm64(d[0], rr);
        }
      });
      double *pb = part[nred++ & 1];
      block_sums64<2, T>(d, b, pb, shw);
      if (!(ok = barrier())) break;
      grid_sums64<T>(2 * b, pb, sh, tot);
      if (threadIdx.x < b) {
        const int c = threadIdx.x;
        ss.rho[c] = make_double2(tot[c], 0.0);
        ss.rnorm2[c] = tot[c];
        if (tot[c] <= ss.tol2 * ss.bnorm2[c]) ss.active[c] = 0;  // only the odd sites are left to solve
      }
      n_active = __syncthreads_count(threadIdx.x < b && ss.active[threadIdx.x]);
    }
    for (int iter = 0; n_active > 0 && iter < a.max_iters; ++iter) {
      ++done;
      if (blockIdx.x == 0 && threadIdx.x == 0) a.gs->iters = done;
      odd_phase(a.p);  // A
      if (!(ok = barrier())) break;
      {
        double d[2] = {0.0, 0.0};
        for_sites(0, [&](const EoSite &s, int64_t q, bool valid) {  // B
          double2 p[6], v[6];
          schur_row(s, a.p, q, p, v);
          if (!valid) return;
          double2 rh[6];
#pragma unroll
          for (int k = 0; k < 6; ++k) rh[k] = a.rhat[q + own[k]];
#pragma unroll
          for (int k = 0; k < 6; ++k) {
            a.v[q + own[k]] = v[k];
            cdot64(d[0], d[1], rh[k], v[k]);
          }
        });
        double *pb = part[nred++ & 1];
        block_sums64<2, T>(d, b, pb, shw);
        if (!(ok = barrier())) break;
        grid_sums64<T>(2 * b, pb, sh, tot);
        if (threadIdx.x < b) fin_alpha(&ss, threadIdx.x, make_double2(tot[threadIdx.x], tot[b + threadIdx.x]));
        __syncthreads();
      }
      const double2 al = ss.alpha[j], mal = cneg(al);
      for_sites(0, [&](const EoSite &, int64_t q, bool valid) {  // S
        if (!valid) return;
        double2 r[6], v[6];
#pragma unroll
        for (int k = 0; k < 6; ++k) {
          r[k] = a.r[q + own[k]];
          v[k] = a.v[q + own[k]];
        }
#pragma unroll
        for (int k = 0; k < 6; ++k) a.r[q + own[k]] = caxpy(mal, v[k], r[k]);
      });
      if (!(ok = barrier())) break;
      odd_phase(a.r);  // C
      if (!(ok = barrier())) break;
      {
        double d[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
        for_sites(0, [&](const EoSite &s, int64_t q, bool valid) {  // D
          double2 sv[6], t[6];
          schur_row(s, a.r, q, sv, t);
          if (!valid) return;
          double2 rh[6];
#pragma unroll
          for (int k = 0; k < 6; ++k) rh[k] = a.rhat[q + own[k]];
#pragma unroll
          for (int k = 0; k < 6; ++k) {
            a.t[q + own[k]] = t[k];
            cdot64(d[0], d[1], t[k], sv[k]);    // t^H s
            norm64(d[2], t[k]);                 // t^H t
            cdot64(d[3], d[4], rh[k], sv[k]);   // rhat^H s
            cdot64(d[5], d[6], rh[k], t[k]);    // rhat^H t
            norm64(d[7], sv[k]);                // s^H s
          }
        });
        double *pb = part[nred++ & 1];
        block_sums64<8, T>(d, b, pb, shw);
        if (!(ok = barrier())) break;
        grid_sums64<T>(8 * b, pb, sh, tot);
        if (threadIdx.x < b) {
          const double *x = tot + threadIdx.x;
          fin_omega_beta(&ss, threadIdx.x, make_double2(x[0], x[b]), make_double2(x[2 * b], 0.0),
                         make_double2(x[3 * b], x[4 * b]), make_double2(x[5 * b], x[6 * b]),
                         make_double2(x[7 * b], 0.0));
        }
        n_active = __syncthreads_count(threadIdx.x < b && ss.active[threadIdx.x]);
        if (threadIdx.x == 0) ss.n_active = n_active;
      }
      {  // E
        const double2 om = ss.omega[j], mom = cneg(om), be = ss.beta[j];
        const bool act = ss.active[j] != 0, moves = act || al.x != 0.0 || al.y != 0.0;
        for_sites(0, [&](const EoSite &s, int64_t q, bool valid) {
          if (!valid || !moves) return;  // (a column that stopped earlier)
          double2 *xs = a.x + (int64_t)eo_lex(s) * 12 * P + j;
          double2 sv[6], p[6], x[6], t[6], v[6];
#pragma unroll
          for (int k = 0; k < 6; ++k) {
            sv[k] = a.r[q + own[k]];
            p[k] = a.p[q + own[k]];
            x[k] = xs[own[k]];
            t[k] = a.t[q + own[k]];
            v[k] = a.v[q + own[k]];
          }
#pragma unroll
          for (int k = 0; k < 6; ++k) {
            xs[own[k]] = caxpy(om, sv[k], caxpy(al, p[k], x[k]));
            const double2 rn = caxpy(mom, t[k], sv[k]);
            a.r[q + own[k]] = rn;
            if (act) a.p[q + own[k]] = caxpy(be, caxpy(mom, v[k], p[k]), rn);
          }
        });
        if (!(ok = barrier())) break;  // p (and x) are read at neighbours next
      }
    }
    if (!ok) break;
    // x_o = (z_o + H x_e / 2) / D for the columns of this cycle
    const bool mine = cyc_act[j] != 0;
    for_sites(1, [&](const EoSite &s, int64_t, bool valid) {
      double2 S[2][3];
      hop64(ln, a.U, LexLoad64{a.x}, a.g, s, S[0], S[1]);
      if (!valid || !mine) return;
      const int64_t lex = (int64_t)eo_lex(s) * 12 * P + j;
#pragma unroll
      for (int k = 0; k < 6; ++k) {
        const double2 zz = a.z[lex + own[k]], h = S[k / 3][k % 3];
        const double f = k < 3 ? isc : -isc;
        a.x[lex + own[k]] = make_double2(fma(f, h.x, dinv * zz.x), fma(f, h.y, dinv * zz.y));
      }
    });
    if (!(ok = barrier())) break;
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

constexpr int kEo64Threads = 256;

int launch_persistent_eo64(const Eo64Args &ea, cudaStream_t st) {
  static int max_grid = 0;
  auto *kern = k_bicgstab_eo64<kEo64Threads>;
  if (!max_grid) {
    int nb = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kern, kEo64Threads, 0);
    if (e != cudaSuccess) return cuda_fail(e, "persistent solver occupancy");
    if (nb < 1) return fail(DTR_ECUDA, "persistent solver cannot be resident");
    max_grid = nb * device_sms();
    if (max_grid > kPersistMaxGrid) max_grid = kPersistMaxGrid;
  }
  const int grid = (ea.grid > 0 && ea.grid < max_grid) ? ea.grid : max_grid;
  Eo64Args copy = ea;
  void *args[] = {&copy};
  DTR_CUDA(cudaLaunchCooperativeKernel((const void *)kern, dim3(grid), dim3(kEo64Threads), args, 0, st));
  count_launches(1);
  if (persist_profile().on) return persist_account(ea.gs, (double)ea.g.V * ea.b, st);
  return DTR_OK;
}

}  // namespace dtr
