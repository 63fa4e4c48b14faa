// Plain dslash (A or A^H) on internal fields, and the canonical <-> internal
// layout conversions used at the C-ABI boundary.
#include "dslash_core.cuh"

namespace dtr {

// FP32: two blocks of 256 to an SM (128 registers) for the loads in flight.  FP64 is bound by its pipe either way, but
// keeps an SM full with 256 threads: blocks of 64, so that the last ones spread over the SMs (8^4 x 32 in blocks of 256
// is 3.4 rounds of one to an SM).  A 4^4 call with its copies: 68 -> 33 us.
template <typename R> constexpr int dslash_block() { return sizeof(R) == 4 ? 256 : 64; }
template <typename R, int SGN>
__global__ void __launch_bounds__(dslash_block<R>(), sizeof(R) == 4 ? 2 : 4) dslash_kernel(const typename cplx_t<R>::type *__restrict__ U,
                                                     const typename cplx_t<R>::type *__restrict__ in,
                                                     typename cplx_t<R>::type *__restrict__ out, Geom g, int b,
                                                     int logb, R diag) {
  typedef typename cplx_t<R>::type C;
  const int64_t n = (int64_t)g.V << logb;
  for (int64_t it = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; it < n; it += (int64_t)gridDim.x * blockDim.x) {
    const int j = (int)(it & (b - 1));
    const int s = (int)(it >> logb);
    C o[12], self[12];
    dslash_site<SGN, R>(U, in, g, b, s, j, diag, o, self);
    C *q = out + (int64_t)s * 12 * b + j;
#pragma unroll
    for (int c = 0; c < 12; ++c) q[c * b] = o[c];
  }
}

static int ilog2(int b) {
  int l = 0;
  while ((1 << l) < b) ++l;
  return l;
}

template <typename R>
void launch_dslash(const typename cplx_t<R>::type *U, const typename cplx_t<R>::type *in,
                   typename cplx_t<R>::type *out, const Geom &g, int b, double m0, int dagger, cudaStream_t st) {
  const int64_t n = (int64_t)g.V * b;
  constexpr int T = dslash_block<R>();
  const unsigned grid = (unsigned)((n + T - 1) / T);
  if (dagger)
    dslash_kernel<R, -1><<<grid, T, 0, st>>>(U, in, out, g, b, ilog2(b), (R)(4.0 + m0));
  else
    dslash_kernel<R, 1><<<grid, T, 0, st>>>(U, in, out, g, b, ilog2(b), (R)(4.0 + m0));
  count_launches(1);
}

template void launch_dslash<double>(const double2 *, const double2 *, double2 *, const Geom &, int, double, int,
                                    cudaStream_t);
template void launch_dslash<float>(const float2 *, const float2 *, float2 *, const Geom &, int, double, int,
                                   cudaStream_t);

// ------------------------------------------------------------------ layouts
// Canonical [column][dof] to [dof][b] and back: a transposition, bound by HBM.  A block moves a tile of kTile / b
// dofs by b columns through shared memory, so that both sides are read and written in whole lines (one element per
// thread straight across left the column side with a 16-byte piece of each line: 32^3 x 64 x 16, FP64, unpack 8.1 ms
// and pack 2.3 ms; 16^3 x 32 x 16 FP32 491 and 141 us).
constexpr int kTile = 2048, kPerThread = kTile / 256;

template <typename C> __device__ __forceinline__ C as_c(double2 v);
template <> __device__ __forceinline__ double2 as_c<double2>(double2 v) { return v; }
template <> __device__ __forceinline__ float2 as_c<float2>(double2 v) { return f64_to_f32(v); }
__device__ __forceinline__ double2 as_d(double2 v) { return v; }
__device__ __forceinline__ double2 as_d(float2 v) { return f32_to_f64(v); }

template <typename R>
__global__ void __launch_bounds__(256) pack_kernel(const double2 *__restrict__ canon,
                                                   typename cplx_t<R>::type *__restrict__ internal, int64_t N,
                                                   int nrhs, int logb) {
  typedef typename cplx_t<R>::type C;
  extern __shared__ __align__(16) unsigned char smem[];
  C *sm = (C *)smem;
  const int b = 1 << logb, logt = 11 - logb, TI = 1 << logt;  // dofs of a tile
  const int64_t tiles = (N + TI - 1) >> logt;
  for (int64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
    const int64_t i0 = t << logt;
    double2 v[kPerThread];
#pragma unroll
    for (int u = 0; u < kPerThread; ++u) {
      const int e = u * 256 + threadIdx.x, j = e >> logt;
      const int64_t i = i0 + (e & (TI - 1));
      v[u] = (j < nrhs && i < N) ? canon[(int64_t)j * N + i] : make_double2(0.0, 0.0);
    }
#pragma unroll
    for (int u = 0; u < kPerThread; ++u) {
      const int e = u * 256 + threadIdx.x;
      sm[(e >> logt) * (TI + 1) + (e & (TI - 1))] = as_c<C>(v[u]);
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < kPerThread; ++u) {
      const int e = u * 256 + threadIdx.x, ii = e >> logb;
      if (i0 + ii < N) internal[(i0 << logb) + e] = sm[(e & (b - 1)) * (TI + 1) + ii];
    }
    __syncthreads();
  }
}

template <typename R>
__global__ void __launch_bounds__(256) unpack_kernel(const typename cplx_t<R>::type *__restrict__ internal,
                                                     double2 *__restrict__ canon, int64_t N, int nrhs, int logb) {
  typedef typename cplx_t<R>::type C;
  extern __shared__ __align__(16) unsigned char smem[];
  C *sm = (C *)smem;
  const int b = 1 << logb, logt = 11 - logb, TI = 1 << logt;
  const int64_t tiles = (N + TI - 1) >> logt;
  for (int64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
    const int64_t i0 = t << logt;
    C v[kPerThread];
#pragma unroll
    for (int u = 0; u < kPerThread; ++u) {
      const int e = u * 256 + threadIdx.x;
      v[u] = i0 + (e >> logb) < N ? internal[(i0 << logb) + e] : mk<C>(0.0, 0.0);
    }
#pragma unroll
    for (int u = 0; u < kPerThread; ++u) {
      const int e = u * 256 + threadIdx.x;
      sm[(e & (b - 1)) * (TI + 1) + (e >> logb)] = v[u];
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < kPerThread; ++u) {
      const int e = u * 256 + threadIdx.x, j = e >> logt, ii = e & (TI - 1);
      if (j < nrhs && i0 + ii < N) canon[(int64_t)j * N + i0 + ii] = as_d(sm[j * (TI + 1) + ii]);
    }
    __syncthreads();
  }
}

// Blocks of at most kSmallBlock values go one value a thread: the tiles' chain of loads, barrier and stores is longer
// than all of that takes (an FP32 stencil call, tiles and this: 6x4x10x6 x 3 40.6 and 38.1 us, 8^4 x 2 42.7 and 41.2 us;
// from 8^4 x 8, 393 k values, on the tiles are as fast, at 8^3 x 16 x 16 56 us against 67).
constexpr int64_t kSmallBlock = 1 << 18;
template <typename R>
__global__ void __launch_bounds__(256) pack_small_kernel(const double2 *__restrict__ canon,
                                                         typename cplx_t<R>::type *__restrict__ internal, int N, int nrhs,
                                                         int logb) {
  typedef typename cplx_t<R>::type C;
  const int e = blockIdx.x * 256 + threadIdx.x, i = e >> logb, j = e & ((1 << logb) - 1);
  if (i < N) internal[e] = j < nrhs ? as_c<C>(canon[j * N + i]) : mk<C>(0.0, 0.0);
}
template <typename R>
__global__ void __launch_bounds__(256) unpack_small_kernel(const typename cplx_t<R>::type *__restrict__ internal,
                                                           double2 *__restrict__ canon, int N, int nrhs, int logb) {
  const int e = blockIdx.x * 256 + threadIdx.x;
  if (e < N * nrhs) canon[e] = as_d(internal[((e % N) << logb) + e / N]);
}

// one column: a plain conversion
template <typename D, typename S>
__global__ void __launch_bounds__(256) convert_kernel(const S *__restrict__ in, D *__restrict__ out, int64_t n) {
  for (int64_t e = (int64_t)blockIdx.x * 256 + threadIdx.x; e < n; e += (int64_t)gridDim.x * 256) {
    out[e] = as_c<D>(as_d(in[e]));
  }
}

static unsigned tile_grid(int64_t N, int b) {
  const int64_t t = (N * b + kTile - 1) / kTile;
  return (unsigned)(t < 65536 ? (t < 1 ? 1 : t) : 65536);
}
template <typename C> static size_t tile_bytes(int b) { return (size_t)(kTile + b) * sizeof(C); }

template <typename R>
void launch_pack(const double2 *canon, typename cplx_t<R>::type *internal, int64_t V, int nrhs, int b,
                 cudaStream_t st) {
  typedef typename cplx_t<R>::type C;
  const int64_t N = V * 12;
  if (b == 1)
    convert_kernel<C, double2><<<tile_grid(N, 8), 256, 0, st>>>(canon, internal, N);
  else if (N * b <= kSmallBlock)
    pack_small_kernel<R><<<(unsigned)((N * b + 255) / 256), 256, 0, st>>>(canon, internal, (int)N, nrhs, ilog2(b));
  else
    pack_kernel<R><<<tile_grid(N, b), 256, tile_bytes<C>(b), st>>>(canon, internal, N, nrhs, ilog2(b));
  count_launches(1);
}
template <typename R>
void launch_unpack(const typename cplx_t<R>::type *internal, double2 *canon, int64_t V, int nrhs, int b,
                   cudaStream_t st) {
  typedef typename cplx_t<R>::type C;
  const int64_t N = V * 12;
  if (b == 1)
    convert_kernel<double2, C><<<tile_grid(N, 8), 256, 0, st>>>(internal, canon, N);
  else if (N * b <= kSmallBlock)
    unpack_small_kernel<R><<<(unsigned)((N * nrhs + 255) / 256), 256, 0, st>>>(internal, canon, (int)N, nrhs, ilog2(b));
  else
    unpack_kernel<R><<<tile_grid(N, b), 256, tile_bytes<C>(b), st>>>(internal, canon, N, nrhs, ilog2(b));
  count_launches(1);
}

template void launch_pack<double>(const double2 *, double2 *, int64_t, int, int, cudaStream_t);
template void launch_pack<float>(const double2 *, float2 *, int64_t, int, int, cudaStream_t);
template void launch_unpack<double>(const double2 *, double2 *, int64_t, int, int, cudaStream_t);
template void launch_unpack<float>(const float2 *, double2 *, int64_t, int, int, cudaStream_t);

}  // namespace dtr
