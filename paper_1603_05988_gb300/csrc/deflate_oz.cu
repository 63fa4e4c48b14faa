// Deflation projection of general FP64 blocks on the tensor cores: C = V^H [Z, g5 Z] and x0 = V W from exact integer
// products, where that is as accurate as FP64 sums.
//
// FP64 runs at two lanes a clock per SM, so the plain contraction costs 8 N k b FP64 instructions (16^3 x 32, k = 64,
// b = 16: 24 ms, and 17 ms for x0).  Here every real column of V and Z is written as integers of 54 bits times a power
// of two (relative to the column's largest entry), the integers as seven balanced base-256 digits (Ozaki, Ogita, Oishi
// and Rump's error-free splitting, Numer. Algorithms 59, 2012), and the digit products run as BF16 mma with FP32
// accumulation: a digit is exact in BF16, a product at most 2^14, and 128 of them times the seven digit pairs of one
// weight stay below 2^24, so nothing is rounded.  The weights 256^5 and up are kept (34 of the 49 digit pairs); what is
// dropped is 2^-57 of the product of the column maxima, below the rounding of an FP64 sum.  The sums of one weight go to
// 64-bit integers, and to FP64 once at the end.
//
// Integers are fixed point where FP64 floats: an entry is off by up to 2^-55 of its column's largest, so a product of two
// entries that are both small for their columns loses digits.  Two tests on the device send such blocks to the FP64
// kernels (a point source; vectors that decay from opposite ends):
//   C   S = sum of the products of the entries' moduli, in units of the columns' powers of two, must reach a bound T
//       (k_oz_mass).  The digits' error goes with the squares that meet a rounded partner: T^2 = 4 (sum |v|^2 + sum |z|^2
//       where v is rounded + 2^-13 n for the dropped pairs), or n / 2 for n nonzero entries of z if that is less.  At S = T
//       it is 0.06 2^-53 of sum |v| |z|; FP64 chains come to 0.02 to 0.3 (49152 dofs, 24 families of graded, localised,
//       sparse and plain columns).  Gaussian columns reach 6 T (FP64) and 12 T (FP32) there, growing with sqrt(n).
//   x0  sixteen neighbouring entries of a column, together, must be 2^50 times the error that they can have: that of V's
//       entries where V is FP64 (2^-55 / sqrt(3) of the columns' powers of two, times the weights), and the digit pairs that
//       are dropped (k_oz_expand).  FP32 and BF16 entries are exact in 54 bits down to 2^-30 of the largest, those below are
//       counted tile by tile.  Largest errors of 16 entries above the line 7e-16, FP64 sums 9e-16 (spaces of the
//       eigensolver, 8^4 to 16^3 x 32, k = 16 to 100); its spaces at 16^4, FP64, are partly below.
//
// Digits come from shifts and byte permutes on the integer pipe.  A digit plane of Z that is zero over a stage is
// skipped: probing noise (entries 0, +-1, +-i) has one digit.
//
// 16^3 x 32, FP32 space, k = 64, b = 16, with x0: 42.0 -> 5.7 ms.  Relative error against exact sums there: x0
// 4.8e-16 -> 1.6e-16, C 8.6e-17 -> 8.5e-17 (the FP64 kernels add in a chain).
#include "deflate_oz.cuh"

#include <cmath>

namespace dtr {

constexpr int kDig = 7;          // digits
constexpr int kMinW = 5;         // least digit weight kept: pairs (i, j) with i + j >= kMinW
constexpr int kGrp = 2 * kDig - 1 - kMinW;  // weights kept
constexpr int kIntBits = 54;     // an entry below 2^e becomes an integer below 2^54: its top digit is at most 64

// ------------------------------------------------------------------ digits
// entry times 2^(kIntBits - e), rounded to an integer, plus 128 in each of the seven digits: byte i is digit i + 128
__device__ __forceinline__ unsigned long long biased(unsigned long long mant, int sh, bool neg) {
  unsigned long long q;
  if (sh >= 0)
    q = mant << sh;
  else if (sh > -60)
    q = (mant + (1ull << (-sh - 1))) >> -sh;
  else
    q = 0;
  const unsigned long long bias = 0x0080808080808080ull;
  return neg ? bias - q : bias + q;
}
__device__ __forceinline__ unsigned long long digits_of(float f, int e) {
  const unsigned b = __float_as_uint(f);
  const int ex = (b >> 23) & 0xff;
  const unsigned long long m = ex ? (b & 0x7fffffu) | 0x800000u : 0u;  // (subnormal: far below the column's largest)
  return biased(m, ex - 150 + kIntBits - e, b >> 31);
}
__device__ __forceinline__ unsigned long long digits_of(double d, int e) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(d);
  const int ex = (int)(b >> 52) & 0x7ff;
  const unsigned long long m = ex ? (b & 0xfffffffffffffull) | 0x10000000000000ull : 0ull;
  return biased(m, ex - 1075 + kIntBits - e, b >> 63);
}
struct Dig2 {  // the digits of a complex entry
  unsigned long long re, im;
};
__device__ __forceinline__ Dig2 dig(float2 v, int e) { return Dig2{digits_of(v.x, e), digits_of(v.y, e)}; }
__device__ __forceinline__ Dig2 dig(double2 v, int e) { return Dig2{digits_of(v.x, e), digits_of(v.y, e)}; }
__device__ __forceinline__ Dig2 dig(bfc2 v, int e) { return dig(__bfloat1622float2(v), e); }
constexpr unsigned long long kNoDig = 0x0080808080808080ull;
// entry times 2^-e
__device__ __forceinline__ float2 scaled(float2 v, int e) { return make_float2(ldexpf(v.x, -e), ldexpf(v.y, -e)); }
__device__ __forceinline__ float2 scaled(double2 v, int e) {
  return f64_to_f32(make_double2(scalbn(v.x, -e), scalbn(v.y, -e)));
}
__device__ __forceinline__ float2 scaled(bfc2 v, int e) { return scaled(__bfloat1622float2(v), e); }
// whether the integer of an FP32 (or BF16) entry loses bits; b: its bits without the sign
__device__ __forceinline__ int loses_bits(unsigned b, int e) {
  const int x = (int)(b >> 23), sh = x - 150 + kIntBits - e;
  return sh < 0 && b != 0u && (x == 0 || sh <= -24 || (b & ((1u << -sh) - 1u)) != 0u);
}
__device__ __forceinline__ int loses_bits(float2 v, int e) {
  const unsigned a = __float_as_uint(v.x) & 0x7fffffffu, b = __float_as_uint(v.y) & 0x7fffffffu;
  if ((int)(min(a, b) >> 23) >= 150 - kIntBits + e) return 0;  // nearly always
  return loses_bits(a, e) + loses_bits(b, e);
}
__device__ __forceinline__ int loses_bits(bfc2 v, int e) { return loses_bits(__bfloat1622float2(v), e); }
__device__ __forceinline__ int loses_bits(double2, int) { return 0; }  // (nearly all do: not counted)

// digit i of a biased integer as a float (exact): 2^23 + byte, minus 2^23 + 128
__device__ __forceinline__ float digit(unsigned long long q, int i) {
  const unsigned w = i < 4 ? (unsigned)q : (unsigned)(q >> 32);
  return __uint_as_float(__byte_perm(w, 0x4b000000u, 0x7640 | (i & 3))) - 8388736.f;
}
// digits i of re and im as a BF16 pair
__device__ __forceinline__ unsigned digit_pair(const Dig2 &d, int i) {
  return __byte_perm(__float_as_uint(digit(d.re, i)), __float_as_uint(digit(d.im, i)), 0x7632);
}
// bit i: digit i is not zero in re or im
__device__ __forceinline__ int digit_mask(const Dig2 &d) {
  const unsigned long long x = (d.re ^ kNoDig) | (d.im ^ kNoDig);
  int m = 0;
#pragma unroll
  for (int i = 0; i < kDig; ++i) m |= ((x >> (8 * i)) & 0xff) ? 1 << i : 0;
  return m;
}

// -------------------------------------------------------------- exponents
// e with |entry| < 2^e over a column; kBad: an entry is not finite, or all are so small that the integers would lose
// bits (subnormals among them); kZero: the column is zero
constexpr int kBad = 1 << 20, kZero = -(1 << 20);

// emax[m] = largest biased exponent field of column m over all rows (0: none above the subnormals)
__device__ __forceinline__ int exp_field(float2 v) {
  return max((int)(__float_as_uint(v.x) >> 23) & 0xff, (int)(__float_as_uint(v.y) >> 23) & 0xff);
}
__device__ __forceinline__ int exp_field(double2 v) {
  return max((__double2hiint(v.x) >> 20) & 0x7ff, (__double2hiint(v.y) >> 20) & 0x7ff);
}
__device__ __forceinline__ int exp_field(bfc2 v) { return exp_field(__bfloat1622float2(v)); }
__device__ __forceinline__ bool is_zero(float2 v) { return v.x == 0.f && v.y == 0.f; }
__device__ __forceinline__ bool is_zero(double2 v) {
  return (((unsigned long long)__double_as_longlong(v.x) | (unsigned long long)__double_as_longlong(v.y)) << 1) == 0;
}
__device__ __forceinline__ bool is_zero(bfc2 v) { return is_zero(__bfloat1622float2(v)); }

// stat[c]: 0 while the column is all zeros, else 1 + the largest exponent field; count[c] (or NULL): nonzero entries
template <typename T>
__global__ void __launch_bounds__(256)
    k_oz_exp(const T *__restrict__ F, int64_t rows, int cols, int *__restrict__ stat, int *__restrict__ count) {
  __shared__ int most[256], number[256];
  for (int c0 = 0; c0 < cols; c0 += 256) {
    const int w = min(256, cols - c0), g = 256 / w;  // g rows of w columns at once
    const int c = threadIdx.x % w, r = threadIdx.x / w;
    most[threadIdx.x] = number[threadIdx.x] = 0;
    __syncthreads();
    if (r < g) {
      int m = 0, n = 0;
      for (int64_t i = (int64_t)blockIdx.x * g + r; i < rows; i += (int64_t)gridDim.x * g) {
        const T v = F[i * cols + c0 + c];
        if (is_zero(v)) continue;
        m = max(m, 1 + exp_field(v));
        ++n;
      }
      if (m) atomicMax(&most[c], m);  // (neither the largest nor the count depends on the order)
      if (n) atomicAdd(&number[c], n);
    }
    __syncthreads();
    if (threadIdx.x < w && number[threadIdx.x]) {
      atomicMax(&stat[c0 + threadIdx.x], most[threadIdx.x]);
      if (count) atomicAdd(&count[c0 + threadIdx.x], number[threadIdx.x]);
    }
    __syncthreads();
  }
}
// From a largest field (stat) to the exponent, 0 for a zero column, kBad; least: smallest exponent whose integers keep
// every bit of the storage type.
__device__ __forceinline__ int exp_of(int s, int bias, int top, int least) {
  if (s == 0) return 0;
  const int e = s - 1 - bias + 1;
  return s - 1 >= top || e < least ? kBad : e;
}
__device__ __forceinline__ int exp_of_z(int s) { return exp_of(s, 1023, 0x7ff, -800); }
// all columns' (one block); bad[0]: whether any column fails, bad[1]: 0
__global__ void k_oz_exp_finish(int *stat, int cols, int bias, int top, int least, int *bad) {
  int any = 0;
  for (int c = threadIdx.x; c < cols; c += blockDim.x) {
    const int e = exp_of(stat[c], bias, top, least);
    stat[c] = e;
    any |= e == kBad;
  }
  any = __syncthreads_or(any);
  if (threadIdx.x == 0) bad[0] = any ? 1 : 0, bad[1] = 0;
}

// sq[m] += 2^32 sum |v|^2 of column m in units of its power of two, lost[m]: entries that lose bits
template <typename T>
__global__ void __launch_bounds__(256)
    k_oz_squares(const T *__restrict__ F, int64_t rows, int cols, const int *__restrict__ ev,
                 unsigned long long *__restrict__ sq, int *__restrict__ lost) {
  __shared__ unsigned long long sum[256];
  __shared__ int number[256];
  for (int c0 = 0; c0 < cols; c0 += 256) {
    const int w = min(256, cols - c0), g = 256 / w;
    const int c = threadIdx.x % w, r = threadIdx.x / w;
    sum[threadIdx.x] = 0;
    number[threadIdx.x] = 0;
    __syncthreads();
    if (r < g) {
      const int e = ev[c0 + c];
      float s = 0.f;
      int n = 0;
      for (int64_t i = (int64_t)blockIdx.x * g + r; i < rows; i += (int64_t)gridDim.x * g) {
        const T v = F[i * cols + c0 + c];
        const float2 u = scaled(v, e);
        s = fmaf(u.x, u.x, fmaf(u.y, u.y, s));
        n += loses_bits(v, e);
      }
      atomicAdd(&sum[c], (unsigned long long)(s * 4294967296.f));
      if (n) atomicAdd(&number[c], n);
    }
    __syncthreads();
    if (threadIdx.x < w) {
      atomicAdd(&sq[c0 + threadIdx.x], sum[threadIdx.x]);
      if (number[threadIdx.x]) atomicAdd(&lost[c0 + threadIdx.x], number[threadIdx.x]);
    }
    __syncthreads();
  }
}
// v2[m]: the sum, lost2[m]: largest sum of squares that can meet a rounded entry of v (FP64 spaces: no limit); *lossy: set
// if a column has entries that lose bits
__global__ void k_oz_limits(const unsigned long long *__restrict__ sq, const int *__restrict__ lost, int cols, bool rounded,
                            float *__restrict__ v2, float *__restrict__ lost2, int *lossy) {
  for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < cols; c += gridDim.x * blockDim.x) {
    v2[c] = (float)sq[c] * 0x1p-32f;
    lost2[c] = rounded ? 3e38f : 2.f * (float)lost[c];
    if (lost[c]) *lossy = 1;
  }
}

// ------------------------------------------------------------------- mma
__device__ __forceinline__ void ldsm4(unsigned (&r)[4], unsigned addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void ldsm4t(unsigned (&r)[4], unsigned addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void mma(float (&c)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
               : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// Sums of one 16 x 16 tile of a warp by digit weight: FP32 (exact up to 128 dofs or vectors), then two 64-bit integers
// per output, weights kMinW .. kMinW + 3 and kMinW + 4 .. kMinW + 7.
struct Acc {
  float c[kGrp][2][4];
  long long lo[2][4], hi[2][4];
  __device__ __forceinline__ Acc() {
#pragma unroll
    for (int t = 0; t < 2; ++t)
#pragma unroll
      for (int q = 0; q < 4; ++q) lo[t][q] = hi[t][q] = 0;
    clear();
  }
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int g = 0; g < kGrp; ++g)
#pragma unroll
      for (int t = 0; t < 2; ++t)
#pragma unroll
        for (int q = 0; q < 4; ++q) c[g][t][q] = 0.f;
  }
  __device__ __forceinline__ void flush() {
#pragma unroll
    for (int t = 0; t < 2; ++t)
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        long long l = 0, h = 0;
#pragma unroll
        for (int g = 3; g >= 0; --g) {
          l = l * 256 + __float2int_rn(c[g][t][q]);
          h = h * 256 + __float2int_rn(c[g + 4][t][q]);
        }
        lo[t][q] += l;
        hi[t][q] += h;
      }
    clear();
  }
  // the sum times 2^-(2 kIntBits)
  __device__ __forceinline__ double value(int t, int q) const {
    constexpr double wl = 1.0 / (double)(1ull << 34) / (double)(1ull << 34);  // 2^(8 kMinW - 2 kIntBits)
    return fma((double)hi[t][q], wl * 4294967296.0, (double)lo[t][q] * wl);
  }
};
static_assert(8 * kMinW - 2 * kIntBits == -68 && kGrp == 8, "weights of Acc::value and Acc::flush");

// all digit pairs of one 16-deep step; pa, pb: bytes from one digit plane to the next
template <bool TRANS_A>
__device__ __forceinline__ void step(Acc &s, unsigned a, unsigned pa, unsigned b, unsigned pb, int mask_b) {
  unsigned fb[kDig][4];
#pragma unroll
  for (int j = 0; j < kDig; ++j)
    if (mask_b >> j & 1) ldsm4t(fb[j], b + j * pb);
#pragma unroll
  for (int i = 0; i < kDig; ++i) {
    unsigned fa[4];
    if (TRANS_A)
      ldsm4t(fa, a + i * pa);
    else
      ldsm4(fa, a + i * pa);
#pragma unroll
    for (int j = kDig - 1; j >= 0; --j) {
      if (i + j < kMinW) continue;
      if (!(mask_b >> j & 1)) continue;
      mma(s.c[i + j - kMinW][0], fa, fb[j][0], fb[j][1]);
      mma(s.c[i + j - kMinW][1], fa, fb[j][2], fb[j][3]);
    }
  }
}

// ------------------------------------------------------------------- mass
// largest of |re|, |im| times 2^-e as BF16 bits, rounded down (0 below 2^-126)
__device__ __forceinline__ unsigned mag(float2 v, int e) {
  const unsigned m = max(__float_as_uint(v.x) & 0x7fffffffu, __float_as_uint(v.y) & 0x7fffffffu);
  const int x = (int)(m >> 23), r = x - e;
  return x == 0 || r < 1 ? 0u : (unsigned)r << 7 | (m >> 16 & 0x7fu);
}
__device__ __forceinline__ unsigned mag(double2 v, int e) {
  const unsigned m = max((unsigned)__double2hiint(v.x) & 0x7fffffffu, (unsigned)__double2hiint(v.y) & 0x7fffffffu);
  const int x = (int)(m >> 20), r = x - 896 - e;
  return x == 0 || r < 1 ? 0u : (unsigned)r << 7 | (m >> 13 & 0x7fu);
}
__device__ __forceinline__ unsigned mag(bfc2 v, int e) { return mag(__bfloat1622float2(v), e); }

// mass[m b + j] += 2^16 sum over sites of |v| |z| (moduli as above: a lower bound, so part of the sites may do), z2[j] +=
// sum |z|^2 (an upper bound); the last block compares with T and sets *fail for a pair that falls short.  Sites: every
// step-th (REST = false: here ez still holds k_oz_exp's fields, which the last block turns into exponents, setting *bad),
// or all but these (run if *need is set).  A block: 64 vectors x 16 columns, stages of 4 sites as BF16 in shared memory;
// eight warps of 16 x 8 sums.  Its loads are issued together, past the ends too (on valid entries, not used): one by one
// behind their tests a stage took 8 us instead of 2.
constexpr int kMM = 64, kMJ = 16, kMK = 48;
constexpr int kMAs = (kMM + 8) * 2, kMBs = (kMJ + 8) * 2;  // bytes of a dof row
template <typename VC, bool REST>
__global__ void __launch_bounds__(256)
    k_oz_mass(const VC *__restrict__ Vd, const int *__restrict__ ev, const double2 *__restrict__ Z,
              int *ez, const int *__restrict__ count, int *bad, const int *__restrict__ need, int k, int b, int nsites,
              int step, const float *__restrict__ v2, const float *__restrict__ lost2,
              unsigned long long *__restrict__ mass, unsigned *__restrict__ z2, unsigned *__restrict__ arrived, int *fail) {
  __shared__ __align__(16) unsigned char sm[kMK * (kMAs + kMBs)];
  __shared__ float zsum[8][kMJ];
  __shared__ int last;
  if (REST && (*bad || !*need)) return;  // (settled by the kernel before: the same for all blocks)
  unsigned short *As = (unsigned short *)sm, *Bs = (unsigned short *)(sm + kMK * kMAs);
  const int first = (nsites + step - 1) / step, total = REST ? nsites - first : first;
  const int i0 = (int)((int64_t)total * blockIdx.x / gridDim.x), i1 = (int)((int64_t)total * (blockIdx.x + 1) / gridDim.x);
  const int m0 = blockIdx.y * kMM, j0 = blockIdx.z * kMJ;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int am = threadIdx.x % kMM, ad = threadIdx.x / kMM, bj = threadIdx.x % kMJ, bd = threadIdx.x / kMJ;
  const bool va = m0 + am < k, vb = j0 + bj < b;
  const int ma = va ? m0 + am : k - 1, jb = vb ? j0 + bj : b - 1;
  const int ea = ev[ma], eb = REST ? ez[jb] : exp_of_z(ez[jb]);
  const unsigned base = (unsigned)__cvta_generic_to_shared(sm);
  const unsigned a_addr = base + ((lane >> 4) * 8 + (lane & 7)) * kMAs + ((w & 3) * 16 + (lane >> 3 & 1) * 8) * 2;
  const unsigned b_addr = base + kMK * kMAs + (lane & 15) * kMBs + (w >> 2) * 16;
  float c[4] = {0.f, 0.f, 0.f, 0.f}, zz = 0.f;
  for (int i = i0; i < i1; i += 4) {
    VC a[kMK * kMM / 256];
    double2 z[kMK * kMJ / 256];
#pragma unroll
    for (int u = 0; u < kMK * kMM / 256; ++u) {
      const int d = ad + u * (256 / kMM), q = min(i + d / 12, i1 - 1);
      const int64_t s = REST ? q + q / (step - 1) + 1 : (int64_t)q * step;
      a[u] = Vd[(s * 12 + d % 12) * k + ma];
    }
#pragma unroll
    for (int u = 0; u < kMK * kMJ / 256; ++u) {
      const int d = bd + u * (256 / kMJ), q = min(i + d / 12, i1 - 1);
      const int64_t s = REST ? q + q / (step - 1) + 1 : (int64_t)q * step;
      z[u] = Z[(s * 12 + d % 12) * b + jb];
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < kMK * kMM / 256; ++u) {
      const int d = ad + u * (256 / kMM);
      As[d * (kMAs / 2) + am] = (unsigned short)(va && i + d / 12 < i1 ? mag(a[u], ea) : 0u);
    }
#pragma unroll
    for (int u = 0; u < kMK * kMJ / 256; ++u) {
      const int d = bd + u * (256 / kMJ);
      const unsigned q = vb && i + d / 12 < i1 ? mag(z[u], eb) : 0u;
      Bs[d * (kMBs / 2) + bj] = (unsigned short)q;
      zz = fmaf(__uint_as_float(q << 16), __uint_as_float(q << 16), zz);
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < kMK / 16; ++q) {
      unsigned fa[4], b0, b1;
      ldsm4t(fa, a_addr + q * 16 * kMAs);
      asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];"
                   : "=r"(b0), "=r"(b1) : "r"(b_addr + q * 16 * kMBs));
      mma(c, fa, b0, b1);
    }
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int m = m0 + (w & 3) * 16 + (q >> 1) * 8 + (lane >> 2), j = j0 + (w >> 2) * 8 + (lane & 3) * 2 + (q & 1);
    if (m < k && j < b && c[q] > 0.f) atomicAdd(&mass[(int64_t)m * b + j], (unsigned long long)(c[q] * 65536.f));
  }
  zz += __shfl_xor_sync(0xffffffffu, zz, 16);
  if (lane < 16) zsum[w][lane] = zz;
  __syncthreads();
  if (blockIdx.y == 0 && threadIdx.x < kMJ && j0 + threadIdx.x < b) {
    float s = 0.f;
    for (int q = 0; q < 8; ++q) s += zsum[q][threadIdx.x];
    atomicAdd(&z2[j0 + threadIdx.x], (unsigned)ceilf(2.04f * s));  // |z|^2 is at most twice the larger part's, cut by 2^-7
  }
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(arrived, 1u) == gridDim.x * gridDim.y * gridDim.z - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  int low = 0;
#pragma unroll 4
  for (int e = threadIdx.x; e < k * b; e += 256) {
    const int j = e % b, m = e / b;
    const float n = (float)count[j], met = REST || step == 1 ? (float)__ldcg(&z2[j]) : 2.f * n;
    const float t2 = fminf(0.5f * n, 4.f * (v2[m] + fminf(met, lost2[m]) + 0x1p-13f * n));
    low |= (float)__ldcg(&mass[e]) < 65536.f * sqrtf(t2);
  }
  if (__syncthreads_or(low) && threadIdx.x == 0) *fail = 1;
  if (!REST && threadIdx.x < b) {
    const int e = exp_of_z(ez[threadIdx.x]);
    ez[threadIdx.x] = e;
    if (e == kBad) *bad = 1;
  }
}

// ------------------------------------------------------------ contraction
// partial[((chunk * k + m) * 2 + half) * b + j] = sum over the chunk's sites and the half's spins (upper, lower) of
// conj(V[dof][m]) Z[dof][j].  A block: 32 vectors x 16 columns, one half of the spins, one chunk of sites; stages of 8
// sites (48 dofs) as digit planes in shared memory; eight warps of 16 x 16 real outputs.
constexpr int kOM = 32, kOJ = 16, kOK = 48;                // vectors, columns, dofs of a stage
constexpr int kOAs = (2 * kOM + 8) * 2, kOBs = (2 * kOJ + 8) * 2;  // bytes of a dof row (padded: ldmatrix without conflicts)
constexpr int kOAp = kOK * kOAs, kOBp = kOK * kOBs;        // of a digit plane
constexpr int kOBytes = kDig * (kOAp + kOBp);
template <typename VC>
__global__ void __launch_bounds__(256, 2)
    k_oz_contract(const VC *__restrict__ Vd, const int *__restrict__ ev, const double2 *__restrict__ Z,
                  const int *__restrict__ ez, const int *__restrict__ bad, int k, int b, int nsites, int nchunks,
                  double2 *__restrict__ partial) {
  extern __shared__ __align__(16) unsigned char sm[];
  __shared__ int used[2];  // digits of Z that are not zero, of this stage and (cleared) the next
  if (*bad) return;        // the FP64 kernel runs instead
  if (threadIdx.x < 2) used[threadIdx.x] = 0;
  unsigned *As = (unsigned *)sm, *Bs = (unsigned *)(sm + kDig * kOAp);
  const int half = blockIdx.x & 1, chunk = blockIdx.x >> 1;
  const int m0 = blockIdx.y * kOM, j0 = blockIdx.z * kOJ;
  const int s0 = (int)(((int64_t)nsites * chunk) / nchunks), s1 = (int)(((int64_t)nsites * (chunk + 1)) / nchunks);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int am = threadIdx.x % kOM, ad = threadIdx.x / kOM;  // this thread's vector, first dof
  const int bj = threadIdx.x % kOJ, bd = threadIdx.x / kOJ;
  const int ea = m0 + am < k ? ev[m0 + am] : 0, eb = j0 + bj < b ? ez[j0 + bj] : 0;
  const unsigned base = (unsigned)__cvta_generic_to_shared(sm);
  // ldmatrix rows: A planes [dof][2 m + c], B planes [dof][2 j + d], both read transposed
  const unsigned a_addr = base + ((lane >> 4) * 8 + (lane & 7)) * kOAs + ((w & 3) * 16 + (lane >> 3 & 1) * 8) * 2;
  const unsigned b_addr =
      base + kDig * kOAp + ((lane >> 3 & 1) * 8 + (lane & 7)) * kOBs + ((w >> 2) * 16 + (lane >> 4) * 8) * 2;
  Acc acc;
  int stage = 0;
  for (int s = s0; s < s1; s += 8, ++stage) {
    __syncthreads();
    // stage the digits: dof row d = 6 * site + spin-colour of this half
#pragma unroll
    for (int u = 0; u < kOK * kOM / 256; ++u) {
      const int d = ad + u * (256 / kOM), st = s + d / 6;
      Dig2 g{kNoDig, kNoDig};
      if (st < s1 && m0 + am < k) g = dig(Vd[((int64_t)st * 12 + half * 6 + d % 6) * k + m0 + am], ea);
#pragma unroll
      for (int i = 0; i < kDig; ++i) As[(i * kOAp + d * kOAs) / 4 + am] = digit_pair(g, i);
    }
    int mask = 0;
#pragma unroll
    for (int u = 0; u < kOK * kOJ / 256; ++u) {
      const int d = bd + u * (256 / kOJ), st = s + d / 6;
      Dig2 g{kNoDig, kNoDig};
      if (st < s1 && j0 + bj < b) g = dig(Z[((int64_t)st * 12 + half * 6 + d % 6) * b + j0 + bj], eb);
      mask |= digit_mask(g);
#pragma unroll
      for (int i = 0; i < kDig; ++i) Bs[(i * kOBp + d * kOBs) / 4 + bj] = digit_pair(g, i);
    }
    mask = __reduce_or_sync(0xffffffffu, (unsigned)mask);
    if (lane == 0 && mask) atomicOr(&used[stage & 1], mask);
    __syncthreads();
    mask = used[stage & 1];
    if (threadIdx.x == 0) used[(stage + 1) & 1] = 0;
#pragma unroll
    for (int q = 0; q < kOK / 16; ++q)
      step<true>(acc, a_addr + q * 16 * kOAs, kOAp, b_addr + q * 16 * kOBs, kOBp, mask);
    if (stage & 1) acc.flush();  // 96 dofs
  }
  acc.flush();
  // rows 2 m + c sit in lanes 4 apart, columns 2 j, 2 j + 1 in one thread: C = (D00 + D11) + i (D01 - D10)
#pragma unroll
  for (int t = 0; t < 2; ++t)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const double x = acc.value(t, 2 * h), y = acc.value(t, 2 * h + 1);
      const double ox = __shfl_xor_sync(0xffffffffu, x, 4), oy = __shfl_xor_sync(0xffffffffu, y, 4);
      const int row = (w & 3) * 16 + h * 8 + (lane >> 2), col = (w >> 2) * 16 + t * 8 + (lane & 3) * 2;
      const int m = m0 + (row >> 1), j = j0 + (col >> 1);
      if (!(row & 1) && m < k && j < b) {
        const int e = ev[m] + ez[j];
        partial[(((int64_t)chunk * k + m) * 2 + half) * b + j] =
            make_double2(scalbn(x + oy, e), scalbn(y - ox, e));
      }
    }
}

// -------------------------------------------------------------- expansion
// Digit planes of the weights for x0 = V W: Wd[i][2 m + c][2 j + d] as BF16, from W[m][j] 2^ev[m], with rows (Re, Im) of
// V's entry against columns (Re, Im) of x0: (Wr, Wi; -Wi, Wr); ew[j]: exponent of column j, kZero if it is zero; one
// block a column.  least[j]: smallest sum of squares of 16 entries (in the weights' units) for the digits to do, 16 times
// 2^100 the mean square error of an entry: 2/3 2^-110 of the sum of the weights' squares where V is rounded, and, as
// 2^-123 k, the dropped pairs (2^-62 sqrt(2 k)).
__global__ void __launch_bounds__(256) k_oz_weights(const double2 *__restrict__ W, const int *__restrict__ ev, int k,
                                                    int b, bool rounded, unsigned *__restrict__ Wd, int *__restrict__ ew,
                                                    float *__restrict__ least, int *bad) {
  __shared__ int emax, nz;
  __shared__ float sh[256];
  const int j = blockIdx.x;
  if (threadIdx.x == 0) emax = -(1 << 20), nz = 0;
  __syncthreads();
  for (int m = threadIdx.x; m < k; m += 256) {
    const double2 v = W[(int64_t)j * k + m];
    if (is_zero(v)) continue;
    const int f = exp_field(v);
    atomicMax(&emax, f == 0x7ff ? kBad : f - 1022 + ev[m]);
    nz = 1;
  }
  __syncthreads();
  const int e = nz ? emax : 0;
  if (threadIdx.x == 0) {
    ew[j] = nz ? e : kZero;
    if (e > 800 || e < -800) *bad = 1;  // not finite, or out of the integers' reach
  }
  const int64_t plane = (int64_t)2 * k * b;  // 32-bit pairs of a digit plane
  float w2 = 0.f;
  for (int m = threadIdx.x; m < k; m += 256) {
    const double2 v = W[(int64_t)j * k + m];
    const float re = f64_to_f32(scalbn(v.x, ev[m] - e)), im = f64_to_f32(scalbn(v.y, ev[m] - e));
    w2 = fmaf(re, re, fmaf(im, im, w2));
    const Dig2 d = dig(v, e - ev[m]), n = dig(make_double2(-v.y, v.x), e - ev[m]);
#pragma unroll
    for (int i = 0; i < kDig; ++i) {
      Wd[i * plane + (int64_t)(2 * m) * b + j] = digit_pair(d, i);
      Wd[i * plane + (int64_t)(2 * m + 1) * b + j] = digit_pair(n, i);
    }
  }
  sh[threadIdx.x] = w2;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if ((int)threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) least[j] = 16.f * ((rounded ? (2.f / 3.f) * 0x1p-10f * sh[0] : 0.f) + 0x1p-23f * (float)k);
}

// x[dof][j] = sum_m V[dof][m] W[m][j]: a block takes 64 dofs x 16 columns, 32 vectors (64 rows of Wd) a stage.
// *small is set where 16 dofs of a column have squares below the column's `least` in sum (in the weights' units), with an
// allowance for the FP32 and BF16 entries of the tile that lose bits (2/3 2^-110 each, for weights of at most one unit).
// LOSSY: the space has such entries (Gaussian FP32 ones from about 10^8 entries on).
constexpr int kXD = 64, kXM = 32;
constexpr int kXAs = (2 * kXM + 8) * 2, kXBs = (2 * kOJ + 8) * 2;
constexpr int kXAp = kXD * kXAs, kXBp = 2 * kXM * kXBs;
constexpr int kXBytes = kDig * (kXAp + kXBp);
template <typename VC, bool LOSSY>
__global__ void __launch_bounds__(256, 2)
    k_oz_expand(const VC *__restrict__ Vd, const int *__restrict__ ev, const unsigned *__restrict__ Wd,
                const int *__restrict__ ew, const int *__restrict__ bad, int k, int b, int64_t N,
                const float *__restrict__ least, int *small, double2 *__restrict__ x) {
  extern __shared__ __align__(16) unsigned char sm[];
  __shared__ int lost[2];  // entries that lose bits, of this tile and (cleared) the next
  if (*bad) return;        // the FP64 kernel runs instead
  if (LOSSY && threadIdx.x < 2) lost[threadIdx.x] = 0;
  unsigned *As = (unsigned *)sm, *Bs = (unsigned *)(sm + kDig * kXAp);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int j0 = blockIdx.y * kOJ;
  const int am = threadIdx.x % kXM, ad = threadIdx.x / kXM;
  const unsigned base = (unsigned)__cvta_generic_to_shared(sm);
  // A planes [dof][2 m + c] read as they lie, B planes [2 m + c][2 j + d] transposed
  const unsigned a_addr = base + ((w & 3) * 16 + (lane & 15)) * kXAs + (lane >> 4) * 16;
  const unsigned b_addr =
      base + kDig * kXAp + ((lane >> 3 & 1) * 8 + (lane & 7)) * kXBs + ((w >> 2) * 16 + (lane >> 4) * 8) * 2;
  const int64_t plane = (int64_t)2 * k * b;
  const int64_t tiles = (N + kXD - 1) / kXD;
  const bool one = k <= kXM;  // the weights of all vectors stay in shared memory
  int turn = 0;
  for (int64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x, turn ^= 1) {
    const int64_t i0 = tile * kXD;
    Acc acc;
    int stage = 0;
    for (int m0 = 0; m0 < k; m0 += kXM, ++stage) {
      __syncthreads();
      if (LOSSY && m0 == 0 && threadIdx.x == 0) lost[turn ^ 1] = 0;
      int mine = 0;
#pragma unroll
      for (int u = 0; u < kXD * kXM / 256; ++u) {
        const int d = ad + u * (256 / kXM);
        Dig2 g{kNoDig, kNoDig};
        if (i0 + d < N && m0 + am < k) {
          const VC v = Vd[(i0 + d) * k + m0 + am];
          g = dig(v, ev[m0 + am]);
          if (LOSSY) mine += loses_bits(v, ev[m0 + am]);
        }
#pragma unroll
        for (int i = 0; i < kDig; ++i) As[(i * kXAp + d * kXAs) / 4 + am] = digit_pair(g, i);
      }
      if (LOSSY && mine) atomicAdd(&lost[turn], mine);
      if (!one || tile == blockIdx.x) {
        for (int q = threadIdx.x; q < kDig * 2 * kXM * kOJ; q += 256) {
          const int j = q % kOJ, r = q / kOJ % (2 * kXM), i = q / (kOJ * 2 * kXM);
          Bs[(i * kXBp + r * kXBs) / 4 + j] =
              2 * m0 + r < 2 * k && j0 + j < b ? Wd[i * plane + (int64_t)(2 * m0 + r) * b + j0 + j] : 0u;
        }
      }
      __syncthreads();
#pragma unroll
      for (int q = 0; q < 2 * kXM / 16; ++q)
        step<false>(acc, a_addr + q * 32, kXAp, b_addr + q * 16 * kXBs, kXBp, (1 << kDig) - 1);
      if (stage & 1) acc.flush();  // 128 terms
    }
    acc.flush();
    const float allow = LOSSY ? (2.f / 3.f) * 0x1p-10f * 16.f / kXD * (float)lost[turn] : 0.f;
#pragma unroll
    for (int t = 0; t < 2; ++t) {
      const int j = j0 + ((w >> 2) * 16 + t * 8 + (lane & 3) * 2) / 2;
      const int e = j < b ? ew[j] : kZero;
      float sq = 0.f;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int64_t i = i0 + (w & 3) * 16 + h * 8 + (lane >> 2);
        const double re = acc.value(t, 2 * h), im = acc.value(t, 2 * h + 1);
        const float fr = f64_to_f32(re), fi = f64_to_f32(im);
        sq = fmaf(fr, fr, fmaf(fi, fi, sq));
        if (i < N && j < b) x[i * b + j] = make_double2(scalbn(re, e), scalbn(im, e));
      }
#pragma unroll
      for (int o = 4; o < 32; o <<= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
      // (a warp's 16 dofs are all below N or none: N is a multiple of 192)
      if (e != kZero && i0 + (w & 3) * 16 < N && sq < least[j] + allow) *small = 1;
    }
  }
}

// --------------------------------------------------------------- launchers
// per-vector exponents of a deflation space into D->vexp, and what the mass test needs of it behind them
size_t defl_oz_space_bytes(int k) { return 3 * (size_t)k * sizeof(int); }
static float *space_v2(const dtr_defl_s *D) { return (float *)(D->vexp + D->k); }
static float *space_lost2(const dtr_defl_s *D) { return (float *)(D->vexp + 2 * (size_t)D->k); }
int defl_oz_setup(const dtr_defl_s *D, void *scratch, int *bad, cudaStream_t st) {
  const int k = D->k;
  const int64_t N = D->lat.N;
  unsigned long long *sq = (unsigned long long *)scratch;
  int *lost = (int *)(sq + k);
  DTR_CUDA(cudaMemsetAsync(D->vexp, 0, k * sizeof(int), st));
  DTR_CUDA(cudaMemsetAsync(scratch, 0, k * (sizeof(*sq) + sizeof(int)), st));
  const unsigned grid = (unsigned)(8 * device_sms());
  // (an FP32 entry is exact down to 2^-31 of its column's largest; with an exponent of at least -60 subnormals are below)
  if (D->prec == DTR_F64) {
    k_oz_exp<double2><<<grid, 256, 0, st>>>((const double2 *)D->V, N, k, D->vexp, nullptr);
    k_oz_exp_finish<<<1, 256, 0, st>>>(D->vexp, k, 1023, 0x7ff, -800, bad);
    k_oz_squares<double2><<<grid, 256, 0, st>>>((const double2 *)D->V, N, k, D->vexp, sq, lost);
  } else if (D->prec == DTR_F32) {
    k_oz_exp<float2><<<grid, 256, 0, st>>>((const float2 *)D->V, N, k, D->vexp, nullptr);
    k_oz_exp_finish<<<1, 256, 0, st>>>(D->vexp, k, 127, 0xff, -60, bad);
    k_oz_squares<float2><<<grid, 256, 0, st>>>((const float2 *)D->V, N, k, D->vexp, sq, lost);
  } else {
    k_oz_exp<bfc2><<<grid, 256, 0, st>>>((const bfc2 *)D->V, N, k, D->vexp, nullptr);
    k_oz_exp_finish<<<1, 256, 0, st>>>(D->vexp, k, 127, 0xff, -60, bad);
    k_oz_squares<bfc2><<<grid, 256, 0, st>>>((const bfc2 *)D->V, N, k, D->vexp, sq, lost);
  }
  k_oz_limits<<<(unsigned)((k + 255) / 256), 256, 0, st>>>(sq, lost, k, D->prec == DTR_F64, space_v2(D), space_lost2(D),
                                                           bad + 1);
  count_launches(4);
  return DTR_OK;
}

// scratch in ints: [kBadC] and [kBadX], one pair of flags (the second found while the digits run) that send the
// contraction or the expansion to the FP64 kernel; [kNeed] the sampled mass fell short, [kArrived] two block counters,
// [kEz] exponents of Z's columns, [kCount] their nonzero entries, [kZ2] (in the contraction) their sums of squares, [kEw]
// (in the expansion, in the same place) exponents of the weights' columns, [kLeast] (in the expansion, in the counts' place)
// least squares of x0's columns, [kMass] masses (64 bits, k b), behind them the weights' digit planes
constexpr int kBadC = 0, kBadX = 2, kNeed = 4, kArrived = 5, kEz = 64, kCount = 128, kLeast = 128, kZ2 = 192, kEw = 192, kMass = 256;
static size_t planes_at(int k, int b) { return kMass + (size_t)2 * k * b; }
size_t defl_oz_scratch_bytes(int k, int b) {
  return (planes_at(k, b) + (size_t)kDig * 2 * k * b) * sizeof(int);
}
const int *defl_oz_contract_flags(const void *scratch) { return (const int *)scratch + kBadC; }
const int *defl_oz_expand_flags(const void *scratch) { return (const int *)scratch + kBadX; }

template <typename K> static int allow_smem(K kern, int bytes) {
  DTR_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
  return DTR_OK;
}

// Mass test: on part of the sites first, where Gaussian columns pass with a factor of 5 (at 16^3 x 32 a sixth of them in an
// FP64 space, whose entries are all rounded, and a twelfth else), and on the rest if that falls short.
template <typename VC> static int mass_t(const dtr_defl_s *D, const double2 *Z, int b, int *sc, cudaStream_t st) {
  const int V = (int)D->lat.V, k = D->k;
  int step = (int)(std::sqrt((double)D->lat.N) / (D->prec == DTR_F64 ? 200.0 : 100.0));
  step = step < 1 ? 1 : step > 64 ? 64 : step;
  const int tiles = ((k + kMM - 1) / kMM) * ((b + kMJ - 1) / kMJ);
  auto grid = [&](int sites) {
    int n = (4 * device_sms() + tiles - 1) / tiles;
    if (n > (sites + 3) / 4) n = (sites + 3) / 4;
    return dim3(n < 1 ? 1 : n, (k + kMM - 1) / kMM, (b + kMJ - 1) / kMJ);
  };
  unsigned long long *mass = (unsigned long long *)(sc + kMass);
  k_oz_mass<VC, false><<<grid((V + step - 1) / step), 256, 0, st>>>(
      (const VC *)D->V, D->vexp, Z, sc + kEz, sc + kCount, sc + kBadC, sc + kNeed, k, b, V, step, space_v2(D),
      space_lost2(D), mass, (unsigned *)sc + kZ2, (unsigned *)sc + kArrived, sc + (step > 1 ? kNeed : kBadC));
  count_launches(1);
  if (step > 1) {
    k_oz_mass<VC, true><<<grid(V - V / step), 256, 0, st>>>((const VC *)D->V, D->vexp, Z, sc + kEz, sc + kCount, sc + kBadC,
                                                            sc + kNeed, k, b, V, step, space_v2(D), space_lost2(D), mass,
                                                            (unsigned *)sc + kZ2, (unsigned *)sc + kArrived + 1,
                                                            sc + kBadC);
    count_launches(1);
  }
  DTR_LAUNCH_CHECK("digit mass");
  return DTR_OK;
}

template <typename VC>
static int contract_t(const dtr_defl_s *D, const double2 *Z, int b, int *sc, int nch, double2 *partial,
                      cudaStream_t st) {
  int rc = allow_smem(k_oz_contract<VC>, kOBytes);
  if (!rc) rc = mass_t<VC>(D, Z, b, sc, st);
  if (rc) return rc;
  const dim3 grid(2 * nch, (D->k + kOM - 1) / kOM, (b + kOJ - 1) / kOJ);
  k_oz_contract<VC><<<grid, 256, kOBytes, st>>>((const VC *)D->V, D->vexp, Z, sc + kEz, sc + kBadC, D->k, b,
                                               (int)D->lat.V, nch, partial);
  count_launches(1);
  return DTR_OK;
}
int defl_oz_contract(const dtr_defl_s *D, const double2 *Z, int b, void *scratch, int max_chunks, double2 *partial,
                     int *chunks, cudaStream_t st) {
  int *sc = (int *)scratch;
  const int V = (int)D->lat.V, sms = device_sms();
  DTR_CUDA(cudaMemsetAsync(sc, 0, planes_at(D->k, b) * sizeof(int), st));
  k_oz_exp<double2><<<(unsigned)(8 * sms), 256, 0, st>>>(Z, (int64_t)V * 12, b, sc + kEz, sc + kCount);
  count_launches(1);
  const int tiles = 2 * ((D->k + kOM - 1) / kOM) * ((b + kOJ - 1) / kOJ);
  int nch = (4 * sms + tiles - 1) / tiles;  // about two rounds of two blocks to an SM
  if (nch > V / 16) nch = V / 16 > 0 ? V / 16 : 1;
  if (nch > max_chunks) nch = max_chunks;
  *chunks = nch;
  if (D->prec == DTR_F64) return contract_t<double2>(D, Z, b, sc, nch, partial, st);
  if (D->prec == DTR_F32) return contract_t<float2>(D, Z, b, sc, nch, partial, st);
  return contract_t<bfc2>(D, Z, b, sc, nch, partial, st);
}

template <typename VC, bool LOSSY>
static int expand_t(const dtr_defl_s *D, int b, int *sc, double2 *x, cudaStream_t st) {
  int rc = allow_smem(k_oz_expand<VC, LOSSY>, kXBytes);
  if (rc) return rc;
  const int64_t N = D->lat.N, tiles = (N + kXD - 1) / kXD;
  const int nj = (b + kOJ - 1) / kOJ;
  int64_t gx = 2 * device_sms() / nj;
  if (gx < 1) gx = 1;
  if (gx > tiles) gx = tiles;
  k_oz_expand<VC, LOSSY><<<dim3((unsigned)gx, nj), 256, kXBytes, st>>>(
      (const VC *)D->V, D->vexp, (const unsigned *)(sc + planes_at(D->k, b)), sc + kEw, sc + kBadX, D->k, b, N,
      (const float *)(sc + kLeast), sc + kBadX + 1, x);
  count_launches(1);
  return DTR_OK;
}
int defl_oz_expand(const dtr_defl_s *D, const double2 *W, int b, void *scratch, double2 *x, cudaStream_t st) {
  int *sc = (int *)scratch;
  DTR_CUDA(cudaMemsetAsync(sc + kBadX, 0, 2 * sizeof(int), st));
  k_oz_weights<<<b, 256, 0, st>>>(W, D->vexp, D->k, b, D->prec == DTR_F64, (unsigned *)(sc + planes_at(D->k, b)),
                                  sc + kEw, (float *)(sc + kLeast), sc + kBadX);
  count_launches(1);
  if (D->prec == DTR_F64) return expand_t<double2, false>(D, b, sc, x, st);
  if (D->prec == DTR_F32)
    return D->vlossy ? expand_t<float2, true>(D, b, sc, x, st) : expand_t<float2, false>(D, b, sc, x, st);
  return D->vlossy ? expand_t<bfc2, true>(D, b, sc, x, st) : expand_t<bfc2, false>(D, b, sc, x, st);
}

}  // namespace dtr
