// Jacobi sweeps of Eq. 1, S <- C Q S Q^T + (1 - C) I, on a symmetric S held
// in 64-bit fixed point (value * 2^60), as two products per sweep:
//   T = (C Q S)^T,   S' = Q T,   with S' + (1 - C) I on the diagonal.
//
// What bounds a sweep is the gather of one row segment per edge.  In FP64 it
// was bound by the FP64 pipe instead (GB300 issues FP64 at 1/64 of the FP32
// rate): the adds ran at 0.5 values a clock and SM.  Here the row sums are
// exact integer sums (96 bits), and the division by the in-degree is a product
// with a 64-bit reciprocal, rounded once: an error below 2^-60 a product,
// where FP64 sums of d values of size s lose up to d 2^-53 s.
//
// Work split: a CTA takes 64 rows x 64 columns, a warp one row at a time with
// two adjacent columns per lane (512-byte row segments).  CTAs of one column
// slab (64 columns of all rows, n * 512 bytes: 10 MB at n = 20,000) run next to
// each other, so the gathers stay in L2 and the rows of nodes with many
// out-neighbours in L1.  A row of more than LONG_ROW nonzeros is gathered by
// the whole CTA.  The first product is written transposed through shared
// memory; of the second only the tiles on or above the diagonal are formed
// (S' is symmetric), written together with their mirrors and compared with
// the old S for the stopping test.
#include "sr_internal.h"

namespace sr {

namespace {

constexpr int SB = 64;         // rows and columns of a CTA's tile
constexpr int LONG_ROW = 96;   // longer rows are gathered by the whole CTA

// 96-bit two's-complement sum
struct Acc96 {
  uint32_t w0, w1, w2;
};
__device__ __forceinline__ void acc_add(Acc96& a, long long v) {
  const uint32_t lo = (uint32_t)(unsigned long long)v;
  const uint32_t hi = (uint32_t)((unsigned long long)v >> 32);
  const uint32_t sx = (uint32_t)((int32_t)hi >> 31);
  asm("add.cc.u32 %0, %0, %3;\n\taddc.cc.u32 %1, %1, %4;\n\taddc.u32 %2, %2, %5;"
      : "+r"(a.w0), "+r"(a.w1), "+r"(a.w2)
      : "r"(lo), "r"(hi), "r"(sx));
}
__device__ __forceinline__ void acc_add(Acc96& a, const Acc96& b) {
  asm("add.cc.u32 %0, %0, %3;\n\taddc.cc.u32 %1, %1, %4;\n\taddc.u32 %2, %2, %5;"
      : "+r"(a.w0), "+r"(a.w1), "+r"(a.w2)
      : "r"(b.w0), "r"(b.w1), "r"(b.w2));
}

// The sum times r.r * 2^-(64 + r.s), rounded to nearest (r.r = 0: times one)
__device__ __forceinline__ long long acc_scale(const Acc96& a, const SweepScale& r) {
  const bool neg = (int32_t)a.w2 < 0;
  unsigned long long lo = ((unsigned long long)a.w1 << 32) | a.w0;
  uint32_t hi = a.w2;
  if (neg) {
    lo = ~lo + 1ull;
    hi = ~hi + (lo == 0ull ? 1u : 0u);
  }
  if (r.r == 0ull) return neg ? -(long long)lo : (long long)lo;
  unsigned __int128 t = (unsigned __int128)hi * r.r + __umul64hi(lo, r.r);
  t += r.s ? ((unsigned __int128)1 << (r.s - 1)) : (unsigned __int128)((lo * r.r) >> 63);
  const long long v = (long long)(t >> r.s);
  return neg ? -v : v;
}

// Sums over the nonzeros [e0, e1) of a row (pool offset st) of the columns
// c, c + 1 of X; every lane of the warp takes part.  |value| < 1.875 * 2^60, so
// four values add in 64 bits.
__device__ __forceinline__ void sweep_gather(const int32_t* __restrict__ col, int64_t st, int e0,
                                             int e1, const long long* __restrict__ X, int64_t ld,
                                             int64_t c, Acc96& s0, Acc96& s1) {
  const int lane = threadIdx.x & 31;
  for (int b = e0; b < e1; b += 32) {
    const int m = min(32, e1 - b);
    const int id = lane < m ? __ldg(col + st + b + lane) : 0;
    for (int u = 0; u < m; u += 4) {
      longlong2 v[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int64_t x = __shfl_sync(0xffffffffu, id, u + k);
        v[k] = make_longlong2(0, 0);
        if (u + k < m) v[k] = *reinterpret_cast<const longlong2*>(X + x * ld + c);
      }
      acc_add(s0, (v[0].x + v[1].x) + (v[2].x + v[3].x));
      acc_add(s1, (v[0].y + v[1].y) + (v[2].y + v[3].y));
    }
  }
}

template <bool SECOND>
__global__ void __launch_bounds__(256) k_sweep(DevAdj in, const SweepScale* __restrict__ scales,
                                               const long long* __restrict__ X, int64_t ld,
                                               long long* __restrict__ Y,
                                               const long long* __restrict__ Sold,
                                               long long diag, int n_diag,
                                               unsigned long long* __restrict__ maxd) {
  __shared__ long long tile[SB][SB + 1];
  __shared__ Acc96 part[8][SB];
  __shared__ int longs[SB];
  __shared__ int n_long;
  __shared__ unsigned long long wmax[8];
  const int I = blockIdx.x, J = blockIdx.y;
  if (SECOND && I > J) return;  // the whole CTA
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t row0 = (int64_t)I * SB, col0 = (int64_t)J * SB;
  const int64_t c = col0 + 2 * lane;
  if (threadIdx.x == 0) n_long = 0;
  __syncthreads();
  for (int i = 0; i < SB / 8; ++i) {
    const int r = warp * (SB / 8) + i;
    const int64_t a = row0 + r;
    const int len = in.len[a];
    if (len > LONG_ROW) {
      if (lane == 0) longs[atomicAdd(&n_long, 1)] = r;
      continue;
    }
    Acc96 s0 = {0u, 0u, 0u}, s1 = {0u, 0u, 0u};
    if (len > 0) {
      sweep_gather(in.col, in.start[a], 0, len, X, ld, c, s0, s1);
      const SweepScale sc = scales[a];
      tile[r][2 * lane] = acc_scale(s0, sc);
      tile[r][2 * lane + 1] = acc_scale(s1, sc);
    } else {
      tile[r][2 * lane] = 0;
      tile[r][2 * lane + 1] = 0;
    }
  }
  __syncthreads();
  const int nl = n_long;
  for (int q = 0; q < nl; ++q) {
    const int r = longs[q];
    const int64_t a = row0 + r;
    const int len = in.len[a];
    const int per = ((len + 7) / 8 + 3) & ~3;
    Acc96 s0 = {0u, 0u, 0u}, s1 = {0u, 0u, 0u};
    sweep_gather(in.col, in.start[a], min(len, warp * per), min(len, (warp + 1) * per), X, ld, c,
                 s0, s1);
    part[warp][2 * lane] = s0;
    part[warp][2 * lane + 1] = s1;
    __syncthreads();
    if (threadIdx.x < SB) {
      Acc96 s = part[0][threadIdx.x];
#pragma unroll
      for (int w = 1; w < 8; ++w) acc_add(s, part[w][threadIdx.x]);
      tile[r][threadIdx.x] = acc_scale(s, scales[a]);
    }
    __syncthreads();
  }
  if (!SECOND) {
    for (int k = warp; k < SB; k += 8) {
      long long* y = Y + (col0 + k) * ld + row0;
      y[lane] = tile[lane][k];
      y[lane + 32] = tile[lane + 32][k];
    }
    return;
  }
  if (I == J) {
    if (threadIdx.x < SB && row0 + threadIdx.x < n_diag) tile[threadIdx.x][threadIdx.x] += diag;
    __syncthreads();
    // one of the two roundings of a pair of mirrored entries for both
    for (int r = warp; r < SB; r += 8)
      for (int k = lane; k < r; k += 32) tile[r][k] = tile[k][r];
    __syncthreads();
  }
  unsigned long long m = 0;
  for (int r = warp; r < SB; r += 8) {
    long long* y = Y + (row0 + r) * ld + col0;
    const long long* o = Sold + (row0 + r) * ld + col0;
#pragma unroll
    for (int h = 0; h < SB; h += 32) {
      const long long v = tile[r][h + lane];
      const long long d = v - o[h + lane];
      m = max(m, (unsigned long long)(d < 0 ? -d : d));
      y[h + lane] = v;
    }
  }
  if (I != J)
    for (int k = warp; k < SB; k += 8) {
      long long* y = Y + (col0 + k) * ld + row0;
      y[lane] = tile[lane][k];
      y[lane + 32] = tile[lane + 32][k];
    }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (lane == 0) wmax[warp] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
#pragma unroll
    for (int w = 1; w < 8; ++w) m = max(m, wmax[w]);
    // most tiles change less than one seen already
    if (m > *(volatile unsigned long long*)maxd) atomicMax(maxd, m);
  }
}

// What the fixed-point form cannot take: *flags |= 1 for an entry of
// magnitude 1.875 or more (or a NaN), 2 for a pair of mirrored entries further
// apart than tol.  One CTA per pair of 32 x 32 blocks.
template <typename T>
__global__ void k_sweep_check(const T* __restrict__ S, int64_t ld, double tol,
                              unsigned int* __restrict__ flags) {
  const int bi = blockIdx.y, bj = blockIdx.x;
  if (bj < bi) return;
  __shared__ T t2[32][33];
  for (int r = threadIdx.y; r < 32; r += 8)
    t2[r][threadIdx.x] = S[(int64_t)(bj * 32 + r) * ld + bi * 32 + threadIdx.x];
  __syncthreads();
  unsigned int f = 0;
  for (int r = threadIdx.y; r < 32; r += 8) {
    const T x = S[(int64_t)(bi * 32 + r) * ld + bj * 32 + threadIdx.x];
    const T y = t2[threadIdx.x][r];
    if (!(fabs(x) < T(1.875)) || !(fabs(y) < T(1.875))) f |= 1u;
    if (!(fabs(x - y) <= (T)tol)) f |= 2u;
  }
  f = __reduce_or_sync(0xffffffffu, f);
  if (threadIdx.x == 0 && f) atomicOr(flags, f);
}

// x * 2^59 rounded to nearest (half away from zero), |x| < 2, on the integer
// pipe: a conversion from or to a 64-bit type issues at the FP64 rate
__device__ __forceinline__ long long fixed59(uint64_t mant, int sh, bool neg) {
  long long v = 0;
  if (sh >= 0)
    v = (long long)(mant << sh);
  else if (sh > -60)
    v = (long long)((mant + (1ull << (-sh - 1))) >> -sh);
  return neg ? -v : v;
}
__device__ __forceinline__ long long to_fixed59(float x) {
  const uint32_t b = __float_as_uint(x);
  const int e = (int)((b >> 23) & 0xffu);
  if (e == 0) return 0;  // below 2^-126
  return fixed59((b & 0x7fffffu) | 0x800000u, e - 127 - 23 + 59, (b >> 31) != 0);
}
__device__ __forceinline__ long long to_fixed59(double x) {
  const uint64_t b = (uint64_t)__double_as_longlong(x);
  const int e = (int)((b >> 52) & 0x7ffu);
  if (e == 0) return 0;
  return fixed59((b & 0xfffffffffffffull) | 0x10000000000000ull, e - 1023 - 52 + 59,
                 (b >> 63) != 0);
}
// v * 2^-60 rounded to nearest even
template <typename T>
__device__ __forceinline__ T from_fixed60(long long v) {
  if (v == 0) return T(0);
  const uint64_t a = v < 0 ? (uint64_t)-v : (uint64_t)v;
  const int lz = __clzll((long long)a);
  const uint64_t m = a << lz;
  constexpr int DROP = sizeof(T) == 4 ? 40 : 11;
  const uint64_t rem = m & ((1ull << DROP) - 1), half = 1ull << (DROP - 1);
  uint64_t q = m >> DROP;  // leading one included
  q += (rem > half || (rem == half && (q & 1))) ? 1 : 0;
  const int e = 63 - lz - 60;
  // adding the significand with its leading one carries into the exponent
  if constexpr (sizeof(T) == 4)
    return __uint_as_float((((uint32_t)(e + 126) << 23) + (uint32_t)q) |
                           (v < 0 ? 0x80000000u : 0u));
  else
    return __longlong_as_double((long long)((((uint64_t)(e + 1022) << 52) + q) |
                                            (v < 0 ? 0x8000000000000000ull : 0ull)));
}

// The mean of each pair of mirrored entries in fixed point, both places
// (S and F may be the same memory: a CTA reads its two blocks, then writes them)
template <typename T>
__global__ void k_to_fixed(const T* S, long long* F, int64_t ld) {
  const int bi = blockIdx.y, bj = blockIdx.x;
  if (bj < bi) return;
  __shared__ long long t1[32][33], t2[32][33];
  // value * 2^59: the sum of the two is their mean * 2^60
  for (int r = threadIdx.y; r < 32; r += 8) {
    t1[r][threadIdx.x] = to_fixed59(S[(int64_t)(bi * 32 + r) * ld + bj * 32 + threadIdx.x]);
    t2[r][threadIdx.x] = to_fixed59(S[(int64_t)(bj * 32 + r) * ld + bi * 32 + threadIdx.x]);
  }
  __syncthreads();
  for (int r = threadIdx.y; r < 32; r += 8) {
    F[(int64_t)(bi * 32 + r) * ld + bj * 32 + threadIdx.x] =
        t1[r][threadIdx.x] + t2[threadIdx.x][r];
    if (bi != bj)
      F[(int64_t)(bj * 32 + r) * ld + bi * 32 + threadIdx.x] =
          t2[r][threadIdx.x] + t1[threadIdx.x][r];
  }
}

// S = F * 2^-60, rounded once (S and F may be the same memory)
template <typename T>
__global__ void k_from_fixed(const long long* F, T* S, int64_t count) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < count;
       e += (int64_t)gridDim.x * blockDim.x)
    S[e] = from_fixed60<T>(F[e]);
}

}  // namespace

void launch_sweep_fixed(const DevAdj& in, const SweepScale* s1, const SweepScale* s2,
                        const long long* S, int64_t ld, int n_pad, long long* T, long long* Snew,
                        long long diag, int n_diag, unsigned long long* maxd, cudaStream_t st) {
  const dim3 grid(n_pad / SB, n_pad / SB);
  k_sweep<false><<<grid, 256, 0, st>>>(in, s1, S, ld, T, nullptr, 0, 0, nullptr);
  k_sweep<true><<<grid, 256, 0, st>>>(in, s2, T, ld, Snew, S, diag, n_diag, maxd);
}

void launch_sweep_check(const void* S, int prec, int n_pad, int64_t ld, double tol,
                        unsigned int* flags, cudaStream_t st) {
  const dim3 grid(n_pad / 32, n_pad / 32), block(32, 8);
  if (prec == 64)
    k_sweep_check<double><<<grid, block, 0, st>>>((const double*)S, ld, tol, flags);
  else
    k_sweep_check<float><<<grid, block, 0, st>>>((const float*)S, ld, tol, flags);
}

void launch_to_fixed(const void* S, int prec, long long* F, int n_pad, int64_t ld,
                     cudaStream_t st) {
  const dim3 grid(n_pad / 32, n_pad / 32), block(32, 8);
  if (prec == 64)
    k_to_fixed<double><<<grid, block, 0, st>>>((const double*)S, F, ld);
  else
    k_to_fixed<float><<<grid, block, 0, st>>>((const float*)S, F, ld);
}

void launch_from_fixed(const long long* F, void* S, int prec, int64_t count, cudaStream_t st) {
  const int blocks = 8192;
  if (prec == 64)
    k_from_fixed<double><<<blocks, 256, 0, st>>>(F, (double*)S, count);
  else
    k_from_fixed<float><<<blocks, 256, 0, st>>>(F, (float*)S, count);
}

}  // namespace sr
