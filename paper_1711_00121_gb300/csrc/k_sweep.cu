// Jacobi sweeps of Eq. 1, S <- C Q S Q^T + (1 - C) I, on a symmetric S held
// in 64-bit fixed point (value * 2^57), as two products per sweep:
//   T = (C Q S)^T,   S' = Q T,   with S' + (1 - C) I on the diagonal.
//
// What a sweep cannot do without is the gather of one row segment per edge.  In
// FP64 it was bound by the FP64 pipe (GB300 issues FP64 at 1/64 of the FP32
// rate).  Here the row sums are exact integer sums and the division by the
// in-degree is a product with a 63-bit reciprocal, rounded once: an error
// below 2^-57 a product, where one FP64 rounding of a value near 1 loses 2^-54.
// The error is absolute: an entry below 2^-4 holds fewer bits than in FP64, one
// below 2^-58 becomes zero (a first S stops at a change of 1e-13, some 2^-43).
// Rows of up to 32 nonzeros sum in 64 bits (|value| < 1.875: 32 of them stay
// below 2^63), longer ones flush such sums into 96 bits: with 96-bit sums for
// every row the kernels were bound by instruction issue.
//
// Work split: a CTA takes 32 rows x 128 columns, a warp one row at a time with
// four columns per lane (1 KB row segments, four nonzeros in flight).  CTAs of
// one column slab (128 columns of all rows, n KB) run next to each other, so
// the gathers stay in L2 and some of them in L1.  What bounds them now is the
// latency of those gathers at 9 to 10 TB/s out of L2: 64 columns and 512-byte
// segments took 10% longer, 8 in flight 5%, 2 in flight 8%.  A row of more than
// LONG_ROW nonzeros is gathered by the whole CTA.
// The first product is written transposed through shared memory; of the
// second only the tiles that reach the diagonal or above are formed (S' is
// symmetric), written together with their mirrors and compared with the old S
// for the stopping test.
#include "fixed64.h"

namespace sr {

namespace {

constexpr int NV = 2;         // pairs of columns per lane, 64 columns apart
constexpr int SR_ROWS = 32;    // rows of a CTA's tile
constexpr int SC_COLS = 64 * NV;  // columns of a CTA's tile
constexpr int WROWS = SR_ROWS / 8;  // rows of a warp
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

// The sum of a longer row times its factor r * 2^-(63 + s), s >= 5
__device__ __forceinline__ long long acc_scale(const Acc96& a, const SweepScale& f) {
  const bool neg = (int32_t)a.w2 < 0;
  unsigned long long lo = ((unsigned long long)a.w1 << 32) | a.w0;
  uint32_t hi = a.w2;
  if (neg) {
    lo = ~lo + 1ull;
    hi = ~hi + (lo == 0ull ? 1u : 0u);
  }
  const int s = f.sh;  // s - 1
  const unsigned __int128 t = (unsigned __int128)hi * f.r + __umul64hi(lo, f.r);
  const long long v = (long long)((t + ((unsigned __int128)1 << (s - 1))) >> s);
  return neg ? -v : v;
}

// Sums over m <= 32 nonzeros of the lane's columns, lane e holding the id of
// nonzero e: x's segment is at xc + x * pitch bytes.  Every lane takes part.
__device__ __forceinline__ void gather32(int id, int m, const char* __restrict__ xc,
                                         uint32_t pitch, long long (&s)[2 * NV]) {
  constexpr int NB = 4;
  for (int u = 0; u < m; u += NB) {
    longlong2 v[NB][NV];
#pragma unroll
    for (int k = 0; k < NB; ++k) {
      const uint32_t x = (uint32_t)__shfl_sync(0xffffffffu, id, u + k);
      const char* p = xc + (uint64_t)x * pitch;
#pragma unroll
      for (int q = 0; q < NV; ++q) {
        v[k][q] = make_longlong2(0, 0);
        if (u + k < m) v[k][q] = *reinterpret_cast<const longlong2*>(p + q * 512);
      }
    }
#pragma unroll
    for (int q = 0; q < NV; ++q)
#pragma unroll
      for (int k = 0; k < NB; k += 2) {
        s[2 * q] += v[k][q].x + v[k + 1][q].x;
        s[2 * q + 1] += v[k][q].y + v[k + 1][q].y;
      }
  }
}

// The same over the nonzeros [e0, e1) of a row whose ids start at col
__device__ __forceinline__ void gather_long(const int32_t* __restrict__ col, int e0, int e1,
                                            const char* __restrict__ xc, uint32_t pitch,
                                            Acc96 (&a)[2 * NV]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int q = 0; q < 2 * NV; ++q) a[q] = Acc96{0u, 0u, 0u};
  for (int b = e0; b < e1; b += 32) {
    const int m = min(32, e1 - b);
    const int id = lane < m ? __ldg(col + b + lane) : 0;
    long long s[2 * NV] = {};
    gather32(id, m, xc, pitch, s);
#pragma unroll
    for (int q = 0; q < 2 * NV; ++q) acc_add(a[q], s[q]);
  }
}

template <bool SECOND>
__global__ void __launch_bounds__(256, 4) k_sweep(DevAdj in, const SweepScale* __restrict__ scales,
                                               const long long* __restrict__ X, int64_t ld,
                                               long long* __restrict__ Y,
                                               const long long* __restrict__ Sold,
                                               long long diag, int n_diag,
                                               unsigned long long* __restrict__ maxd) {
  __shared__ long long tile[SR_ROWS][SC_COLS + 1];
  __shared__ Acc96 part[8][SC_COLS];
  __shared__ int longs[SR_ROWS];
  __shared__ int n_long;
  __shared__ unsigned long long wmax[8];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t row0 = (int64_t)blockIdx.x * SR_ROWS, col0 = (int64_t)blockIdx.y * SC_COLS;
  if (SECOND && row0 >= col0 + SC_COLS) return;  // below the diagonal: the whole CTA
  const char* xc = reinterpret_cast<const char*>(X + col0 + 2 * lane);
  const uint32_t pitch = (uint32_t)ld * 8u;
  if (threadIdx.x == 0) n_long = 0;
  // lane i < WROWS: extent of the warp's row i
  const int r0 = warp * WROWS;
  int my_len = 0;
  int64_t my_st = 0;
  if (lane < WROWS) {
    my_len = in.len[row0 + r0 + lane];
    my_st = in.start[row0 + r0 + lane];
  }
  __syncthreads();
  int len = __shfl_sync(0xffffffffu, my_len, 0);
  const int64_t st0 = __shfl_sync(0xffffffffu, my_st, 0);  // every lane takes part
  int id = lane < len ? __ldg(in.col + st0 + lane) : 0;
#pragma unroll
  for (int i = 0; i < WROWS; ++i) {
    const int r = r0 + i;
    // the next row's ids are on their way while this row is gathered
    int len1 = 0, id1 = 0;
    if (i + 1 < WROWS) {
      len1 = __shfl_sync(0xffffffffu, my_len, i + 1);
      const int64_t st1 = __shfl_sync(0xffffffffu, my_st, i + 1);
      if (lane < len1) id1 = __ldg(in.col + st1 + lane);
    }
    if (len <= 32) {
      const SweepScale f = scales[row0 + r];
      long long s[2 * NV] = {};
      gather32(id, len, xc, pitch, s);
#pragma unroll
      for (int q = 0; q < 2 * NV; ++q) tile[r][64 * (q / 2) + 2 * lane + (q & 1)] = fixed_scale(s[q], f);
    } else if (len <= LONG_ROW) {
      Acc96 a[2 * NV];
      gather_long(in.col + __shfl_sync(0xffffffffu, my_st, i), 0, len, xc, pitch, a);
      const SweepScale f = scales[row0 + r];
#pragma unroll
      for (int q = 0; q < 2 * NV; ++q) tile[r][64 * (q / 2) + 2 * lane + (q & 1)] = acc_scale(a[q], f);
    } else if (lane == 0) {
      longs[atomicAdd(&n_long, 1)] = r;
    }
    len = len1;
    id = id1;
  }
  __syncthreads();
  const int nl = n_long;
  for (int q = 0; q < nl; ++q) {
    const int r = longs[q];
    const int64_t a = row0 + r;
    const int L = in.len[a];
    const int per = ((L + 7) / 8 + 3) & ~3;
    Acc96 sum[2 * NV];
    gather_long(in.col + in.start[a], min(L, warp * per), min(L, (warp + 1) * per), xc, pitch,
                sum);
#pragma unroll
    for (int q = 0; q < 2 * NV; ++q) part[warp][64 * (q / 2) + 2 * lane + (q & 1)] = sum[q];
    __syncthreads();
    if (threadIdx.x < SC_COLS) {
      Acc96 s = part[0][threadIdx.x];
#pragma unroll
      for (int w = 1; w < 8; ++w) acc_add(s, part[w][threadIdx.x]);
      tile[r][threadIdx.x] = acc_scale(s, scales[a]);
    }
    __syncthreads();
  }
  if (!SECOND) {
    for (int k = warp; k < SC_COLS; k += 8) Y[(col0 + k) * ld + row0 + lane] = tile[lane][k];
    return;
  }
  // columns [k0, SC_COLS) of the tile are written; from km on they lie
  // strictly above the diagonal's 32 x 32 block and are mirrored
  const int k0 = row0 > col0 ? (int)(row0 - col0) : 0;
  const int km = row0 >= col0 ? k0 + SR_ROWS : 0;
  if (row0 >= col0) {
    // the diagonal block: add (1 - C), and the upper of two mirrored entries
    // (they are rounded in a different order) for both
    const int t = threadIdx.x;
    if (t < SR_ROWS && row0 + t < n_diag) tile[t][k0 + t] += diag;
    __syncthreads();
    for (int r = warp; r < SR_ROWS; r += 8)
      if (lane < r) tile[r][k0 + lane] = tile[lane][k0 + r];
    __syncthreads();
  }
  unsigned long long m = 0;
  for (int r = warp; r < SR_ROWS; r += 8) {
    long long* y = Y + (row0 + r) * ld + col0;
    const long long* o = Sold + (row0 + r) * ld + col0;
    for (int h = k0; h < SC_COLS; h += 32) {
      const long long v = tile[r][h + lane];
      const long long d = v - o[h + lane];
      m = max(m, (unsigned long long)(d < 0 ? -d : d));
      y[h + lane] = v;
    }
  }
  for (int k = km + warp; k < SC_COLS; k += 8)
    Y[(col0 + k) * ld + row0 + lane] = tile[lane][k];
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

// The mean of each pair of mirrored entries in fixed point, both places (FIX;
// S and F may be the same memory: a CTA reads its two blocks, then writes
// them), and what the fixed-point form cannot take (CHECK): *flags |= 1 for an
// entry of magnitude 1.875 or more (or a NaN), 2 for a pair of mirrored entries
// further apart than tol.  upper: the 128-tiles below the diagonal are taken
// as the mirrors of those above, unread.  One CTA per pair of 32 x 32 blocks.
template <typename T, bool CHECK, bool FIX>
__global__ void k_to_fixed(const T* S, long long* F, int64_t ld, int upper, double tol,
                           unsigned int* __restrict__ flags) {
  const int bi = blockIdx.y, bj = blockIdx.x;
  if (bj < bi) return;
  const bool one = upper && (bi * 32) / PT < (bj * 32) / PT;
  __shared__ T x1[32][33], x2[32][33];
  for (int r = threadIdx.y; r < 32; r += 8) {
    x1[r][threadIdx.x] = S[(int64_t)(bi * 32 + r) * ld + bj * 32 + threadIdx.x];
    if (!one) x2[r][threadIdx.x] = S[(int64_t)(bj * 32 + r) * ld + bi * 32 + threadIdx.x];
  }
  __syncthreads();
  unsigned int f = 0;
  for (int r = threadIdx.y; r < 32; r += 8) {
    const T x = x1[r][threadIdx.x];
    const T y = one ? x : x2[threadIdx.x][r];
    if (CHECK) {
      if (!(fabs(x) < T(1.875)) || !(fabs(y) < T(1.875))) f |= 1u;
      if (!one && !(fabs(x - y) <= (T)tol)) f |= 2u;
    }
    if (FIX) {
      // value * 2^56: the sum of the two is their mean * 2^57
      F[(int64_t)(bi * 32 + r) * ld + bj * 32 + threadIdx.x] = fixed_of(x, 0) + fixed_of(y, 0);
      if (bi != bj) {
        const T v = x1[threadIdx.x][r];
        const T w = one ? v : x2[r][threadIdx.x];
        F[(int64_t)(bj * 32 + r) * ld + bi * 32 + threadIdx.x] = fixed_of(v, 0) + fixed_of(w, 0);
      }
    }
  }
  if (CHECK) {
    f = __reduce_or_sync(0xffffffffu, f);
    if (threadIdx.x == 0 && f) atomicOr(flags, f);
  }
}

// S = F * 2^-57, rounded once (S and F may be the same memory); upper: the
// 128-tiles on or above the diagonal only
template <typename T>
__global__ void k_from_fixed(const long long* F, T* S, int64_t ld, int upper) {
  const int bi = blockIdx.y, bj = blockIdx.x;  // 32 rows x 128 columns
  if (upper && (bi * 32) / PT > bj) return;
  for (int r = threadIdx.y; r < 32; r += 8) {
    const int64_t o = (int64_t)(bi * 32 + r) * ld + bj * PT + threadIdx.x;
#pragma unroll
    for (int q = 0; q < PT; q += 32) S[o + q] = fixed_value<T>(F[o + q], -57);
  }
}

}  // namespace

// Loads the kernels of the sweeps and of the way back (a kernel loaded at its
// first launch can fail there for want of memory).
cudaError_t sweep_fixed_ready(int prec) {
  const void* fn[4] = {(const void*)k_sweep<false>, (const void*)k_sweep<true>,
                       prec == 64 ? (const void*)k_to_fixed<double, false, true>
                                  : (const void*)k_to_fixed<float, false, true>,
                       prec == 64 ? (const void*)k_from_fixed<double>
                                  : (const void*)k_from_fixed<float>};
  for (const void* f : fn) {
    cudaFuncAttributes a;
    const cudaError_t e = cudaFuncGetAttributes(&a, f);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

void launch_sweep_fixed(const DevAdj& in, const SweepScale* s1, const SweepScale* s2,
                        const long long* S, int64_t ld, int n_pad, long long* T, long long* Snew,
                        long long diag, int n_diag, unsigned long long* maxd, cudaStream_t st) {
  const dim3 grid(n_pad / SR_ROWS, n_pad / SC_COLS);
  k_sweep<false><<<grid, 256, 0, st>>>(in, s1, S, ld, T, nullptr, 0, 0, nullptr);
  k_sweep<true><<<grid, 256, 0, st>>>(in, s2, T, ld, Snew, S, diag, n_diag, maxd);
}

void launch_to_fixed(const void* S, int prec, long long* F, int n_pad, int64_t ld, int upper,
                     bool check, double tol, unsigned int* flags, cudaStream_t st) {
  const dim3 grid(n_pad / 32, n_pad / 32), block(32, 8);
  if (prec == 64) {
    const double* s = (const double*)S;
    if (!F)
      k_to_fixed<double, true, false><<<grid, block, 0, st>>>(s, F, ld, upper, tol, flags);
    else if (check)
      k_to_fixed<double, true, true><<<grid, block, 0, st>>>(s, F, ld, upper, tol, flags);
    else
      k_to_fixed<double, false, true><<<grid, block, 0, st>>>(s, F, ld, upper, tol, flags);
  } else {
    const float* s = (const float*)S;
    if (check)
      k_to_fixed<float, true, true><<<grid, block, 0, st>>>(s, F, ld, upper, tol, flags);
    else
      k_to_fixed<float, false, true><<<grid, block, 0, st>>>(s, F, ld, upper, tol, flags);
  }
}

void launch_from_fixed(const long long* F, void* S, int prec, int n_pad, int64_t ld, int upper,
                       cudaStream_t st) {
  const dim3 grid(n_pad / PT, n_pad / 32), block(32, 8);
  if (prec == 64)
    k_from_fixed<double><<<grid, block, 0, st>>>(F, (double*)S, ld, upper);
  else
    k_from_fixed<float><<<grid, block, 0, st>>>(F, (float*)S, ld, upper);
}

}  // namespace sr
