// Column mode (§7): SimRank columns without a dense S, in O(Kn + m) memory
// per column.
//  - Procedure 1 (PartialSim) on a block of B columns: forward steps
//    X_t = Q^T X_{t-1} over the out-lists (row b of Q^T X sums X[a,:] / d_a
//    over the out-neighbours a of b), stored for t = 0..K, then the Horner
//    steps Y <- X_{K-t} + C Q Y over the in-lists; result (1-C) Y.
//  - The change of a column through the stored updates (Eq. 70-71):
//    Y[a, c] += sum_k xi_k[a] eta_k[x_c] + eta_k[a] xi_k[x_c].
// Blocks are row-major [node][B]; the arithmetic is in the storage
// precision (FP32 or FP64).  With FP32 the change through the stored updates
// is one dense product per block: Y += A G with A = [xi_k, eta_k of every
// update] (n x 2 U (K+1), straight from the tile-blocked panels) and G the
// matching values at the block's columns.
#include <algorithm>

#include "quotient.h"
#include "sr_internal.h"

namespace sr {

namespace {

// X0[x_c][c] = 1 (the other entries are zero beforehand)
template <typename T>
__global__ void k_col_unit(const int32_t* __restrict__ cols, int B, int ldb, T* __restrict__ X0) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c < B) X0[(int64_t)cols[c] * ldb + c] = (T)1;
}

// Column 0 of X0 = the indicator of the distinct ids cols[0 .. g0), column c
// (1 <= c < B) = e_{cols[g0 + c - 1]}: Procedure 1 is linear in its start
// vector, so column 0 of its result is the sum of the g0 columns.
template <typename T>
__global__ void k_col_unit_grouped(const int32_t* __restrict__ cols, int g0, int B, int ldb,
                                   T* __restrict__ X0) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q < g0) X0[(int64_t)cols[q] * ldb] = (T)1;
  else if (q < g0 + B - 1) X0[(int64_t)cols[q] * ldb + (q - g0 + 1)] = (T)1;
}

// Y[a][c] = s * X[a][c] (X may be null: Y = 0), a < n_rows, c < B
template <typename T>
__global__ void k_col_fill(const T* __restrict__ X, double s, T* __restrict__ Y, int64_t count) {
  const T sv = (T)s;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < count;
       e += (int64_t)gridDim.x * blockDim.x)
    Y[e] = X ? sv * X[e] : (T)0;
}

// Four (FP32) or two (FP64) adjacent columns as one 16-byte access, or half
// of that (VEC columns of type T).
template <typename T, int VEC>
struct ColVec {
  T v[VEC];
};
template <typename T, int VEC>
__device__ __forceinline__ ColVec<T, VEC> ld_cols(const T* p) {
  ColVec<T, VEC> r;
  if constexpr (sizeof(T) * VEC == 16) {
    const uint4 x = *reinterpret_cast<const uint4*>(p);
    memcpy(&r, &x, 16);
  } else {
    const uint2 x = *reinterpret_cast<const uint2*>(p);
    memcpy(&r, &x, 8);
  }
  return r;
}
template <typename T, int VEC>
__device__ __forceinline__ void st_cols(T* p, const ColVec<T, VEC>& r) {
  if constexpr (sizeof(T) * VEC == 16) {
    uint4 x;
    memcpy(&x, &r, 16);
    *reinterpret_cast<uint4*>(p) = x;
  } else {
    uint2 x;
    memcpy(&x, &r, 8);
    *reinterpret_cast<uint2*>(p) = x;
  }
}
template <typename T, int VEC>
__device__ __forceinline__ void add_cols(T* p, const ColVec<T, VEC>& r) {
  if constexpr (sizeof(T) == 4 && VEC == 4) {
    atomicAdd(reinterpret_cast<float4*>(p), make_float4(r.v[0], r.v[1], r.v[2], r.v[3]));
  } else if constexpr (sizeof(T) == 4 && VEC == 2) {
    atomicAdd(reinterpret_cast<float2*>(p), make_float2(r.v[0], r.v[1]));
  } else {
#pragma unroll
    for (int c = 0; c < VEC; ++c) atomicAdd(p + c, r.v[c]);
  }
}

// One SpMM step on a block of ldb columns (ldb a multiple of 4), one warp per
// row chunk (at most kChunk = 32 nonzeros of one adjacency row) and 32 * VEC
// columns (blockIdx.y):
//   forward (Q^T, out-lists): Y[row][c]  = sum_e w_e nodes[col_e] X[col_e][c]
//                             (in FP64 X comes divided, k_col_quotient: no nodes)
//   Horner  (Q,   in-lists):  Y[row][c]  = add_scale Xadd[row][c]
//                                          + nodes[row] sum_e w_e X[col_e][c]
// nodes holds 1 / d (or 1 / in-weight) per node, times the step's scale for
// Horner; w_e = 1 without weights.  A row of one chunk (most rows; an empty
// row has one empty chunk) is written once; the chunks of a longer row add
// theirs to the row that k_col_prefill has set.
//
// Bound by the gathered bytes (FP32) or by GB300's FP64 rate of one FMA per
// gathered value (FP64).  A warp takes `per` consecutive chunks; a chunk's
// column ids and factors are loaded once, one per lane, two chunks ahead of
// their use, and broadcast by shuffles, so that the loop holds a gather and an
// FMA per value and no division, index load or degree load.
template <typename T, int VEC, bool FORWARD>
__global__ void __launch_bounds__(256, 6) k_col_rows(
    const RowChunk* __restrict__ chunks, int64_t count, int per, const int32_t* __restrict__ col,
    const float* __restrict__ ew, const T* __restrict__ nodes, const T* __restrict__ X,
    const T* __restrict__ Xadd, T add_scale, T* __restrict__ Y, int ldb) {
  constexpr unsigned full = 0xffffffffu;
  constexpr int NB = 4;  // gathers in flight per lane
  const int lane = threadIdx.x & 31;
  const int64_t q0 = ((int64_t)blockIdx.x * 8 + (threadIdx.x >> 5)) * per;
  if (q0 >= count) return;  // the whole warp
  const int nq = (int)min((int64_t)per, count - q0);  // <= 32
  const int c = ((int)blockIdx.y * 32 + lane) * VEC;
  const bool act = c < ldb;
  // lane i holds chunk q0 + i
  RowChunk mine;
  mine.row = mine.len = 0;
  mine.start = 0;
  if (lane < nq) mine = chunks[q0 + lane];
  // column id of nonzero `lane` of chunk i, and its factor
  auto col_of = [&](int i) -> int {
    const int len = __shfl_sync(full, mine.len, i) & 0xffff;
    const int64_t st = __shfl_sync(full, mine.start, i);
    return (i < nq && lane < len) ? col[st + lane] : 0;
  };
  auto factor_of = [&](int i, int a) -> T {
    const int len = __shfl_sync(full, mine.len, i) & 0xffff;
    const int64_t st = __shfl_sync(full, mine.start, i);
    T w = T(0);
    if (i < nq && lane < len) {
      w = FORWARD && sizeof(T) == 4 ? nodes[a] : T(1);
      if (ew) w *= (T)ew[st + lane];
    }
    return w;
  };
  int a = col_of(0);
  T w = factor_of(0, a);
  int a1 = col_of(1);
  for (int i = 0; i < nq; ++i) {
    const T w1 = factor_of((i + 1) & 31, a1);
    const int a2 = col_of((i + 2) & 31);
    const int row = __shfl_sync(full, mine.row, i);
    const int lf = __shfl_sync(full, mine.len, i);
    const int len = lf & 0xffff;
    const bool only = (lf & CH_ONLY) != 0;
    const int64_t o = (int64_t)row * ldb + c;
    ColVec<T, VEC> acc;
#pragma unroll
    for (int u = 0; u < VEC; ++u) acc.v[u] = T(0);
    for (int e = 0; e < len; e += NB) {
      ColVec<T, VEC> x[NB];
#pragma unroll
      for (int u = 0; u < NB; ++u) {
        const int64_t b = __shfl_sync(full, a, e + u);
        if (act && e + u < len) {
          x[u] = ld_cols<T, VEC>(X + b * ldb + c);
        } else {
#pragma unroll
          for (int z = 0; z < VEC; ++z) x[u].v[z] = T(0);
        }
      }
#pragma unroll
      for (int u = 0; u < NB; ++u) {
        if (e + u >= len) break;
        const T we = __shfl_sync(full, w, e + u);
#pragma unroll
        for (int z = 0; z < VEC; ++z) acc.v[z] += we * x[u].v[z];
      }
    }
    if (!FORWARD && len > 0) {
      const T rs = nodes[row];
#pragma unroll
      for (int z = 0; z < VEC; ++z) acc.v[z] *= rs;
    }
    if (act) {
      if (only) {
        if (!FORWARD && Xadd) {
          const ColVec<T, VEC> base = ld_cols<T, VEC>(Xadd + o);
#pragma unroll
          for (int z = 0; z < VEC; ++z) acc.v[z] += add_scale * base.v[z];
        }
        st_cols<T, VEC>(Y + o, acc);
      } else {
        add_cols<T, VEC>(Y + o, acc);
      }
    }
    a = a1;
    w = w1;
    a1 = a2;
  }
}

// The rows of more than one chunk before k_col_rows adds to them:
// Y[row][c] = add_scale * Xadd[row][c] (0 without Xadd), one CTA per row.
template <typename T>
__global__ void k_col_prefill(const int32_t* __restrict__ rows, const T* __restrict__ Xadd,
                              T add_scale, T* __restrict__ Y, int ldb) {
  const int64_t o = (int64_t)rows[blockIdx.x] * ldb;
  for (int c = threadIdx.x; c < ldb; c += blockDim.x)
    Y[o + c] = Xadd ? add_scale * Xadd[o + c] : T(0);
}

// U[a][c] = X[a][c] / (in-degree or in-weight of a) by its reciprocal (quotient.h:
// three FP64 operations where a division takes some ten), 0 for a node without
// in-neighbours.  One pass over the block before an FP64 forward step (a gradient
// over 600 pairs at n = 5,000: 13.0 to 14.3 ms); a product with the reciprocal
// inside the step rounds twice.  One CTA per row.
__global__ void __launch_bounds__(128)
    k_col_quotient(const double* __restrict__ X, const int32_t* __restrict__ in_len,
                   const double* __restrict__ wsum, const double* __restrict__ recip, int ldb,
                   double* __restrict__ U) {
  const int64_t a = blockIdx.x;
  const double r = recip[a], d = wsum ? wsum[a] : (double)in_len[a];
  const double* x = X + a * ldb;
  double* u = U + a * ldb;
  if (fx_bits(r) == 0) {  // (a test on the FP64 pipe would count)
    for (int c = threadIdx.x; c < ldb; c += 128) u[c] = 0.0;
    return;
  }
  bool again = false;
  for (int c = threadIdx.x; c < ldb; c += 128) {
    const double v = quotient_fast(x[c], d, r);
    again |= !quotient_ok(v);
    u[c] = v;
  }
  // a second look at the rare others, out of the loop
  if (again)
    for (int c = threadIdx.x; c < ldb; c += 128) u[c] = quotient(x[c], d, r);
}

// out[a] = scale / (in-degree or in-weight of a), 0 without in-neighbours
template <typename T>
__global__ void k_col_scales(const int32_t* __restrict__ in_len, const double* __restrict__ wsum,
                             double scale, int n_rows, T* __restrict__ out) {
  const int a = blockIdx.x * blockDim.x + threadIdx.x;
  if (a >= n_rows) return;
  const T d = wsum ? (T)wsum[a] : (T)in_len[a];
  out[a] = in_len[a] > 0 ? (T)scale / d : T(0);
}

int num_sms_for_narrow() {
  static int sms = 0;
  if (sms == 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0)
      sms = 152;
  }
  return sms;
}

// Narrow blocks (B = BW <= 4 columns, e.g. the two old columns of one update):
// persistent warps, each taking four row chunks at a time (a chunk has at
// most 32 nonzeros): an 8-lane group per chunk, up to four nonzeros per lane
// gathered at once, the group's sums combined by shuffles within the group
// and added by its first lane.  The forward step reads X already divided by
// the in-degree (or in-weight) of each row (k_col_prescale).
template <typename T, bool FORWARD, int BW>
__global__ void __launch_bounds__(256) k_col_chunk_narrow(
    const RowChunk* __restrict__ chunks, int64_t count, const int32_t* __restrict__ col,
    const float* __restrict__ ew, const int32_t* __restrict__ in_len,
    const double* __restrict__ wsum, const T* __restrict__ X, T* __restrict__ Y, double scale) {
  const int lane = threadIdx.x & 31, g = lane >> 3, gl = lane & 7;
  const int64_t nwarps = (int64_t)gridDim.x * (blockDim.x >> 5);
  // the loop bound depends on the warp only: every lane runs every shuffle
  for (int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; w * 4 < count;
       w += nwarps) {
    const int64_t q = w * 4 + g;
    RowChunk ch;
    ch.row = 0;
    ch.len = 0;
    ch.start = 0;
    if (q < count) ch = chunks[q];
    ch.len = chunk_len(ch);
    int a[4];
    T wt[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int e = gl + 8 * u;
      a[u] = (e < ch.len) ? col[ch.start + e] : -1;
      wt[u] = (e < ch.len && ew) ? (T)ew[ch.start + e] : T(1);
    }
    T acc[BW];
#pragma unroll
    for (int c = 0; c < BW; ++c) acc[c] = T(0);
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (a[u] >= 0) {
#pragma unroll
        for (int c = 0; c < BW; ++c) acc[c] += wt[u] * X[(int64_t)a[u] * BW + c];
      }
#pragma unroll
    for (int c = 0; c < BW; ++c)
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) acc[c] += __shfl_xor_sync(0xffffffffu, acc[c], o, 8);
    if (gl == 0 && ch.len > 0) {
      const T rs = FORWARD ? T(1) : (T)scale / (wsum ? (T)wsum[ch.row] : (T)in_len[ch.row]);
#pragma unroll
      for (int c = 0; c < BW; ++c) atomicAdd(&Y[(int64_t)ch.row * BW + c], rs * acc[c]);
    }
  }
}

// Z[a][c] = X[a][c] / (in-degree of a, or its in-weight), a < n_rows, c < B
template <typename T>
__global__ void k_col_prescale(const T* __restrict__ X, const int32_t* __restrict__ in_len,
                               const double* __restrict__ wsum, int B, int64_t count,
                               T* __restrict__ Z) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < count;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t a = e / B;
    const T d = wsum ? (T)wsum[a] : (T)in_len[a];
    Z[e] = d != T(0) ? X[e] / d : T(0);
  }
}

// Y[a][c] += sum_k xi_k[a] eta_k[x_c] + eta_k[a] xi_k[x_c] for one stored
// update (tile-blocked panels P[T][which][k][128]); the panel values at the
// block's columns are staged in shared memory.
template <typename T, typename TP>
__global__ void k_col_apply(const TP* __restrict__ P, int K1, const int32_t* __restrict__ cols,
                            int B, int ldb, int n_rows, T* __restrict__ Y) {
  extern __shared__ double sg[];  // [B][2*K1]: xi_k[x_c], eta_k[x_c]
  for (int e = threadIdx.x; e < B * K1; e += blockDim.x) {
    const int c = e / K1, k = e % K1;
    const int64_t x = cols[c];
    const int64_t base = ((x / PT) * 2) * (int64_t)K1 * PT + (int64_t)k * PT + (x % PT);
    sg[c * 2 * K1 + k] = (double)P[base];
    sg[c * 2 * K1 + K1 + k] = (double)P[base + (int64_t)K1 * PT];
  }
  __syncthreads();
  const int64_t a = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (a >= n_rows) return;
  const int64_t ba = ((a / PT) * 2) * (int64_t)K1 * PT + (a % PT);
  for (int c = 0; c < B; ++c) {
    const double* g = sg + c * 2 * K1;
    double acc = 0.0;
    for (int k = 0; k < K1; ++k)
      acc += (double)P[ba + (int64_t)k * PT] * g[K1 + k] +
             (double)P[ba + (int64_t)(K1 + k) * PT] * g[k];
    Y[a * ldb + c] = (T)((double)Y[a * ldb + c] + acc);
  }
}

// G[u][r][c] for the FP32 product: r = which * K1 + k, the value of the
// OTHER vector of term k of update u at column x_c (eta_k[x_c] pairs with
// xi_k[a], xi_k[x_c] with eta_k[a]); c < B, zero for c in [B, Bp).
__global__ void k_col_gvals(const float* const* __restrict__ hist, int K1,
                            const int32_t* __restrict__ cols, int B, int Bp,
                            float* __restrict__ G) {
  const int u = blockIdx.y;
  const float* P = hist[u];
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < 2 * K1 * Bp; e += gridDim.x * blockDim.x) {
    const int r = e / Bp, c = e % Bp;
    const int which = r / K1, k = r % K1;
    float v = 0.f;
    if (c < B) {
      const int64_t x = cols[c];
      v = P[(((x / PT) * 2 + (1 - which)) * (int64_t)K1 + k) * PT + (x % PT)];
    }
    G[((int64_t)u * 2 * K1 + r) * Bp + c] = v;
  }
}

// Y[a][c] += sum_u sum_r A_u[a][r] G[u][r][c] for the 128 rows of tile
// blockIdx.x and the 128 columns of group blockIdx.y (256 threads, an 8 x 8
// block of outputs each; the r-chunks of A and G are staged in shared memory:
// A_u's tile-blocked panel slice [r][128 rows] is already in that layout).
constexpr int CG_KC = 16;
__global__ void __launch_bounds__(256) k_col_corr(const float* const* __restrict__ hist, int U,
                                                  int K1, const float* __restrict__ G, int Bp,
                                                  int B, int ldb, int n_rows,
                                                  float* __restrict__ Y) {
  __shared__ __align__(16) float sA[CG_KC][PT];
  __shared__ __align__(16) float sG[CG_KC][PT];
  const int T = blockIdx.x, c0 = blockIdx.y * PT;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  float acc[8][8];
#pragma unroll
  for (int r = 0; r < 8; ++r)
#pragma unroll
    for (int c = 0; c < 8; ++c) acc[r][c] = 0.f;
  const int R = 2 * K1;
  for (int u = 0; u < U; ++u) {
    const float* Pt = hist[u] + (int64_t)T * 2 * K1 * PT;  // [r][128], r = which * K1 + k
    const float* Gu = G + (int64_t)u * R * Bp;
    for (int r0 = 0; r0 < R; r0 += CG_KC) {
      const int kc = min(CG_KC, R - r0);
      __syncthreads();
      for (int e = tid; e < kc * PT / 4; e += 256) {
        const int rr = e / (PT / 4), q = e % (PT / 4);
        reinterpret_cast<float4*>(sA[rr])[q] =
            reinterpret_cast<const float4*>(Pt + (int64_t)(r0 + rr) * PT)[q];
        float4 g = make_float4(0.f, 0.f, 0.f, 0.f);
        const int cc = c0 + 4 * q;
        if (cc < Bp) g = *reinterpret_cast<const float4*>(Gu + (int64_t)(r0 + rr) * Bp + cc);
        reinterpret_cast<float4*>(sG[rr])[q] = g;
      }
      __syncthreads();
      for (int rr = 0; rr < kc; ++rr) {
        float a[8], g[8];
        const float4 a0 = reinterpret_cast<const float4*>(sA[rr])[ty];
        const float4 a1 = reinterpret_cast<const float4*>(sA[rr])[16 + ty];
        const float4 g0 = reinterpret_cast<const float4*>(sG[rr])[tx];
        const float4 g1 = reinterpret_cast<const float4*>(sG[rr])[16 + tx];
        a[0] = a0.x; a[1] = a0.y; a[2] = a0.z; a[3] = a0.w;
        a[4] = a1.x; a[5] = a1.y; a[6] = a1.z; a[7] = a1.w;
        g[0] = g0.x; g[1] = g0.y; g[2] = g0.z; g[3] = g0.w;
        g[4] = g1.x; g[5] = g1.y; g[6] = g1.z; g[7] = g1.w;
#pragma unroll
        for (int r = 0; r < 8; ++r)
#pragma unroll
          for (int c = 0; c < 8; ++c) acc[r][c] = fmaf(a[r], g[c], acc[r][c]);
      }
    }
  }
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    const int64_t row = (int64_t)T * PT + ((r < 4) ? ty * 4 + r : 64 + ty * 4 + (r - 4));
    if (row >= n_rows) continue;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      const int col = c0 + ((c < 4) ? tx * 4 + c : 64 + tx * 4 + (c - 4));
      if (col < B) Y[row * ldb + col] += acc[r][c];
    }
  }
}

// out[c * n + a] = Y[a][c] (column-major output, optional FP32), transposed
// in 32 x 32 blocks through shared memory so that both sides are read and
// written in rows (200,000 x 256, FP32: 226 us when read column by column).
template <typename T, typename TO>
__global__ void k_col_out(const T* __restrict__ Y, int B, int ldb, int n, TO* __restrict__ out) {
  __shared__ T tile[32][33];
  const int a0 = blockIdx.x * 32, c0 = blockIdx.y * 32;
  for (int r = threadIdx.y; r < 32; r += 8)
    if (a0 + r < n && c0 + (int)threadIdx.x < B)
      tile[r][threadIdx.x] = Y[(int64_t)(a0 + r) * ldb + c0 + threadIdx.x];
  __syncthreads();
  for (int r = threadIdx.y; r < 32; r += 8)
    if (c0 + r < B && a0 + (int)threadIdx.x < n)
      out[(int64_t)(c0 + r) * n + a0 + threadIdx.x] = (TO)tile[threadIdx.x][r];
}

// column c of a row-major [n][B] block into a contiguous FP64 vector
template <typename T>
__global__ void k_col_extract(const T* __restrict__ Y, int B, int c, int n, double* __restrict__ v) {
  const int a = blockIdx.x * blockDim.x + threadIdx.x;
  if (a < n) v[a] = (double)Y[(int64_t)a * B + c];
}

}  // namespace

// One wide step (ldb > 4) over the row chunks L; a warp covers 512 bytes of a
// row.  Chunks per warp: up to 8 in FP32, as long as every SM keeps some 64
// warps to run (200,000 nodes x 256 columns: 9.6 ms a query with 8, 10.8 ms
// with 1; with 8 gathers in flight per lane instead of 4, 13-15 ms: they push
// the rows that are gathered often out of L1).  FP64 is bound by its FMAs and
// takes one chunk per warp (gradient, 5,000 nodes: 13.0 ms with 1, 15.1 ms
// with 8).
template <typename T>
static void wide_step(const ChunkList& L, const int32_t* adj, const float* w, bool forward,
                      const T* nodes, const T* X, const T* Xadd, double add_scale, T* Y, int ldb,
                      cudaStream_t st) {
  constexpr int VEC = 16 / sizeof(T);
  if (L.multi_count > 0)
    k_col_prefill<T><<<(unsigned)L.multi_count, 128, 0, st>>>(L.multi, Xadd, (T)add_scale, Y, ldb);
  if (L.count <= 0) return;
  const int groups = (ldb + 32 * VEC - 1) / (32 * VEC);
  const int64_t warps = (int64_t)num_sms_for_narrow() * 64;
  const int per = sizeof(T) == 8 ? 1
                                 : (int)std::max<int64_t>(
                                       1, std::min<int64_t>(8, L.count * groups / warps));
  const dim3 grid((unsigned)((L.count + 8 * per - 1) / (8 * per)), (unsigned)groups);
  if (forward)
    k_col_rows<T, VEC, true><<<grid, 256, 0, st>>>(L.chunks, L.count, per, adj, w, nodes, X,
                                                   nullptr, T(0), Y, ldb);
  else
    k_col_rows<T, VEC, false><<<grid, 256, 0, st>>>(L.chunks, L.count, per, adj, w, nodes, X, Xadd,
                                                    (T)add_scale, Y, ldb);
}

template <typename T>
static void partial_sim_block_t(const ChunkList& fwd, const ChunkList& hor, const int32_t* out_col,
                                const int32_t* in_col, const WeightView& wv, const int32_t* in_len,
                                const int32_t* cols, int B, int ldb, int n_rows, int K, double C,
                                T* xs, T* y0, T* y1, T* result, T* scales, cudaStream_t st,
                                int group0) {
  const int64_t blk = (int64_t)n_rows * ldb;
  const int fill_blocks = 4096;
  k_col_fill<T><<<fill_blocks, 256, 0, st>>>(nullptr, 0.0, xs, blk);
  if (group0 > 1)
    k_col_unit_grouped<T><<<(group0 + B + 126) / 128, 128, 0, st>>>(cols, group0, B, ldb, xs);
  else
    k_col_unit<T><<<(B + 127) / 128, 128, 0, st>>>(cols, B, ldb, xs);
  if (K == 0) {
    k_col_fill<T><<<fill_blocks, 256, 0, st>>>(xs, 1.0 - C, result, blk);
    return;
  }
  T* bufs[2] = {y0, y1};
  if (ldb > 4) {
    // wide blocks: 1 / d per node, and C / d, (1 - C) C / d for the Horner steps
    T* inv = scales;
    T* hs = scales + n_rows;
    T* hl = scales + 2 * (int64_t)n_rows;
    const int nb = (n_rows + 255) / 256;
    k_col_scales<T><<<nb, 256, 0, st>>>(in_len, wv.wsum, 1.0, n_rows, inv);
    k_col_scales<T><<<nb, 256, 0, st>>>(in_len, wv.wsum, C, n_rows, hs);
    k_col_scales<T><<<nb, 256, 0, st>>>(in_len, wv.wsum, (1.0 - C) * C, n_rows, hl);
    for (int t = 1; t <= K; ++t) {
      const T* X = xs + (int64_t)(t - 1) * blk;
      T* Y = xs + (int64_t)t * blk;
      if constexpr (sizeof(T) == 8)  // y0 is free until the Horner steps
        launch_col_forward64(fwd, out_col, wv, in_len, n_rows, inv, X, y0, Y, ldb, st);
      else
        wide_step<T>(fwd, out_col, wv.out_w, true, inv, X, nullptr, 0.0, Y, ldb, st);
    }
    const T* y = xs + (int64_t)K * blk;
    for (int t = 1; t <= K; ++t) {
      T* dst = (t == K) ? result : bufs[t & 1];
      wide_step<T>(hor, in_col, wv.in_w, false, t == K ? hl : hs, y,
                       xs + (int64_t)(K - t) * blk, t == K ? 1.0 - C : 1.0, dst, ldb, st);
      y = dst;
    }
    return;
  }
  // narrow blocks: a group of 8 lanes per chunk; the forward input divided once per row
  auto narrow_step = [&](const ChunkList& L, const int32_t* adj, const float* w, bool forward,
                         const T* X, T* Y, double scale) {
    if (L.filled <= 0) return;
    // persistent: at most 8 CTAs of 8 warps per SM, four chunks per warp at a time
    const int64_t want = (L.filled + 31) / 32;
    const unsigned grid = (unsigned)std::min<int64_t>(want, (int64_t)num_sms_for_narrow() * 8);
#define SR_NARROW(BW)                                                                          \
  do {                                                                                         \
    if (forward)                                                                               \
      k_col_chunk_narrow<T, true, BW><<<grid, 256, 0, st>>>(L.chunks, L.filled, adj, w, in_len, \
                                                            wv.wsum, X, Y, scale);             \
    else                                                                                       \
      k_col_chunk_narrow<T, false, BW><<<grid, 256, 0, st>>>(L.chunks, L.filled, adj, w, in_len, \
                                                             wv.wsum, X, Y, scale);            \
  } while (0)
    switch (ldb) {
      case 1: SR_NARROW(1); break;
      case 2: SR_NARROW(2); break;
      case 3: SR_NARROW(3); break;
      default: SR_NARROW(4); break;
    }
#undef SR_NARROW
  };
  for (int t = 1; t <= K; ++t) {
    T* dst = xs + (int64_t)t * blk;
    k_col_fill<T><<<fill_blocks, 256, 0, st>>>(nullptr, 0.0, dst, blk);
    // y0 is free until the Horner steps: it holds X divided by the row degrees
    k_col_prescale<T><<<fill_blocks, 256, 0, st>>>(xs + (int64_t)(t - 1) * blk, in_len, wv.wsum,
                                                   ldb, blk, y0);
    narrow_step(fwd, out_col, wv.out_w, true, y0, dst, 1.0);
  }
  // Horner: y = x_K; y <- x_{K-t} + C Q y; result (1-C) y (the last step folds the scale)
  const T* y = xs + (int64_t)K * blk;
  for (int t = 1; t <= K; ++t) {
    T* dst = (t == K) ? result : bufs[t & 1];
    const double s = (t == K) ? 1.0 - C : 1.0;
    k_col_fill<T><<<fill_blocks, 256, 0, st>>>(xs + (int64_t)(K - t) * blk, s, dst, blk);
    narrow_step(hor, in_col, wv.in_w, false, y, dst, s * C);
    y = dst;
  }
}

void launch_partial_sim_block(const ChunkList& fwd, const ChunkList& hor, const int32_t* out_col,
                              const int32_t* in_col, const int32_t* in_len, const int32_t* cols,
                              int B, int ldb, int n_rows, int K, double C, int prec, void* xs,
                              void* y0, void* y1, void* result, void* scales, cudaStream_t st,
                              const WeightView& wv, int group0) {
  if (prec == 64)
    partial_sim_block_t<double>(fwd, hor, out_col, in_col, wv, in_len, cols, B, ldb, n_rows, K, C,
                                (double*)xs, (double*)y0, (double*)y1, (double*)result,
                                (double*)scales, st, group0);
  else
    partial_sim_block_t<float>(fwd, hor, out_col, in_col, wv, in_len, cols, B, ldb, n_rows, K, C,
                               (float*)xs, (float*)y0, (float*)y1, (float*)result, (float*)scales,
                               st, group0);
}

void launch_col_scales64(const WeightView& wv, const int32_t* in_len, int n_rows, double* inv,
                         cudaStream_t st) {
  k_col_scales<double><<<(n_rows + 255) / 256, 256, 0, st>>>(in_len, wv.wsum, 1.0, n_rows, inv);
}

// Y = Q^T X (FP64 blocks [n_rows][ldb]); U: X over the in-degrees or in-weights
void launch_col_forward64(const ChunkList& fwd, const int32_t* out_col, const WeightView& wv,
                          const int32_t* in_len, int n_rows, const double* inv, const double* X,
                          double* U, double* Y, int ldb, cudaStream_t st) {
  k_col_quotient<<<n_rows, 128, 0, st>>>(X, in_len, wv.wsum, inv, ldb, U);
  wide_step<double>(fwd, out_col, wv.out_w, true, nullptr, U, nullptr, 0.0, Y, ldb, st);
}

// Yn = add_scale * Xadd + Q Y (FP64 blocks [n_rows][ldb])
void launch_col_horner64(const ChunkList& hor, const int32_t* in_col, const WeightView& wv,
                         const double* inv, const double* Xadd, double add_scale, const double* Y,
                         double* Yn, int ldb, cudaStream_t st) {
  wide_step<double>(hor, in_col, wv.in_w, false, inv, Y, Xadd, add_scale, Yn, ldb, st);
}

// The columns of one update's panels staged by a CTA take 16 (K + 1) bytes each:
// as many columns per launch as fit in its shared memory (908 at K = 15).
template <typename T, typename TP>
static cudaError_t col_apply_t(const TP* P, int K1, const int32_t* cols, int B, int ldb,
                               int n_rows, T* Y, cudaStream_t st) {
  constexpr int most = 227 * 1024;
  static std::atomic<unsigned long long> done{0};
  const cudaError_t e = smem_attr_once((const void*)k_col_apply<T, TP>, most, done);
  if (e != cudaSuccess) return e;
  const int per = std::max(1, most / (2 * K1 * (int)sizeof(double)));
  const int threads = 128, blocks = (n_rows + threads - 1) / threads;
  for (int c0 = 0; c0 < B; c0 += per) {
    const int b = std::min(per, B - c0);
    k_col_apply<T, TP><<<blocks, threads, (size_t)b * 2 * K1 * sizeof(double), st>>>(
        P, K1, cols + c0, b, ldb, n_rows, Y + c0);
  }
  return cudaSuccess;
}

cudaError_t launch_col_apply(const void* P, int p_prec, int K1, const int32_t* cols, int B,
                             int ldb, int n_rows, int prec, void* Y, cudaStream_t st) {
  if (prec == 64 && p_prec == 64)
    return col_apply_t((const double*)P, K1, cols, B, ldb, n_rows, (double*)Y, st);
  if (prec == 64)
    return col_apply_t((const float*)P, K1, cols, B, ldb, n_rows, (double*)Y, st);
  if (p_prec == 64)
    return col_apply_t((const double*)P, K1, cols, B, ldb, n_rows, (float*)Y, st);
  return col_apply_t((const float*)P, K1, cols, B, ldb, n_rows, (float*)Y, st);
}

void launch_col_corr(const float* const* hist, int U, int K1, const int32_t* cols, int B, int ldb,
                     int n_rows, float* G, float* Y, cudaStream_t st) {
  if (U <= 0 || B <= 0) return;
  const int Bp = (B + 3) / 4 * 4;
  k_col_gvals<<<dim3((2 * K1 * Bp + 255) / 256, U), 256, 0, st>>>(hist, K1, cols, B, Bp, G);
  k_col_corr<<<dim3(n_rows / PT, (B + PT - 1) / PT), 256, 0, st>>>(hist, U, K1, G, Bp, B, ldb,
                                                                   n_rows, Y);
}

void launch_col_out(const void* Y, int prec, int B, int ldb, int n, void* out, int out_fp64,
                    cudaStream_t st) {
  const dim3 grid((n + 31) / 32, (B + 31) / 32), block(32, 8);
  if (prec == 64) {
    if (out_fp64)
      k_col_out<double, double><<<grid, block, 0, st>>>((const double*)Y, B, ldb, n, (double*)out);
    else
      k_col_out<double, float><<<grid, block, 0, st>>>((const double*)Y, B, ldb, n, (float*)out);
  } else {
    if (out_fp64)
      k_col_out<float, double><<<grid, block, 0, st>>>((const float*)Y, B, ldb, n, (double*)out);
    else
      k_col_out<float, float><<<grid, block, 0, st>>>((const float*)Y, B, ldb, n, (float*)out);
  }
}

void launch_col_extract(const void* Y, int prec, int B, int c, int n, double* v, cudaStream_t st) {
  if (prec == 64)
    k_col_extract<double><<<(n + 255) / 256, 256, 0, st>>>((const double*)Y, B, c, n, v);
  else
    k_col_extract<float><<<(n + 255) / 256, 256, 0, st>>>((const float*)Y, B, c, n, v);
}

}  // namespace sr
