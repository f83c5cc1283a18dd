// One-shot batch update (rank-2r Sylvester form).  For a whole batch,
// dQ = U V^T with U = [e_{j_1} .. e_{j_r}] (the r distinct sinks) and
// V_t = Q_new[j_t,:]^T - Q[j_t,:]^T.  The proof of Thm 2 (Eq. 23-28) carries
// over column by column: Delta S = sum_k C^{k+1} Q_new^k T Q_new^kT with
// T = U W^T + W U^T, W = Q S V + U Lambda / 2, Lambda = V^T S V.  With
// V_t = a_t Q[j_t,:]^T + b_t e_{D_t} (e_{D_t} = inserted minus deleted sources
// of sink j_t) and Eq. 33 (Q S Q[j,:]^T = (S_{*,j} - (1-C) e_j) / C), W and
// Lambda need only the S rows of the batch's endpoints.  These kernels build
// W and Lambda, the panels Xi_k = C^{k+1} Q_new^k U, H_k = Q_new^k W, and the
// operand layouts of the two S-update kernels.
#include <cuda_fp16.h>

#include <algorithm>

#include "fixed64.h"
#include "sr_internal.h"

namespace sr {

namespace {

// Zc[t][a] = sum_{e in [off[t], off[t+1])} sign[e] * S[src[e], a]
template <typename T>
__global__ void k_signed_rows(const T* __restrict__ S, int64_t ld, const int32_t* __restrict__ src,
                              const int8_t* __restrict__ sign, const int64_t* __restrict__ off,
                              int n_pad, double* __restrict__ Zc, int upper) {
  const int t = blockIdx.y;
  const int a = blockIdx.x * blockDim.x + threadIdx.x;
  if (a >= n_pad) return;
  double acc = 0.0;
  for (int64_t e = off[t]; e < off[t + 1]; ++e) {
    const double v = (double)s_at(S, ld, src[e], a, upper != 0);
    acc += sign[e] > 0 ? v : -v;
  }
  Zc[(int64_t)t * n_pad + a] = acc;
}

// B[c * ldb + r] = A[r * lda + c] for r < rows, c < cols (32 x 32 tiles)
__global__ void k_transpose_rect(const double* __restrict__ A, int64_t lda, double* __restrict__ B,
                                 int64_t ldb, int rows, int cols) {
  __shared__ double tile[32][33];
  const int c0 = blockIdx.x * 32, r0 = blockIdx.y * 32;
  for (int q = threadIdx.y; q < 32; q += 8) {
    const int r = r0 + q, c = c0 + threadIdx.x;
    tile[q][threadIdx.x] = (r < rows && c < cols) ? A[(int64_t)r * lda + c] : 0.0;
  }
  __syncthreads();
  for (int q = threadIdx.y; q < 32; q += 8) {
    const int c = c0 + q, r = r0 + threadIdx.x;
    if (c < cols && r < rows) B[(int64_t)c * ldb + r] = tile[threadIdx.x][q];
  }
}

// Lambda[t][u] = V_t^T S V_u with V_t = a_t Q[j_t,:]^T + b_t e_{D_t}:
//   a_t a_u (S[j_t, j_u] - (1-C) [t == u]) / C      (Eq. 33-34)
// + a_t b_u Y[j_t][u] + b_t a_u Y[j_u][t]           (Y = Q Z, row-major)
// + b_t b_u sum_{e in D_t} sign_e Z[src_e][u]       (Z row-major)
template <typename T>
__global__ void k_lambda(const T* __restrict__ S, int64_t ld, const int32_t* __restrict__ sinks,
                         const double* __restrict__ av, const double* __restrict__ bv,
                         const double* __restrict__ Y, const double* __restrict__ Z, int64_t ldz,
                         const int32_t* __restrict__ src, const int8_t* __restrict__ sign,
                         const int64_t* __restrict__ off, int r, double C,
                         double* __restrict__ Lam, int upper) {
  const int u = blockIdx.x * blockDim.x + threadIdx.x;
  const int t = blockIdx.y;
  if (u >= r) return;
  const int jt = sinks[t], ju = sinks[u];
  const double at = av[t], au = av[u], bt = bv[t], bu = bv[u];
  double v = at * au * ((double)s_at(S, ld, jt, ju, upper != 0) - (t == u ? 1.0 - C : 0.0)) / C;
  v += at * bu * Y[(int64_t)jt * ldz + u] + bt * au * Y[(int64_t)ju * ldz + t];
  double d = 0.0;
  for (int64_t e = off[t]; e < off[t + 1]; ++e) {
    const double z = Z[(int64_t)src[e] * ldz + u];
    d += sign[e] > 0 ? z : -z;
  }
  v += bt * bu * d;
  Lam[(int64_t)t * r + u] = v;
}

// Wc[t][a] = a_t (S[j_t, a] - (1-C) [a == j_t]) / C + b_t Yc[t][a]
template <typename T>
__global__ void k_w_assemble(const T* __restrict__ S, int64_t ld, const int32_t* __restrict__ sinks,
                             const double* __restrict__ av, const double* __restrict__ bv,
                             const double* __restrict__ Yc, int n_pad, double C,
                             double* __restrict__ Wc, int upper) {
  const int t = blockIdx.y;
  const int a = blockIdx.x * blockDim.x + threadIdx.x;
  if (a >= n_pad) return;
  const int jt = sinks[t];
  const double s = (double)s_at(S, ld, jt, a, upper != 0) - (a == jt ? 1.0 - C : 0.0);
  Wc[(int64_t)t * n_pad + a] = av[t] * s / C + bv[t] * Yc[(int64_t)t * n_pad + a];
}

// Wc[t][j_u] += Lambda[u][t] / 2  (the U Lambda / 2 term of W; sinks are distinct)
__global__ void k_w_lambda(const int32_t* __restrict__ sinks, const double* __restrict__ Lam, int r,
                           int n_pad, double* __restrict__ Wc) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  const int u = blockIdx.y;
  if (t >= r) return;
  Wc[(int64_t)t * n_pad + sinks[u]] += 0.5 * Lam[(int64_t)u * r + t];
}

// X0 (row-major, ldx): X0[j_t][t] = C for the xi half (columns [0, r))
__global__ void k_xi0(const int32_t* __restrict__ sinks, int r, double C, double* __restrict__ X0,
                      int64_t ldx) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < r) X0[(int64_t)sinks[t] * ldx + t] = C;
}

// Panels for the CUDA-core S update from X_k (row-major FP64, xi half at
// column 0, eta half at column rh): term = slot * r + t of the tile-blocked
// layout P[T][which][term][128] with `terms` terms; ORs AFF bits (term % 64).
template <typename TP>
__global__ void k_pack_ffma(const double* __restrict__ X, int64_t ldx, int rh, int r, int slot,
                            int terms, int nT, TP* __restrict__ Pn, uint64_t* __restrict__ mXi,
                            uint64_t* __restrict__ mEta) {
  // block: 128 rows of tile T, threads over (row, t) with row fastest
  const int T = blockIdx.x;
  const int t = blockIdx.y * 2 + (threadIdx.x >> 7);
  const int row = threadIdx.x & 127;
  __shared__ int anyx[2], anye[2];
  if (threadIdx.x < 2) {
    anyx[threadIdx.x] = 0;
    anye[threadIdx.x] = 0;
  }
  __syncthreads();
  if (t < r) {
    const int64_t a = (int64_t)T * PT + row;
    const double x = X[a * ldx + t];
    const double e = X[a * ldx + rh + t];
    const int term = slot * r + t;
    Pn[(((int64_t)T * 2 + 0) * terms + term) * PT + row] = (TP)x;
    Pn[(((int64_t)T * 2 + 1) * terms + term) * PT + row] = (TP)e;
    if (x != 0.0) anyx[threadIdx.x >> 7] = 1;
    if (e != 0.0) anye[threadIdx.x >> 7] = 1;
  }
  __syncthreads();
  if (threadIdx.x < 2 && blockIdx.y * 2 + threadIdx.x < r) {
    const int term = slot * r + blockIdx.y * 2 + threadIdx.x;
    const unsigned long long bit = 1ull << (term & 63);
    if (anyx[threadIdx.x]) atomicOr((unsigned long long*)&mXi[T], bit);
    if (anye[threadIdx.x]) atomicOr((unsigned long long*)&mEta[T], bit);
  }
}

// Round to TF32 (10 explicit mantissa bits), round-to-nearest-even on the
// dropped 13 bits; the result is an FP32 value whose low 13 bits are zero.
__device__ __forceinline__ float tf32_round(float x) {
  uint32_t u = __float_as_uint(x);
  if ((u & 0x7f800000u) == 0x7f800000u) return x;  // inf / nan unchanged
  const uint32_t lsb = (u >> 13) & 1u;
  u += 0x0fffu + lsb;
  u &= 0xffffe000u;
  return __uint_as_float(u);
}

// Operands of the tensor-core S update from X_k: row-major A_hi, A_lo with
// kd columns; xi terms at column slot * r + t, eta terms at rg + slot * r + t.
// A value x is split as hi = tf32(x), lo = tf32(x - hi).
__global__ void k_pack_tc(const double* __restrict__ X, int64_t ldx, int rh, int r, int slot,
                          int rg, int n_rows, float* __restrict__ Ahi, float* __restrict__ Alo,
                          int64_t kd) {
  const int64_t a = blockIdx.x;
  const int t = blockIdx.y * blockDim.x + threadIdx.x;
  if (t >= r || a >= n_rows) return;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const float x = (float)X[a * ldx + h * rh + t];
    const float hi = tf32_round(x);
    const float lo = tf32_round(x - hi);
    const int64_t c = (int64_t)h * rg + (int64_t)slot * r + t;
    Ahi[a * kd + c] = hi;
    Alo[a * kd + c] = lo;
  }
}

// Tensor-core operands from tile-blocked FP32 panels [T][which][GK1][128]:
// row a of A gets xi terms at columns q < nterms and eta terms at rg + q; the
// other columns of the row are zero.  x = hi + lo, hi = tf32(x), lo = tf32(x - hi).
__global__ void k_pack_tc_tiles(const float* __restrict__ Pp, int GK1, int nterms, int rg,
                                int n_rows, float* __restrict__ Ahi, float* __restrict__ Alo,
                                int64_t kd) {
  const int64_t a = blockIdx.x;
  const int64_t ba = ((a / PT) * 2) * (int64_t)GK1 * PT + (a % PT);
  for (int c = threadIdx.x; c < kd; c += blockDim.x) {
    const int h = c >= rg ? 1 : 0;
    const int q = c - h * rg;
    float x = 0.f;
    if (q < nterms) x = Pp[ba + (int64_t)(h * GK1 + q) * PT];
    const float hi = tf32_round(x);
    Ahi[a * kd + c] = hi;
    Alo[a * kd + c] = tf32_round(x - hi);
  }
}

// Largest |value| of each pending term: maxes[which][q] over all rows (the
// bits of a non-negative float order like the float).  Block (T, which, z)
// takes terms z * 32 + [0, 32) of tile T, one warp per term at a time.
constexpr int TM_TERMS = 32;
__global__ void k_term_max(const float* __restrict__ Pp, int GK1, int nterms,
                           unsigned int* __restrict__ maxes) {
  const int T = blockIdx.x, which = blockIdx.y;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int q1 = min(nterms, (int)(blockIdx.z + 1) * TM_TERMS);
  for (int q = blockIdx.z * TM_TERMS + warp; q < q1; q += blockDim.x >> 5) {
    const float4 v = __ldcg(reinterpret_cast<const float4*>(
        Pp + (((int64_t)T * 2 + which) * GK1 + q) * PT) + lane);
    float m = fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w)));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (lane == 0 && m > 0.f) atomicMax(&maxes[which * nterms + q], __float_as_uint(m));
  }
}

// FP16 tensor-core operands from tile-blocked FP32 panels: as k_pack_tc_tiles,
// after scaling term q's xi column by 2^e_q and its eta column by 2^-e_q,
// e_q = (exponent of max|eta_q| - exponent of max|xi_q|) / 2.  The product
// xi_q eta_q^T is unchanged by the scaling (powers of two are exact) and both
// scaled columns share one magnitude, which keeps them in FP16's normal range.
// x = hi + lo, hi = fp16(x), lo = fp16(x - hi).
// Bhi / Blo (optional): the same rows with their two halves swapped, for a
// pass whose operand rows are too narrow to swap the halves by TMA box.
// Block (T, z) transposes operand columns [64 z, 64 z + 64) of the 128 rows of
// tile T through shared memory: each panel column is read as one contiguous
// 512-byte run, each operand row segment written as one 128-byte run.
constexpr int PK_COLS = 64;
__global__ void __launch_bounds__(256) k_pack_f16_tiles(
    const float* __restrict__ Pp, int GK1, int nterms, int rg, const unsigned int* __restrict__ maxes,
    __half* __restrict__ Ahi, __half* __restrict__ Alo, __half* __restrict__ Bhi,
    __half* __restrict__ Blo, int64_t kd) {
  __shared__ float tile[PK_COLS][PT + 1];
  const int T = blockIdx.x;
  const int c0 = blockIdx.y * PK_COLS;  // rg is a multiple of 32
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int cc = warp; cc < PK_COLS; cc += 8) {
    const int h = c0 + cc >= rg ? 1 : 0;
    const int q = c0 + cc - h * rg;
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (q < nterms) {
      v = __ldcs(reinterpret_cast<const float4*>(Pp + (((int64_t)T * 2 + h) * GK1 + q) * PT) +
                 lane);
      const float mx = __uint_as_float(maxes[q]), me = __uint_as_float(maxes[nterms + q]);
      if (mx > 0.f && me > 0.f) {
        const int e = (ilogbf(me) - ilogbf(mx)) / 2;
        const int sh = h ? -e : e;
        v.x = ldexpf(v.x, sh);
        v.y = ldexpf(v.y, sh);
        v.z = ldexpf(v.z, sh);
        v.w = ldexpf(v.w, sh);
      }
    }
    tile[cc][4 * lane + 0] = v.x;
    tile[cc][4 * lane + 1] = v.y;
    tile[cc][4 * lane + 2] = v.z;
    tile[cc][4 * lane + 3] = v.w;
  }
  __syncthreads();
  // warp w writes rows w, w + 8, ...: lane l the columns 2l, 2l + 1
  for (int r = warp; r < PT; r += 8) {
    const float x0 = tile[2 * lane][r], x1 = tile[2 * lane + 1][r];
    const __half h0 = __float2half_rn(x0), h1 = __float2half_rn(x1);
    const __half l0 = __float2half_rn(x0 - __half2float(h0));
    const __half l1 = __float2half_rn(x1 - __half2float(h1));
    const int c = c0 + 2 * lane;
    const int64_t o = ((int64_t)T * PT + r) * kd;
    *reinterpret_cast<__half2*>(Ahi + o + c) = __halves2half2(h0, h1);
    *reinterpret_cast<__half2*>(Alo + o + c) = __halves2half2(l0, l1);
    if (Bhi) {
      const int cb = c < rg ? c + rg : c - rg;  // rg is even: the pair stays in one half
      *reinterpret_cast<__half2*>(Bhi + o + cb) = __halves2half2(h0, h1);
      *reinterpret_cast<__half2*>(Blo + o + cb) = __halves2half2(l0, l1);
    }
  }
}

}  // namespace

void launch_signed_rows(const void* S, int s_prec, int64_t ld, const int32_t* src, const int8_t* sign,
                        const int64_t* off, int r, int n_pad, double* Zc, cudaStream_t st,
                        int upper) {
  dim3 grid((n_pad + 255) / 256, r);
  if (s_prec == 64)
    k_signed_rows<double><<<grid, 256, 0, st>>>((const double*)S, ld, src, sign, off, n_pad, Zc, upper);
  else
    k_signed_rows<float><<<grid, 256, 0, st>>>((const float*)S, ld, src, sign, off, n_pad, Zc, upper);
}

void launch_transpose_rect(const double* A, int64_t lda, double* B, int64_t ldb, int rows, int cols,
                           cudaStream_t st) {
  dim3 grid((cols + 31) / 32, (rows + 31) / 32), block(32, 8);
  k_transpose_rect<<<grid, block, 0, st>>>(A, lda, B, ldb, rows, cols);
}

void launch_lambda(const void* S, int s_prec, int64_t ld, const int32_t* sinks, const double* av,
                   const double* bv, const double* Y, const double* Z, int64_t ldz,
                   const int32_t* src, const int8_t* sign, const int64_t* off, int r, double C,
                   double* Lam, cudaStream_t st, int upper) {
  dim3 grid((r + 127) / 128, r);
  if (s_prec == 64)
    k_lambda<double><<<grid, 128, 0, st>>>((const double*)S, ld, sinks, av, bv, Y, Z, ldz, src, sign,
                                          off, r, C, Lam, upper);
  else
    k_lambda<float><<<grid, 128, 0, st>>>((const float*)S, ld, sinks, av, bv, Y, Z, ldz, src, sign,
                                         off, r, C, Lam, upper);
}

void launch_w_assemble(const void* S, int s_prec, int64_t ld, const int32_t* sinks, const double* av,
                       const double* bv, const double* Yc, const double* Lam, int r, int n_pad,
                       double C, double* Wc, cudaStream_t st, int upper) {
  dim3 grid((n_pad + 255) / 256, r);
  if (s_prec == 64)
    k_w_assemble<double><<<grid, 256, 0, st>>>((const double*)S, ld, sinks, av, bv, Yc, n_pad, C, Wc, upper);
  else
    k_w_assemble<float><<<grid, 256, 0, st>>>((const float*)S, ld, sinks, av, bv, Yc, n_pad, C, Wc, upper);
  dim3 g2((r + 127) / 128, r);
  k_w_lambda<<<g2, 128, 0, st>>>(sinks, Lam, r, n_pad, Wc);
}

void launch_xi0(const int32_t* sinks, int r, double C, double* X0, int64_t ldx, cudaStream_t st) {
  k_xi0<<<(r + 127) / 128, 128, 0, st>>>(sinks, r, C, X0, ldx);
}

void launch_pack_ffma(const double* X, int64_t ldx, int rh, int r, int slot, int terms, int nT,
                      void* Pn, int p_prec, uint64_t* mXi, uint64_t* mEta, cudaStream_t st) {
  dim3 grid(nT, (r + 1) / 2);
  if (p_prec == 64)
    k_pack_ffma<double><<<grid, 256, 0, st>>>(X, ldx, rh, r, slot, terms, nT, (double*)Pn, mXi, mEta);
  else
    k_pack_ffma<float><<<grid, 256, 0, st>>>(X, ldx, rh, r, slot, terms, nT, (float*)Pn, mXi, mEta);
}

void launch_pack_tc_tiles(const float* Pp, int GK1, int nterms, int rg, int n_rows, float* Ahi,
                          float* Alo, int64_t kd, cudaStream_t st) {
  k_pack_tc_tiles<<<n_rows, 256, 0, st>>>(Pp, GK1, nterms, rg, n_rows, Ahi, Alo, kd);
}

void launch_pack_f16_tiles(const float* Pp, int GK1, int nterms, int rg, int n_rows,
                           unsigned int* maxes, void* Ahi, void* Alo, void* Bhi, void* Blo,
                           int64_t kd, cudaStream_t st) {
  const int nT = n_rows / PT;
  cudaMemsetAsync(maxes, 0, 2 * (size_t)nterms * sizeof(unsigned int), st);
  k_term_max<<<dim3(nT, 2, (nterms + TM_TERMS - 1) / TM_TERMS), 256, 0, st>>>(Pp, GK1, nterms,
                                                                             maxes);
  k_pack_f16_tiles<<<dim3(nT, (unsigned)(kd / PK_COLS)), 256, 0, st>>>(
      Pp, GK1, nterms, rg, maxes, (__half*)Ahi, (__half*)Alo, (__half*)Bhi, (__half*)Blo, kd);
}

void launch_pack_tc(const double* X, int64_t ldx, int rh, int r, int slot, int rg, int n_rows,
                    float* Ahi, float* Alo, int64_t kd, cudaStream_t st) {
  dim3 grid(n_rows, (r + 127) / 128);
  k_pack_tc<<<grid, 128, 0, st>>>(X, ldx, rh, r, slot, rg, n_rows, Ahi, Alo, kd);
}

}  // namespace sr

namespace sr {
namespace {

// Y[row][c] += scale / len(row) * sum_{e in chunk} X[col_e][c] (Q times a
// block of columns, in FP64), for the column quads c = 4 q < ncols; Y zeroed by
// the caller.  A group of LPC lanes takes one row chunk (at most kChunk
// nonzeros), lane l of the group the quad blockIdx.y * LPC + l, so a long row
// is spread over many groups and meets in atomics.
template <int LPC>
__global__ void __launch_bounds__(256) k_spmm_chunks64(const RowChunk* __restrict__ chunks,
                                                       int64_t count,
                                                       const int32_t* __restrict__ col,
                                                       const int32_t* __restrict__ len,
                                                       const double* __restrict__ X, int64_t ldx,
                                                       double* __restrict__ Y, int64_t ldy,
                                                       int ncols, double scale) {
  const int64_t q = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / LPC;
  const int c0 = 4 * ((int)blockIdx.y * LPC + (int)(threadIdx.x % LPC));
  if (q >= count || c0 >= ncols) return;
  RowChunk ch = chunks[q];
  ch.len = chunk_len(ch);
  if (ch.len == 0) return;
  double a0 = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0;
  int e = 0;
  for (; e + 2 <= ch.len; e += 2) {
    const int b0 = __ldg(col + ch.start + e), b1 = __ldg(col + ch.start + e + 1);
    const double2* p0 = reinterpret_cast<const double2*>(X + (int64_t)b0 * ldx + c0);
    const double2* p1 = reinterpret_cast<const double2*>(X + (int64_t)b1 * ldx + c0);
    const double2 u0 = p0[0], v0 = p0[1], u1 = p1[0], v1 = p1[1];
    a0 += u0.x + u1.x;
    a1 += u0.y + u1.y;
    a2 += v0.x + v1.x;
    a3 += v0.y + v1.y;
  }
  if (e < ch.len) {
    const int b0 = __ldg(col + ch.start + e);
    const double2* p0 = reinterpret_cast<const double2*>(X + (int64_t)b0 * ldx + c0);
    const double2 u0 = p0[0], v0 = p0[1];
    a0 += u0.x;
    a1 += u0.y;
    a2 += v0.x;
    a3 += v0.y;
  }
  const double rs = scale / (double)len[ch.row];
  double* y = Y + (int64_t)ch.row * ldy + c0;
  atomicAdd(y + 0, rs * a0);
  atomicAdd(y + 1, rs * a1);
  atomicAdd(y + 2, rs * a2);
  atomicAdd(y + 3, rs * a3);
}

// Largest |value| of every term column of the one-shot block X (FP64
// [n_rows][ldx]): maxes[c] for xi column c < r, maxes[r + c] for the W column
// rh + c, as the bits of an FP32 magnitude (non-negative floats order like
// their bits).  Block (32, 8): a lane per column, 8 row phases.
__global__ void __launch_bounds__(256) k_oneshot_max(const double* __restrict__ X, int64_t ldx,
                                                     int rh, int r, int n_rows,
                                                     unsigned int* __restrict__ maxes) {
  __shared__ float red[8][32];
  const int c2 = blockIdx.x * 32 + threadIdx.x;
  float m = 0.f;
  if (c2 < 2 * r) {
    const int which = c2 >= r ? 1 : 0;
    const int64_t col = (int64_t)which * rh + (c2 - which * r);
    for (int64_t a = (int64_t)blockIdx.y * 8 + threadIdx.y; a < n_rows; a += (int64_t)gridDim.y * 8)
      m = fmaxf(m, (float)fabs(X[a * ldx + col]));
  }
  red[threadIdx.y][threadIdx.x] = m;
  __syncthreads();
  if (threadIdx.y == 0 && c2 < 2 * r) {
#pragma unroll
    for (int y = 1; y < 8; ++y) m = fmaxf(m, red[y][threadIdx.x]);
    if (m > 0.f) atomicMax(&maxes[c2], __float_as_uint(m));
  }
}

// FP16 tensor-core operands of the one-shot update from X_k: term t of the
// slot (xi column t, W column rh + t) goes to columns slot * r + t and
// rg + slot * r + t of A_hi / A_lo, after scaling the xi column by 2^e and the
// W column by 2^-e, e = (exponent of max |W_t| - exponent of max |xi_t|) / 2:
// their product is unchanged (powers of two are exact) and both share one
// magnitude inside FP16's range.  x = hi + lo, hi = fp16(x), lo = fp16(x - hi).
__global__ void k_pack_f16_oneshot(const double* __restrict__ X, int64_t ldx, int rh, int r,
                                   int slot, int rg, int n_rows,
                                   const unsigned int* __restrict__ maxes,
                                   __half* __restrict__ Ahi, __half* __restrict__ Alo, int64_t kd) {
  const int64_t a = blockIdx.x;
  const int t = blockIdx.y * blockDim.x + threadIdx.x;
  if (t >= r || a >= n_rows) return;
  const float mx = __uint_as_float(maxes[t]), me = __uint_as_float(maxes[r + t]);
  const int e = (mx > 0.f && me > 0.f) ? (ilogbf(me) - ilogbf(mx)) / 2 : 0;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const double x = ldexp(X[a * ldx + (int64_t)h * rh + t], h ? -e : e);
    const __half hi = __double2half(x);
    const __half lo = __double2half(x - (double)__half2float(hi));
    const int64_t c = (int64_t)h * rg + (int64_t)slot * r + t;
    Ahi[a * kd + c] = hi;
    Alo[a * kd + c] = lo;
  }
}

template <int LPC>
void spmm_chunks64_t(const RowChunk* chunks, int64_t count, const int32_t* col,
                     const int32_t* len, const double* X, int64_t ldx, double* Y, int64_t ldy,
                     int ncols, double scale, cudaStream_t st) {
  const int quads = ncols / 4;
  const dim3 grid((unsigned)((count * LPC + 255) / 256), (unsigned)((quads + LPC - 1) / LPC));
  k_spmm_chunks64<LPC><<<grid, 256, 0, st>>>(chunks, count, col, len, X, ldx, Y, ldy, ncols,
                                              scale);
}

}  // namespace

void launch_pack_f16_oneshot(const double* X, int64_t ldx, int rh, int r, int slot, int rg,
                             int n_rows, unsigned int* maxes, void* Ahi, void* Alo, int64_t kd,
                             cudaStream_t st) {
  cudaMemsetAsync(maxes, 0, 2 * (size_t)r * sizeof(unsigned int), st);
  const dim3 mg((unsigned)((2 * r + 31) / 32), 64), mb(32, 8);
  k_oneshot_max<<<mg, mb, 0, st>>>(X, ldx, rh, r, n_rows, maxes);
  const dim3 grid((unsigned)n_rows, (unsigned)((r + 127) / 128));
  k_pack_f16_oneshot<<<grid, 128, 0, st>>>(X, ldx, rh, r, slot, rg, n_rows, maxes, (__half*)Ahi,
                                           (__half*)Alo, kd);
}

int launch_spmm_chunks64(const RowChunk* chunks, int64_t count, const int32_t* col,
                         const int32_t* len, const double* X, int64_t ldx, double* Y, int64_t ldy,
                         int ncols, double scale, cudaStream_t st) {
  if (ncols % 4 || ldx % 2 || ldy % 2 || ((uintptr_t)X & 15)) return 1;
  if (count <= 0 || ncols <= 0) return 0;
  const int quads = ncols / 4;
  if (quads <= 8)
    spmm_chunks64_t<8>(chunks, count, col, len, X, ldx, Y, ldy, ncols, scale, st);
  else if (quads <= 16)
    spmm_chunks64_t<16>(chunks, count, col, len, X, ldx, Y, ldy, ncols, scale, st);
  else
    spmm_chunks64_t<32>(chunks, count, col, len, X, ldx, Y, ldy, ncols, scale, st);
  return 0;
}

}  // namespace sr

// ---------------------------------------------------------------------------
// The same steps in 64-bit fixed point.  A step gathers one row segment of the
// 2 r columns per nonzero; in FP64 it was bound by the FP64 adds and by the
// atomics that every row chunk made (k_spmm_chunks64, for an S that is not
// finite).  Here X holds Q^k e_j (xi without its factor C^(k+1), in [0, 1]) and
// W's columns as integers, value * 2^(56 - e): a warp takes a row chunk and 128
// columns, sums exactly, multiplies by 1 / d once and writes a row of one chunk
// directly.  The rounding of a step is 2^-57 of the largest entry of W (one exponent
// for all of its columns: a column of small entries holds fewer bits).  n = 12,000,
// m = 180,000, 2 x 190 columns: 49 us a step (10 TB/s of gathers), 260 us in FP64.
// ---------------------------------------------------------------------------
namespace sr {
namespace {

// X[j_t][t] = 1 (the xi half, zero before), X[a][rh + t] = W_t[a]
__global__ void k_os_fix(const double* __restrict__ Wc, int n_pad, int r, int rh, int e,
                         const int32_t* __restrict__ sinks, long long* __restrict__ X,
                         int64_t ldx) {
  __shared__ double tile[32][33];
  const int a0 = blockIdx.x * 32, t0 = blockIdx.y * 32;
  for (int q = threadIdx.y; q < 32; q += 8)
    tile[q][threadIdx.x] =
        t0 + q < r ? Wc[(int64_t)(t0 + q) * n_pad + a0 + threadIdx.x] : 0.0;
  __syncthreads();
  const int t = t0 + threadIdx.x;
  if (t >= r) return;
  const int j = sinks[t];
  for (int q = threadIdx.y; q < 32; q += 8) {
    const int a = a0 + q;
    X[(int64_t)a * ldx + rh + t] = fixed_of(tile[threadIdx.x][q], e);
    if (a == j) X[(int64_t)a * ldx + t] = 1ll << 56;
  }
}

// *out = max |W| as the bits of an FP32 value not below it (infinity's for an
// infinite or NaN entry)
__global__ void k_os_absmax(const double* __restrict__ W, int64_t count,
                            unsigned int* __restrict__ out) {
  unsigned int m = 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count;
       i += (int64_t)gridDim.x * blockDim.x) {
    const float v = up_abs(W[i]);
    m = max(m, v <= 3.0e38f ? __float_as_uint(v) : 0x7f800000u);
  }
  m = __reduce_max_sync(0xffffffffu, m);
  if ((threadIdx.x & 31) == 0 && m) atomicMax(out, m);
}

// Y[row] = Q X[row] for the row chunks: one warp per chunk and 128 columns (lane:
// two pairs 64 columns apart).  Rows of several chunks start at zero in Y.
__global__ void __launch_bounds__(256, 4) k_os_step(const RowChunk* __restrict__ chunks,
                                                    int64_t count,
                                                    const int32_t* __restrict__ col,
                                                    const int32_t* __restrict__ len,
                                                    const SweepScale* __restrict__ recip,
                                                    const long long* __restrict__ X,
                                                    long long* __restrict__ Y, int ldx) {
  const int lane = threadIdx.x & 31;
  const int64_t q = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
  if (q >= count) return;  // the whole warp
  const RowChunk ch = chunks[q];
  const int m = chunk_len(ch);
  const int id = lane < m ? col[ch.start + lane] : 0;
  const int c = (int)blockIdx.y * 128 + 2 * lane;
  const bool a0 = c < ldx, a1 = c + 64 < ldx;
  long long s[4] = {0, 0, 0, 0};
  for (int u = 0; u < m; u += 4) {
    longlong2 v[4][2];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int64_t x = __shfl_sync(0xffffffffu, id, u + k);
      const longlong2* p = reinterpret_cast<const longlong2*>(X + x * ldx + c);
      v[k][0] = v[k][1] = make_longlong2(0, 0);
      if (u + k < m && a0) v[k][0] = p[0];
      if (u + k < m && a1) v[k][1] = p[32];
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      s[0] += v[k][0].x;
      s[1] += v[k][0].y;
      s[2] += v[k][1].x;
      s[3] += v[k][1].y;
    }
  }
  const SweepScale f = recip[len[ch.row]];
  long long* y = Y + (int64_t)ch.row * ldx + c;
#pragma unroll
  for (int k = 0; k < 4; ++k) s[k] = m ? fixed_scale(s[k], f) : 0;
  if (ch.len & CH_ONLY) {
    if (a0) *reinterpret_cast<longlong2*>(y) = make_longlong2(s[0], s[1]);
    if (a1) *reinterpret_cast<longlong2*>(y + 64) = make_longlong2(s[2], s[3]);
  } else {
    unsigned long long* z = reinterpret_cast<unsigned long long*>(y);
    if (a0) {
      atomicAdd(z, (unsigned long long)s[0]);
      atomicAdd(z + 1, (unsigned long long)s[1]);
    }
    if (a1) {
      atomicAdd(z + 64, (unsigned long long)s[2]);
      atomicAdd(z + 65, (unsigned long long)s[3]);
    }
  }
}

// Y[row] = 0 for the rows of several chunks
__global__ void k_os_zero(const int32_t* __restrict__ rows, long long* __restrict__ Y, int ldx) {
  long long* y = Y + (int64_t)rows[blockIdx.x] * ldx;
  for (int c = threadIdx.x; c < ldx; c += blockDim.x) y[c] = 0;
}

// bits[c] = the width of the largest |entry| of column c (0: all zero)
__global__ void __launch_bounds__(256) k_os_width(const long long* __restrict__ X, int ldx,
                                                  int n_rows, unsigned int* __restrict__ bits) {
  __shared__ unsigned int red[8][32];
  const int c = blockIdx.x * 32 + threadIdx.x;
  unsigned long long m = 0;
  if (c < ldx)
    for (int64_t a = (int64_t)blockIdx.y * 8 + threadIdx.y; a < n_rows; a += (int64_t)gridDim.y * 8) {
      const long long v = X[a * ldx + c];
      m |= (unsigned long long)(v < 0 ? -v : v);
    }
  red[threadIdx.y][threadIdx.x] = 64 - __clzll((long long)m);
  __syncthreads();
  if (threadIdx.y == 0 && c < ldx) {
    unsigned int w = red[0][threadIdx.x];
#pragma unroll
    for (int y = 1; y < 8; ++y) w = max(w, red[y][threadIdx.x]);
    if (w) atomicMax(&bits[c], w);
  }
}

// One value of term t as an integer and its exponent: xi (h = 0) is
// C^(k+1) x 2^-56 with C^(k+1) = ck.r 2^-(63 + ck.sh), W (h = 1) y 2^(e - 56)
__device__ __forceinline__ long long os_entry(long long v, int h, const SweepScale& ck, int e,
                                              int& ex) {
  ex = h ? e - 56 : -61 - ck.sh;
  return h ? v : __mul64hi(v << 6, (long long)ck.r);
}

// FP16 operands as k_pack_f16_oneshot's, from the integers
__global__ void k_os_pack_f16(const long long* __restrict__ X, int64_t ldx, int rh, int r,
                              int slot, int rg, int n_rows, SweepScale ck, int e,
                              const unsigned int* __restrict__ bits, __half* __restrict__ Ahi,
                              __half* __restrict__ Alo, int64_t kd) {
  const int t = blockIdx.y * blockDim.x + threadIdx.x;
  if (t >= r) return;
  const int wx = (int)bits[t], we = (int)bits[rh + t];
  // exponents of the largest magnitudes, up to a common offset of one
  const int bal = (wx && we) ? ((we + e - 56) - (wx - 56 - (ck.sh + 1))) / 2 : 0;
  for (int64_t a = blockIdx.x; a < n_rows; a += gridDim.x) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      int ex;
      const long long v = os_entry(X[a * ldx + (int64_t)h * rh + t], h, ck, e, ex);
      // 24 bits rounded to odd, so that both roundings to FP16 are those of v
      const float x = fixed_value<float, true>(v, ex + (h ? -bal : bal));
      const __half hi = __float2half_rn(x);
      const __half lo = __float2half_rn(x - __half2float(hi));
      const int64_t c = (int64_t)h * rg + (int64_t)slot * r + t;
      Ahi[a * kd + c] = hi;
      Alo[a * kd + c] = lo;
    }
  }
}

__global__ void k_os_pack_tf32(const long long* __restrict__ X, int64_t ldx, int rh, int r,
                               int slot, int rg, int n_rows, SweepScale ck, int e,
                               float* __restrict__ Ahi, float* __restrict__ Alo, int64_t kd) {
  const int t = blockIdx.y * blockDim.x + threadIdx.x;
  if (t >= r) return;
  for (int64_t a = blockIdx.x; a < n_rows; a += gridDim.x) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      int ex;
      const long long v = os_entry(X[a * ldx + (int64_t)h * rh + t], h, ck, e, ex);
      const float x = fixed_value<float>(v, ex);
      const float hi = tf32_rne(x);
      const int64_t c = (int64_t)h * rg + (int64_t)slot * r + t;
      Ahi[a * kd + c] = hi;
      Alo[a * kd + c] = tf32_rne(x - hi);
    }
  }
}

// k_pack_ffma's panels and masks from the integers
template <typename TP>
__global__ void k_os_pack_ffma(const long long* __restrict__ X, int64_t ldx, int rh, int r,
                               int slot, int terms, SweepScale ck, int e, TP* __restrict__ Pn,
                               uint64_t* __restrict__ mXi, uint64_t* __restrict__ mEta) {
  const int T = blockIdx.x;
  const int t = blockIdx.y * 2 + (threadIdx.x >> 7);
  const int row = threadIdx.x & 127;
  if (t >= r) return;  // whole warps
  const int64_t a = (int64_t)T * PT + row;
  const int term = slot * r + t;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    int ex;
    const long long v = os_entry(X[a * ldx + (int64_t)h * rh + t], h, ck, e, ex);
    const TP x = fixed_value<TP>(v, ex);
    Pn[(((int64_t)T * 2 + h) * terms + term) * PT + row] = x;
    if (__any_sync(0xffffffffu, v != 0) && (threadIdx.x & 31) == 0)
      atomicOr((unsigned long long*)(h ? mEta : mXi) + T, 1ull << (term & 63));
  }
}

}  // namespace

void launch_os_absmax(const double* W, int64_t count, unsigned int* out, cudaStream_t st) {
  k_os_absmax<<<608, 256, 0, st>>>(W, count, out);
}

void launch_os_fix(const double* Wc, int n_pad, int r, int rh, int e, const int32_t* sinks,
                   long long* X, int64_t ldx, cudaStream_t st) {
  k_os_fix<<<dim3(n_pad / 32, (r + 31) / 32), dim3(32, 8), 0, st>>>(Wc, n_pad, r, rh, e, sinks, X,
                                                                    ldx);
}

void launch_os_step(const ChunkList& L, const int32_t* col, const int32_t* len,
                    const SweepScale* recip, const long long* X, long long* Y, int ldx,
                    cudaStream_t st) {
  if (L.multi_count > 0) k_os_zero<<<(unsigned)L.multi_count, 128, 0, st>>>(L.multi, Y, ldx);
  const dim3 grid((unsigned)((L.count + 7) / 8), (unsigned)((ldx + 127) / 128));
  k_os_step<<<grid, 256, 0, st>>>(L.chunks, L.count, col, len, recip, X, Y, ldx);
}

void launch_os_pack(const long long* X, int64_t ldx, int rh, int r, int slot, int rg, int n_rows,
                    const SweepScale& ck, int e, int f16, unsigned int* bits, void* Ahi, void* Alo,
                    int64_t kd, cudaStream_t st) {
  const dim3 grid((unsigned)std::min(n_rows, 2432), (unsigned)((r + 127) / 128));
  if (f16) {
    cudaMemsetAsync(bits, 0, (size_t)ldx * sizeof(unsigned int), st);
    k_os_width<<<dim3((unsigned)((ldx + 31) / 32), 64), dim3(32, 8), 0, st>>>(X, (int)ldx, n_rows,
                                                                              bits);
    k_os_pack_f16<<<grid, 128, 0, st>>>(X, ldx, rh, r, slot, rg, n_rows, ck, e, bits,
                                        (__half*)Ahi, (__half*)Alo, kd);
  } else {
    k_os_pack_tf32<<<grid, 128, 0, st>>>(X, ldx, rh, r, slot, rg, n_rows, ck, e, (float*)Ahi,
                                         (float*)Alo, kd);
  }
}

void launch_os_pack_ffma(const long long* X, int64_t ldx, int rh, int r, int slot, int terms,
                         int nT, const SweepScale& ck, int e, void* Pn, int p_prec, uint64_t* mXi,
                         uint64_t* mEta, cudaStream_t st) {
  const dim3 grid(nT, (r + 1) / 2);
  if (p_prec == 64)
    k_os_pack_ffma<double><<<grid, 256, 0, st>>>(X, ldx, rh, r, slot, terms, ck, e, (double*)Pn,
                                                 mXi, mEta);
  else
    k_os_pack_ffma<float><<<grid, 256, 0, st>>>(X, ldx, rh, r, slot, terms, ck, e, (float*)Pn, mXi,
                                                mEta);
}

}  // namespace sr
