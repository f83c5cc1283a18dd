// S pass of one update by exact products of digits on the tensor cores
// (tcgen05), for S in FP64 and for the FP32 pass without a split (tc = 0):
//   S[I,J] += sum_k xi_k[I] eta_k[J]^T + eta_k[I] xi_k[J]^T  (I <= J; Alg 1).
//
// GB300 issues FP64 FMAs at 1/64 of the FP32 rate, so the FP64 pass of the CUDA
// cores (k_s_update) is bound by them: 368 us an update at n = 4,000, K = 15,
// here 42 us (35 us the pass, bound by the integer work of its epilogue, 7 us
// the operands); in FP32 at n = 8,191 83 us with FP32 FMAs, here 57 us (49 us the
// pass, 5.6 TB/s).
// Here every operand value becomes NS signed 9-bit digits, held exactly in FP16:
// v = sum_i d_i 2^-(8 + 9 i), |d_i| <= 256, i = 0 .. NS - 1, after scaling each
// term's two columns by powers of two to below one and to a common magnitude
// of the products, 2^M.  A product of digits i and j has the weight
// 2^-(16 + 9 (i + j)); the products of one weight s = i + j are summed in one FP32
// accumulator, which stays exact: (s + 1) 32 2^16 <= 2^24 at 16 terms a pass.
// Digit products with i + j >= NS are below the last weight and left out.
//   FP64: NS = 7 (62 bits), 28 products; the seven sums are added in a 64-bit
//   integer of unit 2^(M - 57) and rounded to FP64 once.
//   FP32: NS = 5 (44 bits), 15 products; the sums are added by four FP32 FMAs,
//   smallest weight first.
// FP64: what is left out or rounded before the sum with S is below 2^-55 of 2^M.
// FP32: what is left out is below 2^-37 of 2^M, each of the four FMAs rounds its
// partial sum to 2^-24, and the scaling by 2^(M - 16) is exact.  S is rounded once
// a pass of 16 terms, where an FMA chain rounds every partial sum.  All this is
// relative to 2^M, the largest product of two column maxima: entries of S far below
// it hold fewer bits than after an FMA chain.
// An infinite or NaN panel value (meta[1]) is summed by the definition instead.
//
// k_s_update_digits: one CTA per SM over the list of affected tile pairs.  Warp
// 0 loads the digits by TMA (64-byte swizzle): those of tile I, two tiles deep,
// and those of tile J in quarters of 32 columns, a ring of them.  Warp 1 issues
// the MMAs of a quarter (xi of I by eta of J, then eta by xi) into one of two
// TMEM accumulator sets, all digits of J that belong to one digit of I at once:
// N = 32 .. 224 columns; with an MMA per product (N = 32) the pass is bound by
// their issue, 50 us at n = 4,000 in FP64.  Warps 2-17 add the other set to S
// straight from TMEM, each warp 16 rows of 16 columns, with the S values of the
// next quarters already under way.  Every wait is bounded, as in k_tc.cu.
#include <cuda_fp16.h>

#include "fixed64.h"
#include "tc_util.h"

namespace sr {

namespace {

constexpr int DG_TERMS = 16;                // terms of a pass
constexpr int DG_SB = 4 * DG_TERMS;         // bytes of a digit's row: xi and eta terms
constexpr int DG_EPI = 512;                 // epilogue threads: 16 warps
constexpr int DG_THREADS = 64 + DG_EPI;     // and a warp each for TMA and MMA
constexpr int DG_NQ = 32;                   // columns of a quarter
constexpr uint32_t DG_COLS = 512;           // TMEM columns: two sets of NS * DG_NQ

// T: precision of S and the panels
template <typename T>
struct Dig {
  static constexpr bool F64 = sizeof(T) == 8;
  static constexpr int NS = F64 ? 7 : 5;     // digits
  static constexpr int TOT = 8 + 9 * (NS - 1);  // bits of a value
  static constexpr int ROWB = NS * DG_SB;    // bytes of an operand row
  static constexpr int ABYTES = PT * ROWB, BBYTES = DG_NQ * ROWB;
  static constexpr int BR = F64 ? 6 : 8;     // quarters in the ring
  static constexpr int SMEM = 2 * ABYTES + BR * BBYTES;
  static constexpr int AHEAD = F64 ? 1 : 2;  // quarters of S under way
};

// ---- operands

template <typename T>
__device__ __forceinline__ unsigned int mag_word(T v) {
  if constexpr (sizeof(T) == 8)
    return max((unsigned int)((uint64_t)__double_as_longlong(v) >> 32) & 0x7fffffffu,
               v != 0.0 ? 1u : 0u);
  else
    return __float_as_uint(v) & 0x7fffffffu;
}

// where row r of 16 is stored (see frag_row)
template <typename T>
__device__ __forceinline__ int digit_pos(int r) {
  return sizeof(T) == 8 ? r : (r & 16) + 8 * ((r >> 1) & 1) + 2 * ((r >> 2) & 3) + (r & 1);
}

// maxes[which * kc + q] = largest magnitude word of term k0 + q
template <typename T>
__global__ void __launch_bounds__(256) k_digits_max(const T* __restrict__ P, int K1, int k0, int kc,
                                                    unsigned int* __restrict__ maxes) {
  const int lane = threadIdx.x & 31, q = blockIdx.z * 8 + (threadIdx.x >> 5);
  if (q >= kc) return;
  const T* p = P + (((int64_t)blockIdx.x * 2 + blockIdx.y) * K1 + k0 + q) * PT;
  unsigned int m = 0;
#pragma unroll
  for (int u = 0; u < PT / 32; ++u) m = max(m, mag_word(p[u * 32 + lane]));
  m = __reduce_max_sync(0xffffffffu, m);
  if (lane == 0 && m) atomicMax(&maxes[blockIdx.y * kc + q], m);
}

// The digits of 32 rows (a quarter of a tile) per CTA: row a holds, digit by
// digit, [xi terms | eta terms].
template <typename T>
__global__ void __launch_bounds__(256) k_digits_pack(const T* __restrict__ P, int K1, int k0,
                                                     int kc,
                                                     const unsigned int* __restrict__ maxes,
                                                     unsigned char* __restrict__ A,
                                                     int* __restrict__ meta) {
  using D = Dig<T>;
  constexpr int PITCH = D::ROWB / 2 + 8;  // halves of a staged row
  __shared__ __align__(16) __half st[32 * PITCH];
  __shared__ int sft[2][32];  // 2^sft scales the term's column (xi, eta)
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int T0 = blockIdx.x >> 2, part = blockIdx.x & 3;
  if (warp == 0) {
    // |xi_q| < 2^ex, |eta_q| < 2^en; M = the largest ex + en
    constexpr int EB = D::F64 ? 20 : 23, BIAS = D::F64 ? 1022 : 126;
    const unsigned mx = lane < kc ? maxes[lane] : 0u, me = lane < kc ? maxes[kc + lane] : 0u;
    const bool on = mx && me;
    const int ex = max((int)(mx >> EB), 1) - BIAS, en = max((int)(me >> EB), 1) - BIAS;
    const int M = __reduce_max_sync(0xffffffffu, on ? ex + en : -100000);
    const bool bad = (int)(mx >> EB) > 2 * BIAS + 2 || (int)(me >> EB) > 2 * BIAS + 2;
    const bool any_bad = __any_sync(0xffffffffu, bad);
    const int t = on ? ex + en - M : 0;            // <= 0
    const int al = t >= 0 ? 0 : -((-t + 1) / 2);   // floor(t / 2)
    sft[0][lane] = on ? al - ex : -100000;
    sft[1][lane] = on ? (t - al) - en : -100000;
    if (blockIdx.x == 0 && lane == 0) {
      meta[0] = M > -100000 ? M : 0;
      meta[1] = any_bad ? 1 : 0;
    }
  }
  __syncthreads();
  for (int c = warp; c < 2 * DG_TERMS; c += 8) {
    const int which = c / DG_TERMS, q = c % DG_TERMS;
    long long x = 0;
    if (q < kc && sft[which][q] > -100000) {
      const T v = P[(((int64_t)T0 * 2 + which) * K1 + k0 + q) * PT + part * 32 + lane];
      // |v| 2^sft < 1: fixed_of's unit is 2^(e - 56)
      x = fixed_of(v, 56 - D::TOT - sft[which][q]);
    }
#pragma unroll
    for (int i = 0; i < D::NS; ++i) {
      constexpr int B9 = 9;
      const int sh = B9 * (D::NS - 1 - i);
      const long long d = sh ? (x + (1ll << (sh - 1))) >> sh : x;
      x -= d << sh;
      st[lane * PITCH + i * 2 * DG_TERMS + c] = __int2half_rn((int)d);
    }
  }
  __syncthreads();
  const int64_t row0 = (int64_t)T0 * PT + part * 32;
  constexpr int CH = D::ROWB / 16;  // 16-byte chunks of a row
  for (int e = threadIdx.x; e < 32 * CH; e += 256) {
    const int r = e / CH, ch = e % CH;
    *reinterpret_cast<uint4*>(A + (row0 + digit_pos<T>(r)) * D::ROWB + ch * 16) =
        *reinterpret_cast<const uint4*>(st + r * PITCH + ch * 8);
  }
}

// ---- the pass

__device__ __forceinline__ void mma_f16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc,
                                        uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_d),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}

// FP16 operands, FP32 sums, M = 128
__device__ constexpr uint32_t idesc(int N) {
  return (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(PT >> 4) << 24);
}

// K-major, 64-byte swizzle, 8-row groups 512 bytes apart, descriptor version 1
__device__ __forceinline__ uint64_t smem_desc64(uint32_t addr) {
  return (uint64_t)((addr & 0x3FFFFu) >> 4) | (uint64_t)(16u >> 4) << 16 |
         (uint64_t)(512u >> 4) << 32 | (uint64_t)1 << 46 | (uint64_t)4 << 61;
}

__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, int x, int y,
                                            int z, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(dst),
      "l"((uint64_t)map), "r"(x), "r"(y), "r"(z), "r"(bar)
      : "memory");
}

// 16 lanes x 8 columns: thread i has (row i / 4, columns 2 (i % 4) + {0, 1})
// and the same of row i / 4 + 8
__device__ __forceinline__ void tmem_ld16x8(uint32_t taddr, uint32_t (&r)[4]) {
  asm volatile("tcgen05.ld.sync.aligned.16x256b.x1.b32 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(taddr));
}

// v 2^e, in FP64's normal range, rounded to nearest
__device__ __forceinline__ double to_double(long long v, int e) {
  const uint64_t a = v < 0 ? (uint64_t)-v : (uint64_t)v;
  const int lz = __clzll((long long)a);
  const uint64_t m = a << (lz & 63);
  const uint64_t q = (m >> 11) + ((m >> 10) & 1u);  // leading one included
  const uint64_t b = (((uint64_t)(63 - lz + e + 1022) << 52) + q) |
                     ((uint64_t)v & 0x8000000000000000ull);
  return v ? __longlong_as_double((long long)b) : 0.0;
}

// A warp's 16 rows x 16 columns: element x of thread `lane` (x / 4: upper or
// lower 8 rows).  The operand rows of an FP32 pass are stored in such an order
// (digit_pos) that a thread's 4 columns of a row are adjacent, as are the
// 64 bytes of 4 threads in either precision: with a row per thread (32 lines
// per access) the passes are bound by these, 49 us (FP64, n = 4,000) and 73 us
// (FP32, n = 8,191).
template <typename T>
__device__ __forceinline__ int frag_row(int lane, int x) {
  const int r = lane >> 2, b = x >> 2;
  return sizeof(T) == 8 ? r + 8 * b : 4 * (r >> 1) + 2 * b + (r & 1);
}
template <typename T>
__device__ __forceinline__ int frag_col(int lane, int x) {
  const int q = lane & 3, c = x & 3;
  return sizeof(T) == 8 ? 2 * q + 8 * (c >> 1) + (c & 1) : 4 * q + c;
}

// the thread's elements by the definition, from the panels (an infinite or NaN
// value); out of line, it is rarely run
template <typename T>
__device__ __noinline__ void add_direct(T* out, int64_t ld, const T* __restrict__ P,
                                        const uint64_t* __restrict__ mXi,
                                        const uint64_t* __restrict__ mEta, int use_masks, int I,
                                        int J, int row0, int col0, int K1, int k0, int kc) {
  const int lane = threadIdx.x & 31;
  const uint64_t a1 = use_masks ? mXi[I] & mEta[J] : ~0ull;
  const uint64_t a2 = use_masks ? mEta[I] & mXi[J] : ~0ull;
#pragma unroll 1
  for (int e = 0; e < 8; ++e) {
    const int fr = frag_row<T>(lane, e), fc = frag_col<T>(lane, e);
    const T* pi = P + ((int64_t)I * 2 * K1 + k0) * PT + row0 + fr;
    const T* pj = P + ((int64_t)J * 2 * K1 + k0) * PT + col0 + fc;
    T x = T(0);
    for (int k = 0; k < kc; ++k) {
      const uint64_t bit = 1ull << ((k0 + k) & 63);
      if (a1 & bit) x += pi[k * PT] * pj[(K1 + k) * PT];
      if (a2 & bit) x += pi[(K1 + k) * PT] * pj[k * PT];
    }
    out[fr * ld + fc] += x;
  }
}

template <typename T>
__global__ void __launch_bounds__(DG_THREADS, 1)
    k_s_update_digits(const __grid_constant__ CUtensorMap tm_a,
                      const __grid_constant__ CUtensorMap tm_b, T* __restrict__ S, int64_t ld,
                      const uint32_t* __restrict__ tiles, const int* __restrict__ ntiles,
                      const int* __restrict__ meta, const T* __restrict__ P,
                      const uint64_t* __restrict__ mXi, const uint64_t* __restrict__ mEta,
                      int use_masks, int K1, int k0, int kc, int n, long long wait_limit,
                      unsigned long long* __restrict__ counters) {
  using D = Dig<T>;
  constexpr int NS = D::NS, NQ = DG_NQ, NH = PT / NQ, BR = D::BR;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t bar_a_full[2], bar_a_empty[2];
  __shared__ __align__(8) uint64_t bar_b_full[BR], bar_b_empty[BR];
  __shared__ __align__(8) uint64_t bar_acc_full[2], bar_acc_empty[2];
  __shared__ __align__(8) uint64_t bar_drain;
  __shared__ uint32_t tmem_base;
  __shared__ volatile int abort_flag;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t bbase = base + 2 * D::ABYTES;
  const int nt = *ntiles;
  uint32_t a_issued = 0, b_issued = 0;
  if (threadIdx.x == 0) {
    abort_flag = 0;
    for (int b = 0; b < 2; ++b) {
      mbar_init(smem_u32(&bar_a_full[b]), 1);
      mbar_init(smem_u32(&bar_a_empty[b]), 1);
      mbar_init(smem_u32(&bar_acc_full[b]), 1);
      mbar_init(smem_u32(&bar_acc_empty[b]), DG_EPI / 32);
    }
    for (int b = 0; b < BR; ++b) {
      mbar_init(smem_u32(&bar_b_full[b]), 1);
      mbar_init(smem_u32(&bar_b_empty[b]), 1);
    }
    mbar_init(smem_u32(&bar_drain), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&tmem_base)),
                 "r"(DG_COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_base;
  bool ok = true;

  if (warp == 0) {
    // ---------------- TMA producer
    if (lane == 0) {
      for (int t = blockIdx.x; t < nt && ok; t += gridDim.x) {
        const uint32_t pr = tiles[t];
        const uint32_t s = a_issued & 1u, fa = smem_u32(&bar_a_full[s]);
        if (!mbar_wait(smem_u32(&bar_a_empty[s]), ((a_issued >> 1) & 1u) ^ 1u, wait_limit,
                       &abort_flag)) {
          ok = false;
          break;
        }
        mbar_expect_tx(fa, D::ABYTES);
        tma_load_3d(base + s * D::ABYTES, &tm_a, 0, (int)(pr >> 16) * PT, 0, fa);
        ++a_issued;
        for (int h = 0; h < NH; ++h) {
          const uint32_t r = b_issued % BR, fb = smem_u32(&bar_b_full[r]);
          if (!mbar_wait(smem_u32(&bar_b_empty[r]), ((b_issued / BR) & 1u) ^ 1u, wait_limit,
                         &abort_flag)) {
            ok = false;
            break;
          }
          mbar_expect_tx(fb, D::BBYTES);
          tma_load_3d(bbase + r * D::BBYTES, &tm_b, 0, (int)(pr & 0xffffu) * PT + h * NQ, 0, fb);
          ++b_issued;
        }
      }
      if (!ok) abort_flag = 1;
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer: quarter g of the CTA accumulates in set g & 1
    if (lane == 0) {
      uint32_t it = 0, g = 0;
      for (int t = blockIdx.x; t < nt && ok; t += gridDim.x, ++it) {
        const uint32_t s = it & 1u;
        if (!mbar_wait(smem_u32(&bar_a_full[s]), (it >> 1) & 1u, wait_limit, &abort_flag)) {
          ok = false;
          break;
        }
        const uint64_t da = smem_desc64(base + s * D::ABYTES);
        for (int h = 0; h < NH; ++h, ++g) {
          const uint32_t b = g & 1u, r = g % BR;
          if (!mbar_wait(smem_u32(&bar_b_full[r]), (g / BR) & 1u, wait_limit, &abort_flag) ||
              !mbar_wait(smem_u32(&bar_acc_empty[b]), ((g >> 1) & 1u) ^ 1u, wait_limit,
                         &abort_flag)) {
            ok = false;
            break;
          }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint64_t db = smem_desc64(bbase + r * D::BBYTES);
          const uint32_t set = tmem + b * (uint32_t)(NS * NQ);
#pragma unroll
          for (int i = 0; i < NS; ++i) {
            // digit i of I by digits 0 .. NS - 1 - i of J, stored one after
            // another: N = NQ (NS - i) columns, the sums i .. NS - 1
            const uint64_t ai = da + ((i * PT * DG_SB) >> 4);
            mma_f16(set + i * NQ, ai, db + (DG_SB >> 5), idesc(NQ * (NS - i)), i ? 1u : 0u);
            mma_f16(set + i * NQ, ai + (DG_SB >> 5), db, idesc(NQ * (NS - i)), 1u);
          }
          mma_commit(smem_u32(&bar_acc_full[b]));
          mma_commit(smem_u32(&bar_b_empty[r]));
        }
        if (ok) mma_commit(smem_u32(&bar_a_empty[s]));
      }
      if (!ok) abort_flag = 1;
    }
  } else {
    // ---------------- epilogue: warps 2..17
    constexpr int AHEAD = D::AHEAD;
    const int et = threadIdx.x - 64;
    // warps w, w + 4, .. may read the TMEM lanes 32 (w % 4) ..: each takes 16 of
    // them and 16 columns
    const int row0 = (warp & 3) * 32 + ((et >> 7) & 1) * 16, col0 = (et >> 8) * 16;
    const int M = meta[0];
    const bool odd = meta[1] != 0, plain = M > -900 && M < 900;
    float sc1 = 1.f, sc2 = 1.f;  // 2^(M - 16) in two factors
    if (!D::F64) {
      sc1 = ldexpf(1.f, (M - 16) / 2);
      sc2 = ldexpf(1.f, (M - 16) - (M - 16) / 2);
    }
    const uint32_t tl = tmem + ((uint32_t)row0 << 16) + (uint32_t)col0;
    auto at = [&](uint32_t pr) {
      return S + ((int64_t)(pr >> 16) * PT + row0) * ld + (int64_t)(pr & 0xffffu) * PT + col0;
    };
    constexpr int W = 16 / (int)sizeof(T);  // elements of an access
    // the thread's elements 0 .. 3 and 4 .. 7 (8 columns from each other in FP64)
    const int off0 = frag_row<T>(lane, 0) * (int)ld + frag_col<T>(lane, 0);
    const int offr = (frag_row<T>(lane, 4) - frag_row<T>(lane, 0)) * (int)ld;
    auto off = [&](int x) { return off0 + (x >= 4 ? offr : 0) + (x % 4 ? 8 : 0); };
    T sv[AHEAD][8];
    auto fetch = [&](const T* src, T (&v)[8]) {
#pragma unroll
      for (int x = 0; x < 8; x += W)
        *reinterpret_cast<uint4*>(&v[x]) = *reinterpret_cast<const uint4*>(src + off(x));
    };
    uint32_t g = 0;
    unsigned long long my_tiles = 0, my_bytes = 0;
    int t = blockIdx.x;
    uint32_t pr = t < nt ? tiles[t] : 0u;
    if (t < nt) {
#pragma unroll
      for (int h = 0; h < AHEAD; ++h) fetch(at(pr) + h * NQ, sv[h]);
    }
    while (t < nt) {
      const int tn = t + (int)gridDim.x;
      const uint32_t prn = tn < nt ? tiles[tn] : 0u;
      const int I = (int)(pr >> 16), J = (int)(pr & 0xffffu);
      T* const srow = at(pr);
#pragma unroll
      for (int h = 0; h < NH; ++h) {
        const uint32_t b = g & 1u;
        const bool got =
            ok && mbar_wait(smem_u32(&bar_acc_full[b]), (g >> 1) & 1u, wait_limit, &abort_flag);
        ok = __all_sync(0xffffffffu, got);
        if (ok) {
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          T(&v)[8] = sv[h % AHEAD];
          T* const out = srow + h * NQ;
#pragma unroll
          for (int q = 0; q < 2; ++q) {  // 8 columns
            uint32_t a[NS][4];
#pragma unroll
            for (int w = 0; w < NS; ++w)
              tmem_ld16x8(tl + b * (uint32_t)(NS * NQ) + w * NQ + q * 8, a[w]);
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
            if (q == 1) {
              asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
              __syncwarp();
              if (lane == 0) mbar_arrive(smem_u32(&bar_acc_empty[b]));  // the warp has read it
            }
#pragma unroll
            for (int c = 0; c < 4; ++c) {
              T& o = v[(c >> 1) * 4 + q * 2 + (c & 1)];
              if constexpr (D::F64) {
                // sum_w a_w 2^(41 - 9 w), in units of 2^(M - 57)
                auto in = [&](int w) {
                  return (long long)__float2int_rn(__uint_as_float(a[w][c]));
                };
                long long x = (in(0) * (1 << 18) + in(1) * (1 << 9) + in(2)) << 23;
                x += in(3) * (1 << 14) + in(4) * (1 << 5);
                x += (in(5) * (1 << 9) + in(6) + (1 << 12)) >> 13;
                o += plain ? to_double(x, M - 57) : fixed_value_slow(x, M - 57);
              } else {
                float x = __uint_as_float(a[NS - 1][c]);
#pragma unroll
                for (int w = NS - 2; w >= 0; --w)
                  x = fmaf(x, 0.001953125f, __uint_as_float(a[w][c]));  // 2^-9
                o += x * sc1 * sc2;
              }
            }
          }
          if (odd)
            add_direct<T>(out, ld, P, mXi, mEta, use_masks, I, J, row0, col0 + h * NQ, K1, k0, kc);
          else {
#pragma unroll
            for (int x = 0; x < 8; x += W)
              *reinterpret_cast<uint4*>(out + off(x)) = *reinterpret_cast<const uint4*>(&v[x]);
          }
          if (h + AHEAD < NH)
            fetch(out + AHEAD * NQ, v);
          else if (tn < nt)
            fetch(at(prn) + (h + AHEAD - NH) * NQ, v);
        }
        ++g;
      }
      if (!ok) break;
      if (et == 0) {
        const long long vr = max(0, min(PT, n - I * PT)), vc = max(0, min(PT, n - J * PT));
        my_tiles += 1;
        my_bytes += (unsigned long long)(vr * vc) * 2ull * sizeof(T);
      }
      t = tn;
      pr = prn;
    }
    if (!ok) abort_flag = 1;
    if (et == 0 && my_tiles) {
      if (k0 == 0) {  // an update's tiles and S count once, in its first pass
        atomicAdd(&counters[CNT_TILES_TOUCHED], my_tiles);
        atomicAdd(&counters[CNT_S_BYTES], my_bytes);
      }
      atomicAdd(&counters[CNT_PANEL_BYTES],
                my_tiles * 4ull * (unsigned long long)kc * PT * sizeof(T));
    }
  }

  __syncthreads();
  if (abort_flag) {
    // copies and MMAs in flight after a stop end before shared memory and TMEM go
    if (warp == 0 && lane == 0) {
      for (uint32_t i = a_issued > 2u ? a_issued - 2u : 0u; i < a_issued; ++i)
        mbar_drain_wait(smem_u32(&bar_a_full[i & 1u]), (i >> 1) & 1u);
      for (uint32_t i = b_issued > (uint32_t)BR ? b_issued - BR : 0u; i < b_issued; ++i)
        mbar_drain_wait(smem_u32(&bar_b_full[i % BR]), (i / BR) & 1u);
    }
    if (warp == 1 && lane == 0) {
      mma_commit(smem_u32(&bar_drain));
      mbar_drain_wait(smem_u32(&bar_drain), 0u);
    }
  }
  if (threadIdx.x == 0 && abort_flag)
    atomicExch(&counters[CNT_STATUS], (unsigned long long)SR_ERR_TIMEOUT);
  if (warp == 1) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"(DG_COLS));
  }
}

// Operand rows as (64 bytes of a digit, row, digit): a box of `rows` rows lays
// its digits one after another in shared memory.
bool make_digit_map(CUtensorMap* m, const void* ptr, int n_pad, int ns, int rows) {
  EncodeFn f = encode_fn();
  if (!f) return false;
  const cuuint64_t dims[3] = {(cuuint64_t)(DG_SB / 2), (cuuint64_t)n_pad, (cuuint64_t)ns};
  const cuuint64_t strides[2] = {(cuuint64_t)(ns * DG_SB), (cuuint64_t)DG_SB};
  const cuuint32_t box[3] = {(cuuint32_t)(DG_SB / 2), (cuuint32_t)rows, (cuuint32_t)ns};
  const cuuint32_t estr[3] = {1, 1, 1};
  return f(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, const_cast<void*>(ptr), dims, strides, box, estr,
           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B,
           CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <typename T>
int digits_passes(T* S, int64_t ld, const T* P, int K1, int nT, int n_pad, const uint32_t* tiles,
                  const int* ntiles, const uint64_t* mXi, const uint64_t* mEta, int use_masks,
                  int n, unsigned char* scratch, int64_t* counters, int grid,
                  long long wait_limit, cudaStream_t st) {
  using D = Dig<T>;
  // scratch: digits | maxes (32 words) | meta
  unsigned char* A = scratch;
  unsigned int* maxes = reinterpret_cast<unsigned int*>(A + (int64_t)n_pad * D::ROWB);
  int* meta = reinterpret_cast<int*>(maxes + 32);
  CUtensorMap ma, mb;
  if (!make_digit_map(&ma, A, n_pad, D::NS, PT) || !make_digit_map(&mb, A, n_pad, D::NS, DG_NQ))
    return 2;
  const int smem = D::SMEM + 1024;
  static std::atomic<unsigned long long> done{0};
  if (smem_attr_once((const void*)k_s_update_digits<T>, smem, done) != cudaSuccess) return 1;
  for (int k0 = 0; k0 < K1; k0 += DG_TERMS) {
    const int kc = K1 - k0 < DG_TERMS ? K1 - k0 : DG_TERMS;
    cudaMemsetAsync(maxes, 0, 32 * sizeof(unsigned int), st);
    k_digits_max<T><<<dim3(nT, 2, (kc + 7) / 8), 256, 0, st>>>(P, K1, k0, kc, maxes);
    k_digits_pack<T><<<nT * 4, 256, 0, st>>>(P, K1, k0, kc, maxes, A, meta);
    k_s_update_digits<T><<<grid, DG_THREADS, smem, st>>>(
        ma, mb, S, ld, tiles, ntiles, meta, P, mXi, mEta, use_masks, K1, k0, kc, n, wait_limit,
        (unsigned long long*)counters);
  }
  return 0;
}

}  // namespace

size_t digits_scratch_bytes(int s_prec, int n_pad) {
  return (size_t)n_pad * (s_prec == 64 ? Dig<double>::ROWB : Dig<float>::ROWB) + 256;
}

int launch_s_update_digits(void* S, int s_prec, int64_t ld, const void* P, int K1, int nT,
                           int n_pad, const uint32_t* tiles, const int* ntiles,
                           const uint64_t* mXi, const uint64_t* mEta, int use_masks, int n,
                           void* scratch, int64_t* counters, int grid, long long wait_limit,
                           cudaStream_t st) {
  unsigned char* w = (unsigned char*)scratch;
  return s_prec == 64
             ? digits_passes<double>((double*)S, ld, (const double*)P, K1, nT, n_pad, tiles,
                                     ntiles, mXi, mEta, use_masks, n, w, counters, grid,
                                     wait_limit, st)
             : digits_passes<float>((float*)S, ld, (const float*)P, K1, nT, n_pad, tiles, ntiles,
                                    mXi, mEta, use_masks, n, w, counters, grid, wait_limit, st);
}

}  // namespace sr
