// Everything one rank-one (sink-block) update does before its S pass, in one
// cooperative launch:
//   phase 0  graph patch (Thm 1: row j of the in-adjacency gains / loses the
//            sources I); the rows of the current S that gamma reads,
//            sI = sum_t S[I_t, *] and sJ = S[j, *], with the panels of updates
//            whose S pass is still pending added in; per-tile nonzero counts;
//   phase 1  w = Q sI (the SpMV of Thm 3's preprocessing), then gamma (Thm 3
//            insert, Thm 9 delete, Table 2 sink blocks) as eta_0, with
//            xi_0 = C e_j;
//   phase 2  the K steps of the recurrence on the new graph (Eq. 16a),
//            xi_{k+1} = C Q xi_k, eta_{k+1} = Q eta_k;
//   phase 3  the affected-area mask words of every tile (Thm 4) and the list
//            of affected tile pairs of the S pass.
// A bounded grid barrier follows phase 0 and comes before the tile list; what lies
// between waits on counted words (flow form) or on further barriers (item form).
//
// Flow form (default).  The in-lists of all rows, flattened in row order, are
// cut into equal contiguous ranges, one per CTA, one or two nonzeros per
// thread, located once per launch.  Steps are not separated by barriers: a word
// of W[k + 1] counts, in its upper bits, the parts of its row's sum that are
// there, and a thread that gathers it reads it (from L2) until all are.  A step
// then costs one reduction and one load through L2 instead of a reduction, a grid
// barrier and a load.  At n = 20,000, m = 200,000 a step takes 2.5 us (with
// barriers 4.8 in FP64, 2.9 in FP32), at n = 1,000, m = 8,000 1.55 us (2.95 and
// 2.0): about half of it the L2 latency there and back, the rest the gather
// (one 32-byte sector per nonzero and SM every other clock) and the sums.
// w and gamma go the same way (gamma's rows wait for the parts of their means).
// Outside the steps an update costs 25 us at n = 20,000 and 20 us at n = 1,000
// (27 and 21 with a grid barrier after w and a gather of every column's extent):
// round trips to L2 that depend on each other.
// Every CTA is co-resident and a value depends on earlier steps only, so the
// waits end; they are bounded all the same.
// The vectors are kept in 64-bit fixed point (xi without its factor C^(k+1),
// in [0, 1], as value * 2^56; eta as value * 2^(56 - e), |eta| < 2^e from the
// largest entry of the rows that gamma reads): row sums are exact, and the
// division by the in-degree is a product with a 63-bit reciprocal.  GB300
// issues FP64 (and conversions to and from 64-bit types) at 1/64 of the FP32
// rate, which took 1.65 us of each step in FP64.  The error is absolute, 2^-57 of
// the largest entry a step.  An FP64 S rounds its entries above 2^-4 more than
// that; smaller entries of xi and eta hold fewer bits than in FP64 (below 2^-33 of
// the largest fewer than in FP32), and those that round to zero leave the masks.
// A row spread over the lanes of a warp is summed by shuffles, over the warps
// of a CTA through shared memory, and the parts of a row cut by the CTA ranges
// meet in its word by integer reductions.
//
// Item form (a set `item`, more than two nonzeros per thread, or an infinite or
// NaN S).  Every 128-row tile is cut into items of at most `item` flattened
// nonzeros, and items go round-robin to the CTAs (a hub row with thousands of
// in-neighbours spreads over many SMs); each CTA keeps the row extents and
// column indices of its first items in shared memory for all K steps.  Partial
// row sums are combined within a warp and added to the next column with global
// atomics, and a grid barrier ends each step.  The vectors and the arithmetic
// are FP64 (vec64 = 1, or S in FP64) or FP32.
//
// In both forms xi_k and eta_k are interleaved in the working buffer W[k][a]
// (one load per nonzero), and row-wise work (gamma; the copy of the columns into
// the tile-blocked panels that the S pass reads, with the masks) goes by tiles,
// round-robin.
//
// gamma needs w on the OLD graph; only row j of Q changes, so the kernel
// gathers on the patched graph and corrects row j: the sum over the old
// in-neighbours = the sum over the new ones - op * S_II.
//
// The panels the S pass reads have the precision of S; gamma has that of the
// vectors, its row j and lambda are always FP64.  The correction of the rows of S
// by pending panels is summed in the precision of S (those panels are stored in
// it).  The atomic accumulation of the item form makes the last bit of a result
// depend on the order of the additions.
#include <algorithm>

#include "fixed64.h"
#include "fx64.h"
#include "sr_internal.h"

namespace sr {

namespace {

constexpr int PG = 512;     // threads of a prep CTA
constexpr int PREP_MT = 8;  // tiles one CTA may own for row-wise work
constexpr int MAXI = 6;     // items whose row extents stay in shared memory

template <typename V>
struct V2 {
  V x, y;
};

struct alignas(16) PrepItem {
  int64_t start[PT];
  int len[PT];
  int off[PT + 1];
  int T;       // tile
  int e0, e1;  // flattened nonzeros [e0, e1) of the tile
  int cbase;   // nonzeros [e0, e0 + clen) have their column index at cc[cbase ...]
  int clen;
};

__device__ __forceinline__ unsigned int ld_acquire(const unsigned int* p) {
  unsigned int v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Grid barrier on a monotonically increasing arrival counter: barrier number
// b of a launch returns once b * gridDim.x arrivals are visible.  Bounded:
// false after `limit` polls.  The arrival is a release reduction (it orders
// the CTA's earlier writes, made visible to thread 0 by the CTA barrier, before
// it) and the polls are acquire loads, so after the final CTA barrier plain
// (L1-cached) loads of every thread see every CTA's writes from before the
// barrier.
__device__ __forceinline__ bool prep_barrier(unsigned int* count, unsigned int target,
                                             long long limit, int* s_ok) {
  __syncthreads();
  if (threadIdx.x == 0) {
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(count) : "memory");
    int ok = 1;
    long long it = 0;
    while (ld_acquire(count) < target) {
      if (++it > limit) {
        ok = 0;
        break;
      }
      __nanosleep(16);
    }
    *s_ok = ok;
  }
  __syncthreads();
  return *s_ok != 0;
}

__device__ __forceinline__ void red_add(float* p, float v) {
  asm volatile("red.relaxed.gpu.global.add.f32 [%0], %1;" ::"l"(p), "f"(v) : "memory");
}
__device__ __forceinline__ void red_add(double* p, double v) {
  asm volatile("red.relaxed.gpu.global.add.f64 [%0], %1;" ::"l"(p), "d"(v) : "memory");
}
__device__ __forceinline__ void red_add2(V2<float>* p, float x, float y) {
  asm volatile("red.relaxed.gpu.global.add.v2.f32 [%0], {%1, %2};" ::"l"(p), "f"(x), "f"(y)
               : "memory");
}
__device__ __forceinline__ void red_add2(V2<double>* p, double x, double y) {
  red_add(&p->x, x);
  red_add(&p->y, y);
}
// x != 0 on the integer pipe (GB300 issues FP64 compares at the FP64 rate)
__device__ __forceinline__ bool nz(float x) { return (__float_as_uint(x) << 1) != 0u; }
__device__ __forceinline__ bool nz(double x) {
  return ((unsigned long long)__double_as_longlong(x) << 1) != 0ull;
}
// Gathers of the working vectors go through L1: a column with a large
// out-degree is read by many rows of the same CTA.  Each W[k] is written (by
// atomics, in L2) only in the step before the one that reads it, with a grid
// barrier between, so no L1 line can be stale.
__device__ __forceinline__ V2<float> ld_v2(const V2<float>* p) {
  const float2 v = *reinterpret_cast<const float2*>(p);
  return V2<float>{v.x, v.y};
}
__device__ __forceinline__ V2<double> ld_v2(const V2<double>* p) {
  const double2 v = *reinterpret_cast<const double2*>(p);
  return V2<double>{v.x, v.y};
}

__device__ __forceinline__ V2<float> ld_v2cg(const V2<float>* p) {
  const float2 v = __ldcg(reinterpret_cast<const float2*>(p));
  return V2<float>{v.x, v.y};
}
__device__ __forceinline__ V2<double> ld_v2cg(const V2<double>* p) {
  const double2 v = __ldcg(reinterpret_cast<const double2*>(p));
  return V2<double>{v.x, v.y};
}

// Row extents of tile T (after the patch) and the exclusive scan of their lengths.
__device__ __forceinline__ void item_rows_load(const DevAdj& in, int T, PrepItem& it) {
  const int tid = threadIdx.x;
  if (tid < PT) {
    it.start[tid] = __ldcg(in.start + (int64_t)T * PT + tid);
    it.len[tid] = __ldcg(in.len + (int64_t)T * PT + tid);
  }
  __syncthreads();
  if (tid < 32) {
    int v[4], sum = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      v[q] = it.len[tid * 4 + q];
      sum += v[q];
    }
    int incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, incl, o);
      if (tid >= o) incl += y;
    }
    int run = incl - sum;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      it.off[tid * 4 + q] = run;
      run += v[q];
    }
    if (tid == 31) it.off[PT] = incl;
  }
  __syncthreads();
}

// Item q of the launch: its tile (the last T with ioff[T] <= q) and range.
__device__ __forceinline__ void item_locate(const DevAdj& in, const int* ioff, int nT, int q,
                                            int item, PrepItem& it) {
  int lo = 0, hi = nT;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (ioff[mid] <= q) lo = mid; else hi = mid;
  }
  item_rows_load(in, lo, it);
  if (threadIdx.x == 0) {
    it.T = lo;
    it.e0 = (q - ioff[lo]) * item;
    it.e1 = min(it.off[PT], it.e0 + item);
    it.cbase = 0;
    it.clen = 0;
  }
  __syncthreads();
}

// Combines per-lane partials of equal row keys across a warp (keys are
// non-decreasing with the lane; key < 0 = nothing) and hands each segment's
// nonzero total to emit(key, a, b) once.
template <typename V, typename Emit>
__device__ __forceinline__ void seg_emit(int key, V a, V b, Emit emit) {
  const int lane = threadIdx.x & 31;
  // only as many rounds as the longest run of equal keys needs
  const unsigned same = __match_any_sync(0xffffffffu, key);
  const int span = (int)__reduce_max_sync(0xffffffffu, key >= 0 ? (unsigned)__popc(same) : 1u);
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    if (o >= span) break;
    const int k2 = __shfl_down_sync(0xffffffffu, key, o);
    const V xa = __shfl_down_sync(0xffffffffu, a, o);
    const V xb = __shfl_down_sync(0xffffffffu, b, o);
    if (lane + o < 32 && k2 == key) {
      a += xa;
      b += xb;
    }
  }
  const int kprev = __shfl_up_sync(0xffffffffu, key, 1);
  if (key >= 0 && (lane == 0 || kprev != key) && (nz(a) || nz(b))) emit(key, a, b);
}

// One thread's contiguous run [e0, e1) of an item's nonzeros (flattened order
// of the tile) and the row r holding e0 (r = -1: empty run).  The same for
// every step, so the step loop computes it once for the CTA's first item.
struct Run {
  int e0, e1, r;
};

__device__ __forceinline__ Run item_run(const PrepItem& it) {
  const int n_e = it.e1 - it.e0;
  const int per = (n_e + PG - 1) / PG;
  Run u;
  u.e0 = it.e0 + (int)threadIdx.x * per;
  u.e1 = min(it.e1, u.e0 + per);
  u.r = -1;
  if (u.e0 < u.e1) {
    int lo = 0, hi = PT;
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (it.off[mid] <= u.e0) lo = mid; else hi = mid;
    }
    u.r = lo;
  }
  return u;
}

// Sums gather(b) over the nonzeros of the item's tile, per row, and calls
// emit(r, a, b) with each row's (partial) sums.  Each thread takes its run; a
// row wholly inside one run is emitted by that thread, the first and last row
// of a run go through seg_emit.
template <typename V, typename Gf, typename Emit>
__device__ __forceinline__ void item_gather(const PrepItem& it, const Run& run,
                                            const int* __restrict__ cc,
                                            const int32_t* __restrict__ col, Gf gather,
                                            Emit emit) {
  const int e0 = run.e0, e1 = run.e1;
  int r_first = -1, r_last = -1;
  V fa = V(0), fb = V(0), la = V(0), lb = V(0);
  if (run.r >= 0) {
    int r = run.r;
    r_first = r;
    V pa = V(0), pb = V(0);
    constexpr int B = sizeof(V) == 8 ? 4 : 8;
    for (int e = e0; e < e1; e += B) {
      int rr[B], bb[B];
      int rc = r;
#pragma unroll
      for (int q = 0; q < B; ++q) {
        const int ee = e + q;
        if (ee < e1) {
          while (ee >= it.off[rc + 1]) ++rc;
          rr[q] = rc;
          const int ce = ee - it.e0;
          bb[q] = (ce < it.clen) ? cc[it.cbase + ce]
                                 : __ldcg(col + it.start[rc] + (ee - it.off[rc]));
        } else {
          rr[q] = -1;
          bb[q] = 0;
        }
      }
      V2<V> xv[B];
#pragma unroll
      for (int q = 0; q < B; ++q) xv[q] = (rr[q] >= 0) ? gather(bb[q]) : V2<V>{V(0), V(0)};
#pragma unroll
      for (int q = 0; q < B; ++q) {
        if (rr[q] < 0) break;
        if (rr[q] != r) {
          if (r == r_first) {
            fa = pa;
            fb = pb;
          } else if (nz(pa) || nz(pb)) {
            emit(r, pa, pb);  // row wholly inside this run
          }
          pa = pb = V(0);
          r = rr[q];
        }
        pa += xv[q].x;
        pb += xv[q].y;
      }
    }
    if (r == r_first) {
      fa = pa;
      fb = pb;
    } else {
      r_last = r;
      la = pa;
      lb = pb;
    }
  }
  seg_emit<V>(r_first, fa, fb, emit);
  seg_emit<V>(r_last, la, lb, emit);
}

// A step over an item of at most 2 * PG nonzeros gives each thread at most two
// of them, so a thread's part of every step is fixed by the graph: its columns,
// the rows they fall in (head = row of the first; tail = row of the second
// when it differs) and the shuffle pattern of the warp that adds up the rows
// spread over several lanes.  StepPair holds that, set up once per launch.
template <typename V>
struct StepPair {
  int ca, cb;    // columns of the nonzeros (-1: none)
  int kh, kt;    // head / tail row in the tile (-1: none)
  int span;      // warp-uniform: the longest run of lanes sharing a head row
  unsigned fl;   // bits 0-4: take lane + 2^b's head sum; 5: add lane - 1's tail;
                 // 6: emit the head sum; 7: emit the tail sum; 8-12: the first lane
                 // of the head row's run of lanes
};

template <typename V>
__device__ __forceinline__ void pair_pattern(StepPair<V>& q);

template <typename V>
__device__ __forceinline__ StepPair<V> pair_setup(const PrepItem& it, const int* __restrict__ cc,
                                                  const int32_t* __restrict__ col) {
  const Run run = item_run(it);
  StepPair<V> q;
  q.ca = q.cb = q.kh = q.kt = -1;
  auto column = [&](int e, int r) {
    const int ce = e - it.e0;
    return (ce < it.clen) ? cc[it.cbase + ce] : __ldcg(col + it.start[r] + (e - it.off[r]));
  };
  if (run.r >= 0) {
    q.kh = run.r;
    q.ca = column(run.e0, q.kh);
    if (run.e1 - run.e0 == 2) {
      int r2 = q.kh;
      while (run.e0 + 1 >= it.off[r2 + 1]) ++r2;
      q.cb = column(run.e0 + 1, r2);
      if (r2 != q.kh) q.kt = r2;
    }
  }
  pair_pattern(q);
  return q;
}

// The warp-wide pattern of a step for threads whose (ca, cb, kh, kt) are set:
// row keys must not decrease with the lane.
template <typename V>
__device__ __forceinline__ void pair_pattern(StepPair<V>& q) {
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  // every lane takes part in the warp-wide intrinsics below
  const unsigned same = __match_any_sync(full, q.kh);
  const int seg = (q.kh >= 0) ? __popc(same) : 1;
  q.span = __reduce_max_sync(full, (unsigned)seg);
  // a segment's lanes are consecutive (row keys do not decrease with the lane):
  // a tree over the segment that leaves the total in its first lane only adds,
  // in round b, the partial of lane + 2^b into the lanes at positions 0 mod
  // 2^(b+1), so a segment of s lanes costs s - 1 additions
  const int pos = lane - (__ffs(same) - 1);
  q.fl = (unsigned)(__ffs(same) - 1) << 8;
#pragma unroll
  for (int b = 0; b < 5; ++b) {
    const int k2 = __shfl_down_sync(full, q.kh, 1 << b);
    if (lane + (1 << b) < 32 && k2 == q.kh && q.kh >= 0 && (pos & ((2 << b) - 1)) == 0)
      q.fl |= 1u << b;
  }
  const int kt_prev = __shfl_up_sync(full, q.kt, 1);
  const int kh_prev = __shfl_up_sync(full, q.kh, 1);
  const int kh_next = __shfl_down_sync(full, q.kh, 1);
  if (lane > 0 && q.kh >= 0 && kt_prev == q.kh) q.fl |= 1u << 5;
  if (q.kh >= 0 && (lane == 0 || kh_prev != q.kh)) q.fl |= 1u << 6;
  if (q.kt >= 0 && !(lane < 31 && kh_next == q.kt)) q.fl |= 1u << 7;
}

// One step of the recurrence for a thread set up by pair_setup: gathers its
// (xi_k, eta_k) entries, adds the rows up across the warp and emits each row's
// sum (times C / in-degree for xi, 1 / in-degree for eta; rc / ri hold those
// factors per row of the item's tile) into W[k + 1].
template <typename Gf, typename Emit>
__device__ __forceinline__ void pair_step_fx(const StepPair<double>& q, Gf gather, Emit emit);

template <typename V, typename Gf, typename Emit>
__device__ __forceinline__ void pair_step(const StepPair<V>& q, Gf gather, Emit emit) {
  if constexpr (sizeof(V) == 8) {
    pair_step_fx(q, gather, emit);
    return;
  }
  const unsigned full = 0xffffffffu;
  V ha = V(0), hb = V(0), ta = V(0), tb = V(0);
  if (q.ca >= 0) {
    const V2<V> v = gather(q.ca);
    ha = v.x;
    hb = v.y;
  }
  if (q.cb >= 0) {
    const V2<V> v = gather(q.cb);
    if (q.kt >= 0) {
      ta = v.x;
      tb = v.y;
    } else {
      ha += v.x;
      hb += v.y;
    }
  }
#pragma unroll
  for (int b = 0; b < 5; ++b) {
    if ((1 << b) >= q.span) break;
    const V xa = __shfl_down_sync(full, ha, 1 << b);
    const V xb = __shfl_down_sync(full, hb, 1 << b);
    if (q.fl & (1u << b)) {
      ha += xa;
      hb += xb;
    }
  }
  const V pa = __shfl_up_sync(full, ta, 1);
  const V pb = __shfl_up_sync(full, tb, 1);
  if (q.fl & (1u << 5)) {
    ha += pa;
    hb += pb;
  }
  if ((q.fl & (1u << 6)) && (nz(ha) || nz(hb))) emit(q.kh, ha, hb);
  if ((q.fl & (1u << 7)) && (nz(ta) || nz(tb))) emit(q.kt, ta, tb);
}

// Exact row sums of FP64 values on the integer pipe (fx64.h): the values of
// one row's run of lanes (at most 65: two per lane and an incoming tail, so
// below 2^63 in total) are turned into 64-bit fixed-point numbers with 55
// fraction bits below the run's largest binary exponent, added exactly, and
// the total is rounded to FP64 once.  The error stays below 65 * 2^-55 of the
// largest value, where FP64 additions in any order can lose (n - 1) 2^-53 of
// the sum of the magnitudes.
// pair_step for FP64 vectors with the row sums formed exactly as above: the
// run's largest exponent goes through the same shuffle tree (integer max) and
// back to every lane of the run from its first lane, then the fixed-point
// values through the tree (integer adds).  A tail that ends its row in this
// lane is one value and is emitted as it is.
template <typename Gf, typename Emit>
__device__ __forceinline__ void pair_step_fx(const StepPair<double>& q, Gf gather, Emit emit) {
  const unsigned full = 0xffffffffu;
  double h1x = 0.0, h1y = 0.0, h2x = 0.0, h2y = 0.0, tx = 0.0, ty = 0.0;
  if (q.ca >= 0) {
    const V2<double> v = gather(q.ca);
    h1x = v.x;
    h1y = v.y;
  }
  if (q.cb >= 0) {
    const V2<double> v = gather(q.cb);
    if (q.kt >= 0) {
      tx = v.x;
      ty = v.y;
    } else {
      h2x = v.x;
      h2y = v.y;
    }
  }
  // lane - 1's tail, added into this lane's head row (bit 5)
  double px = __shfl_up_sync(full, tx, 1), py = __shfl_up_sync(full, ty, 1);
  if (!(q.fl & (1u << 5))) px = py = 0.0;
  int ex = max(max(fx_exp(h1x), fx_exp(h2x)), fx_exp(px));
  int ey = max(max(fx_exp(h1y), fx_exp(h2y)), fx_exp(py));
#pragma unroll
  for (int b = 0; b < 5; ++b) {
    if ((1 << b) >= q.span) break;
    const int xe = __shfl_down_sync(full, ex, 1 << b);
    const int ye = __shfl_down_sync(full, ey, 1 << b);
    if (q.fl & (1u << b)) {
      ex = max(ex, xe);
      ey = max(ey, ye);
    }
  }
  const int first = (int)((q.fl >> 8) & 31u);
  ex = __shfl_sync(full, ex, first);
  ey = __shfl_sync(full, ey, first);
  long long fx = fx_of(h1x, ex) + fx_of(h2x, ex) + fx_of(px, ex);
  long long fy = fx_of(h1y, ey) + fx_of(h2y, ey) + fx_of(py, ey);
#pragma unroll
  for (int b = 0; b < 5; ++b) {
    if ((1 << b) >= q.span) break;
    const long long xa = __shfl_down_sync(full, fx, 1 << b);
    const long long xb = __shfl_down_sync(full, fy, 1 << b);
    if (q.fl & (1u << b)) {
      fx += xa;
      fy += xb;
    }
  }
  if ((q.fl & (1u << 6)) && (fx != 0 || fy != 0)) emit(q.kh, fx_value(fx, ex), fx_value(fy, ey));
  if ((q.fl & (1u << 7)) && (nz(tx) || nz(ty))) emit(q.kt, tx, ty);
}

// ---- flow form

struct I2 {
  long long x, y;
};
// A word of W[k] holds, above a sum v, |v| < 2^57, a count in its top 6 bits that
// is FLOW_FULL once all parts of the sum are there: the part with the row's
// first nonzero counts for the others that are missing (FLOW_FULL + 1 - parts),
// each other one for 1.  So a reader needs to know nothing of the row (the
// extents of the gathered rows cost 3 us of an update at n = 20,000), and a row
// without nonzeros is complete from the start.
constexpr int FLOW_CNT = 58;
constexpr int FLOW_CTA = 256;   // nonzeros per CTA while co-resident CTAs are left
constexpr int FLOW_PARTS = 60;  // parts a row may have
constexpr unsigned FLOW_FULL = 63;
constexpr long long FLOW_DONE = (long long)((unsigned long long)FLOW_FULL << FLOW_CNT);

__device__ __forceinline__ I2 ld_flow(const I2* p) {
  I2 v;
  asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];" : "=l"(v.x), "=l"(v.y) : "l"(p)
               : "memory");
  return v;
}
// A first look, which may be served by L1 (other warps of the CTA gather the same
// entries): a line fetched too early shows too few parts and is read again from
// L2.  Nothing older than the zeros of this launch can be there: the grid
// barrier after them ordered them before every later read.
__device__ __forceinline__ I2 look_flow(const I2* p) {
  I2 v;
  asm volatile("ld.relaxed.cta.global.v2.b64 {%0, %1}, [%2];" : "=l"(v.x), "=l"(v.y) : "l"(p)
               : "memory");
  return v;
}
// A row's sum, or one part of it, into its word.  A reduction also where a store
// would do: it reached the readers 0.25 us sooner (a step 2.9 -> 2.6 us).
__device__ __forceinline__ void put_flow1(long long* p, long long v, unsigned w) {
  asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(p),
               "l"((unsigned long long)v + ((unsigned long long)w << FLOW_CNT))
               : "memory");
}
__device__ __forceinline__ void put_flow(I2* p, const I2& v, unsigned w) {
  put_flow1(&p->x, v.x, w);
  put_flow1(&p->y, v.y, w);
}
__device__ __forceinline__ long long ld_flow1(const long long* p) {
  long long v;
  asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
// Whether all parts are there (the count is in the upper half's top bits)
__device__ __forceinline__ bool flow_there(long long v) {
  return (((unsigned)((unsigned long long)v >> 32) + (1u << (FLOW_CNT - 33))) >>
          (FLOW_CNT - 32)) == FLOW_FULL;
}
__device__ __forceinline__ bool flow_there(const I2& v) {
  return flow_there(v.x) && flow_there(v.y);
}

// x / per for 0 <= x < 2^24 (inv = 1 / per)
__device__ __forceinline__ int flow_div(int x, int per, float inv) {
  int q = (int)((float)x * inv);
  if (q * per > x) --q;
  if ((q + 1) * per <= x) ++q;
  return q;
}

// What the part of nonzeros e0 .. counts for of a row with the nonzeros
// rs .. rs + len - 1, cut at the multiples of per.
__device__ __forceinline__ unsigned flow_weight(int rs, int len, int e0, int per, float inv) {
  return rs < e0 ? 1u
                 : FLOW_FULL - (unsigned)(flow_div(rs + len - 1, per, inv) - flow_div(rs, per, inv));
}

// v without its count
__device__ __forceinline__ void flow_strip(I2& v) {
  v.x -= FLOW_DONE;
  v.y -= FLOW_DONE;
}

// Adds up the runs of lanes sharing a row: head sums to the first lane of their
// run, a tail into the next lane's head when that holds the same row.  At most
// 65 values below 2^56 each.
template <typename V>
__device__ __forceinline__ void flow_sum(const StepPair<V>& q, I2& h, const I2& t) {
  constexpr unsigned full = 0xffffffffu;
#pragma unroll
  for (int b = 0; b < 5; ++b) {
    if ((1 << b) >= q.span) break;
    const long long x = __shfl_down_sync(full, h.x, 1 << b);
    const long long y = __shfl_down_sync(full, h.y, 1 << b);
    if (q.fl & (1u << b)) {
      h.x += x;
      h.y += y;
    }
  }
  const long long x = __shfl_up_sync(full, t.x, 1), y = __shfl_up_sync(full, t.y, 1);
  if (q.fl & (1u << 5)) {
    h.x += x;
    h.y += y;
  }
}

// out[d] = 1 / d, r = 2^(62 + L) / d rounded to nearest with 2^(L-1) < d <= 2^L;
// d <= 64: sums of d values below 2^56 may be shifted left by h = 6 - L
__global__ void k_flow_recip(SweepScale* __restrict__ out, int count) {
  const int d = blockIdx.x * blockDim.x + threadIdx.x;
  if (d >= count) return;
  SweepScale f{0ull, 0, 1};
  if (d > 0) {
    const int L = d > 1 ? 32 - __clz(d - 1) : 0;
    const unsigned long long u = (unsigned long long)d;
    if (L == 0) {
      f.r = 1ull << 62;
    } else {
      const unsigned long long q0 = (1ull << 63) / u, r0 = (1ull << 63) % u;
      const unsigned long long m = r0 << (L - 1);
      f.r = (q0 << (L - 1)) + m / u + (2ull * (m % u) >= u ? 1ull : 0ull);
    }
    f.h = max(0, 6 - L);
    f.sh = (L - 1) + f.h - 1;  // 1 / d = r 2^-(63 + L - 1)
  }
  out[d] = f;
}

__device__ void prep_patch(const PatchOp* __restrict__ ops, int64_t begin, int64_t end,
                           const DevAdj& in, const DevAdj& out) {
  for (int64_t o = begin; o < end; ++o) {
    const PatchOp op = ops[o];
    if (op.kind == PK_IN_COPY || op.kind == PK_OUT_COPY) {
      int32_t* c = (op.kind == PK_IN_COPY) ? in.col : out.col;
      for (int e = threadIdx.x; e < op.v; e += blockDim.x) c[op.a + e] = c[op.b + e];
      __syncthreads();
      continue;
    }
    if (threadIdx.x == 0) {
      switch (op.kind) {
        case PK_IN_COL: in.col[op.a] = op.v; break;
        case PK_OUT_COL: out.col[op.a] = op.v; break;
        case PK_IN_LEN: in.len[op.a] = op.v; break;
        case PK_OUT_LEN: out.len[op.a] = op.v; break;
        case PK_IN_START: in.start[op.a] = op.b; break;
        case PK_OUT_START: out.start[op.a] = op.b; break;
        default: break;
      }
    }
    __syncthreads();
  }
}

// Shared memory of the flow form, in the place of the item form's column cache
// (as arrays of their own they took the second CTA of an SM from launches with more
// than 2,270 pending terms, 2,590 with FP32 vectors; now 3,580 and 3,900, at
// n = 20,000).  fsh also holds the partial sums of phase 0.
struct FlowShared {
  SweepScale fsh[PG][2];  // 1 / in-degree of each thread's head / tail row
  int rowmap[2 * PG];     // the row of each of the CTA's nonzeros
  I2 dep[2][PG / 32];     // a warp's part of the row before it
};
constexpr int FLOW_INTS = (int)(sizeof(FlowShared) / sizeof(int));
static_assert(FLOW_INTS % 4 == 0 && sizeof(PrepItem) % 16 == 0, "16-byte alignment");

// V: arithmetic and vector precision; TS: storage precision of S and the panels.
// FLOW: the flow form (p.flat), which falls back to the items; without it the
// item form alone, which the larger kernel spills for (n = 30,000, m = 600,000,
// K = 15 before the S pass: 296 and 311 us with FP64 vectors, 154 and 167 with
// FP32).
template <typename V, typename TS, bool FLOW>
__global__ void __launch_bounds__(PG, 2) k_prep(PrepParams p) {
  extern __shared__ __align__(16) unsigned char dsm[];
  __shared__ V red[4][2][PT];
  __shared__ V rrc[PT], rri[PT];  // C / in-degree and 1 / in-degree of the rows of item 0
  __shared__ unsigned smax[3][PT / 32];
  __shared__ unsigned long long mk[PREP_MT][2];
  __shared__ int wsum[PG / 32];
  __shared__ int s_ok, s_div;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int G = gridDim.x;
  const int nT = p.nT;
  const int mt = p.mt;
  const bool flat = FLOW && p.flat;
  // dynamic shared memory: item slots, column cache, item offsets, pending coefficients
  PrepItem* items = reinterpret_cast<PrepItem*>(dsm);
  int* cc = reinterpret_cast<int*>(items + (MAXI + 1));
  FlowShared& fl = *reinterpret_cast<FlowShared*>(cc);
  auto& fsh = fl.fsh;
  auto& rowmap = fl.rowmap;
  auto& dep = fl.dep;
  int* ioff = cc + max(p.cap, FLOW_INTS);  // [nT + 1]
  // the pending correction of the rows of S is summed in the storage precision of S
  TS* coef = reinterpret_cast<TS*>(ioff + ((p.nT_cap + 1 + 3) & ~3));
  const TS* __restrict__ S = static_cast<const TS*>(p.S);
  TS* P = static_cast<TS*>(p.P);
  V* sI = static_cast<V*>(p.sI);
  V* sJ = static_cast<V*>(p.sJ);
  V2<V>* W = static_cast<V2<V>*>(p.W);
  V2<V>* rinv = static_cast<V2<V>*>(p.rinv);  // (C / in-degree, 1 / in-degree) per row
  const int64_t ldk = p.ldk;
  auto pidx = [ldk](int64_t a, int which, int k) -> int64_t {
    return (((a / PT) * 2 + which) * ldk + k) * PT + (a % PT);
  };
  const int np = p.npend;
  const int koff = p.koff;
  const V Cv = (V)p.C;
  const int K = p.K;
  const int new_len_j = p.d_j + p.op * p.delta;
  unsigned int nb = 0;
  bool alive = true;

  // ---- phase 0: patch (CTA 0), zero W, rows sI / sJ, tile nonzero counts
  if (blockIdx.x == 0) {
    if (p.op_end > p.op_begin) prep_patch(p.ops, p.op_begin, p.op_end, p.in, p.out);
    if (tid == 0 && p.tiles) *p.ntiles = 0;
  }
  I2* F = static_cast<I2*>(p.W);
  auto zero_w = [&]() {
    uint4* w16 = reinterpret_cast<uint4*>(W);
    const int64_t total = (int64_t)(K + 1) * p.n_pad * (int64_t)sizeof(V2<V>) / 16;
    for (int64_t e = (int64_t)blockIdx.x * PG + tid; e < total; e += (int64_t)G * PG)
      w16[e] = make_uint4(0u, 0u, 0u, 0u);
  };
  if (flat) {
    // rows without nonzeros are complete in all steps but the first
    const int blocks = (nT * PT + PG - 1) / PG;
    // (step, rows) units; step K + 1 = the means of phase 1
#pragma unroll 4
    for (int u = blockIdx.x; u < (K + 2) * blocks; u += G) {
      const int k = u / blocks, a = (u - k * blocks) * PG + tid;
      if (a < nT * PT) {
        const int len = a == p.j ? new_len_j : p.in.len[a];
        const long long c = len == 0 && k > 0 ? FLOW_DONE : 0ll;
        if (k <= K)
          *reinterpret_cast<longlong2*>(F + (int64_t)k * p.n_pad + a) = make_longlong2(c, c);
        else
          p.Y[a] = c;
      }
    }
  } else {
    zero_w();
  }
  // rows sI, sJ of tile T, a quarter of the sources per thread, and row lengths:
  // those of the first tile are on their way before the pending coefficients
  // are read
  V vI = V(0), vJ = V(0);
  int L = 0;
  auto s_rows = [&](int T) {
    const int part = tid >> 7;
    const int64_t a = (int64_t)T * PT + (tid & (PT - 1));
    vI = vJ = V(0);
    for (int u = part; u < p.delta; u += 4) vI += (V)s_at(S, p.ld, p.I[u], a, p.upper != 0);
    if (part == 3) vJ = (V)s_at(S, p.ld, p.j, a, p.upper != 0);
    // nonzeros of the tile after the patch (row j is being patched by CTA 0:
    // it counts with its new length; no other row's length changes)
    L = 0;
    if (part == 0) L = (a == p.j) ? new_len_j : p.in.len[a];
  };
  if ((int)blockIdx.x < nT) s_rows(blockIdx.x);
  int mxL = 0;                 // longest row of this thread
  float mxI = 0.f, mxJ = 0.f;  // largest |sI|, |sJ| of the rows of this thread
  bool bad = false;            // one of them is infinite or NaN
  if (np > 0) {
    // c_x[q] = sum_t xi_q[I_t], c_e[q] = sum_t eta_q[I_t]; the same at j
    for (int q = tid; q < np; q += PG) {
      TS cx = TS(0), ce = TS(0);
      for (int t = 0; t < p.delta; ++t) {
        const int64_t x = p.I[t];
        cx += P[pidx(x, 0, q)];
        ce += P[pidx(x, 1, q)];
      }
      coef[q] = cx;
      coef[np + q] = ce;
      coef[2 * np + q] = P[pidx(p.j, 0, q)];
      coef[3 * np + q] = P[pidx(p.j, 1, q)];
    }
    __syncthreads();
  }
  for (int t = 0; t < mt; ++t) {
    const int T = blockIdx.x + t * G;
    if (T >= nT) break;
    const int r = tid & (PT - 1), part = tid >> 7;
    const int64_t a = (int64_t)T * PT + r;
    if (t) s_rows(T);
    // S_cur[x, a] = S[x, a] + sum_q xi_q[x] eta_q[a] + eta_q[x] xi_q[a]: the
    // pending terms are FP32 panels of an FP32 S, so they are added in FP32
    // (on GB300 an FP64 FMA issues at 1/64 of the FP32 rate).  A warp takes every
    // 16th term and four rows per lane, several loads under way: with a row and
    // every fourth term per thread their latency was 3 us more of an update (24
    // pending, n = 20,000, K = 20).
    if constexpr (sizeof(TS) == 4) {
      if (np > 0) {
        static_assert(sizeof(FlowShared::fsh) >= (PG / 32) * 2 * PT * sizeof(float), "partial sums");
        float* cs = reinterpret_cast<float*>(fsh);
        const float* xp = P + pidx((int64_t)T * PT + 4 * lane, 0, 0);
        const float* ep = xp + ldk * PT;
        float4 cI = make_float4(0.f, 0.f, 0.f, 0.f), cJ = cI;
#pragma unroll 4
        for (int q = warp; q < np; q += PG / 32) {
          const float4 xa = *reinterpret_cast<const float4*>(xp + (int64_t)q * PT);
          const float4 ea = *reinterpret_cast<const float4*>(ep + (int64_t)q * PT);
          const float c0 = coef[q], c1 = coef[np + q], c2 = coef[2 * np + q], c3 = coef[3 * np + q];
          cI.x += c0 * ea.x + c1 * xa.x;
          cI.y += c0 * ea.y + c1 * xa.y;
          cI.z += c0 * ea.z + c1 * xa.z;
          cI.w += c0 * ea.w + c1 * xa.w;
          cJ.x += c2 * ea.x + c3 * xa.x;
          cJ.y += c2 * ea.y + c3 * xa.y;
          cJ.z += c2 * ea.z + c3 * xa.z;
          cJ.w += c2 * ea.w + c3 * xa.w;
        }
        *reinterpret_cast<float4*>(cs + (2 * warp) * PT + 4 * lane) = cI;
        *reinterpret_cast<float4*>(cs + (2 * warp + 1) * PT + 4 * lane) = cJ;
        __syncthreads();
        const float* c = cs + 8 * part * PT + r;
        vI += (V)((c[0] + c[2 * PT]) + (c[4 * PT] + c[6 * PT]));
        vJ += (V)((c[PT] + c[3 * PT]) + (c[5 * PT] + c[7 * PT]));
      }
    }
    red[part][0][r] = vI;
    red[part][1][r] = vJ;
    // inclusive scan of the row lengths over the tile (warps 0..3 hold its rows)
    int incl = L;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    if (tid < PT) {
      const V vi = (red[0][0][r] + red[1][0][r]) + (red[2][0][r] + red[3][0][r]);
      const V vj = (red[0][1][r] + red[1][1][r]) + (red[2][1][r] + red[3][1][r]);
      sI[a] = vi;
      sJ[a] = vj;
      if (flat) {
        const float fi = up_abs(vi), fj = up_abs(vj);
        bad |= !(fi <= 3.0e38f) || !(fj <= 3.0e38f);
        mxI = fmaxf(mxI, fi);
        mxJ = fmaxf(mxJ, fj);
        mxL = max(mxL, L);
      }
      int base = 0;
      for (int w = 0; w < warp; ++w) base += wsum[w];
      p.loff[a] = base + incl - L;  // nonzeros of the tile before row a
    }
    if (tid == 0) p.tile_nnz[T] = (wsum[0] + wsum[1]) + (wsum[2] + wsum[3]);
    __syncthreads();
  }
  if (flat) {
    // non-negative floats order like their bits; an infinite or NaN entry puts
    // the bits of infinity there
    if (tid < PT) {
      const unsigned bi = bad ? 0x7f800000u : __float_as_uint(mxI);
      const unsigned wi = __reduce_max_sync(0xffffffffu, bi);
      const unsigned wj = __reduce_max_sync(0xffffffffu, __float_as_uint(mxJ));
      const unsigned wl = __reduce_max_sync(0xffffffffu, (unsigned)mxL);
      if (lane == 0) {
        smax[0][warp] = wi;
        smax[1][warp] = wj;
        smax[2][warp] = wl;
      }
    }
    __syncthreads();
    if (tid < 3) {
      const unsigned m =
          max(max(smax[tid][0], smax[tid][1]), max(smax[tid][2], smax[tid][3]));
      if (m > 0u) atomicMax(p.bar + 2 + tid, m);
    }
  }
  alive = prep_barrier(p.bar, ++nb * G, p.limit, &s_ok);

  // ---- phase 1: the split of the nonzeros over the CTAs; w = Q sI summed by
  // atomics into W[0].x
  int my_items = 0;
  bool flow = false;
  StepPair<V> q0;
  int eI = 0, eG = 0;  // |sI| < 2^eI, |gamma| < 2^eG (flow form)
  bool finite = true;
  const int tper = (nT + PG - 1) / PG;  // tiles a thread adds up
  const int t0 = min(nT, tid * tper), t1 = min(nT, t0 + tper);
  // read together: each is a round trip to L2
  const unsigned b2 = __ldcg(p.bar + 2), b3 = __ldcg(p.bar + 3), b4 = __ldcg(p.bar + 4);
  const int nnz0 = t0 < t1 ? __ldcg(p.tile_nnz + t0) : 0;
  if (alive && flat) {
    const float mI = __uint_as_float(b2), mJ = __uint_as_float(b3);
    // bounds of Thm 3 / Thm 9 / Table 2 with |w_j|, |S_II| / delta^2 <= max |sI| / delta
    // (a first in-link's gamma has no other terms)
    const float gq = p.d_j == 0 ? 0.f : fabsf((float)p.gq);
    const float invC = (float)p.inv_C, m1 = mI * (float)p.inv_delta;
    const float lam = 3.f * m1 + mJ * invC + invC + 1.f;
    const float g = fmaxf(2.f * m1, gq * (m1 + mJ * invC + 0.5f * gq * lam + invC + 1.f)) * 1.01f;
    finite = mI <= 3.0e38f && mJ <= 3.0e38f && g <= 3.0e38f;
    if (finite) {
      eI = mI > 0.f ? ilogbf(mI) + 1 : 0;
      eG = g > 0.f ? ilogbf(g) + 1 : 0;
    }
  }
  if (alive) {
    // ioff[T] = the units of the tiles before T: their nonzeros (flow form,
    // tried first when allowed) or their items of at most `item` nonzeros
    for (int pass = flat && finite ? 0 : 1; pass < 2; ++pass) {
      const int div = pass == 0 ? 1 : p.item;
      int s = 0;
      for (int T = t0; T < t1; ++T) {
        const int c = T == t0 ? nnz0 : __ldcg(p.tile_nnz + T);
        s += div == 1 ? c : (c + div - 1) / div;
      }
      int incl = s;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
      }
      if (lane == 31) wsum[warp] = incl;
      __syncthreads();
      if (warp == 0) {
        const int v = (lane < PG / 32) ? wsum[lane] : 0;
        int w = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int y = __shfl_up_sync(0xffffffffu, w, o);
          if (lane >= o) w += y;
        }
        if (lane < PG / 32) wsum[lane] = w - v;
        if (lane == PG / 32 - 1) {
          ioff[nT] = w;
          // the CTA's share, by one thread (a division would be issued by
          // every thread): nonzeros per CTA (flat pass) or this CTA's items
          const int b = (int)blockIdx.x;
          // (so many that no row has more than FLOW_PARTS parts)
          s_div = pass == 0 ? max((w + G - 1) / G,
                                  ((int)b4 + FLOW_PARTS - 2) / (FLOW_PARTS - 1))
                            : (w > b ? (w - b + G - 1) / G : 0);
        }
      }
      __syncthreads();
      int run = wsum[warp] + incl - s;
      for (int T = t0; T < t1; ++T) {
        ioff[T] = run;
        const int c = T == t0 ? nnz0 : __ldcg(p.tile_nnz + T);
        run += div == 1 ? c : (c + div - 1) / div;
      }
      __syncthreads();
      if (pass == 0) {
        // every CTA computes the same nnz, so the choice is uniform over the grid
        if (s_div <= 2 * PG) {
          flow = true;
          break;
        }
        __syncthreads();  // ioff is rewritten by the item pass
      }
    }
  }
  // ---- flow form: the CTA's nonzeros [e0, e1), two per thread
  const int per = flow ? max(1, s_div) : 1;
  const float inv_per = 1.f / (float)per;
  int wait_w = 0;             // > 0: the emitted run goes on in that many warps more
  bool wait_tail = false;     // it is the tail's (else the head's)
  bool give = false;          // the head sum is the part of a row of an earlier warp
  auto w_head = [&]() { return (q0.fl >> 16) & 63u; };
  auto w_tail = [&]() { return (q0.fl >> 24) & 63u; };
  if (alive && flow) {
    const int nnz = ioff[nT];
    const int e0 = min(nnz, (int)blockIdx.x * per), e1 = min(nnz, e0 + per), cnt = e1 - e0;
    const int E = per <= PG ? 1 : 2;  // nonzeros per thread
    rowmap[tid] = -1;
    rowmap[PG + tid] = -1;
    __syncthreads();
    if (cnt > 0) {
      int T0 = 0, T1 = 0;  // the tiles of e0 and of e1 - 1
      for (int hi = nT; hi - T0 > 1;) {
        const int mid = (T0 + hi) >> 1;
        if (ioff[mid] <= e0) T0 = mid; else hi = mid;
      }
      T1 = T0;
      for (int hi = nT; hi - T1 > 1;) {
        const int mid = (T1 + hi) >> 1;
        if (ioff[mid] <= e1 - 1) T1 = mid; else hi = mid;
      }
      for (int a = T0 * PT + tid; a < (T1 + 1) * PT; a += PG) {
        const int rs = ioff[a / PT] + __ldcg(p.loff + a), len = __ldcg(p.in.len + a);
        if (len > 0 && rs < e1 && rs + len > e0) rowmap[max(rs, e0) - e0] = a;
      }
    }
    __syncthreads();
    // each position's row: the last one that starts at it or before
    const int pos = E * tid;
    const int v0 = rowmap[pos], v1 = E == 2 ? max(v0, rowmap[pos + 1]) : v0;
    int incl = v1;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl = max(incl, y);
    }
    int before = __shfl_up_sync(0xffffffffu, incl, 1);
    if (lane == 0) before = -1;
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    for (int w = 0; w < warp; ++w) before = max(before, wsum[w]);
    const int ra = max(before, v0), rb = max(before, v1);
    rowmap[pos] = ra;
    if (E == 2) rowmap[pos + 1] = rb;
    q0.ca = q0.cb = q0.kh = q0.kt = -1;
    // loads that do not depend on each other are issued together (each round is
    // a trip to L2): the rows' extents; the columns and the rows' factors; sI
    const bool has_a = pos < cnt, has_b = E == 2 && pos + 1 < cnt, two = has_b && rb != ra;
    int la = 0, lb = 0, fa = 0, fb = 0;  // lengths of rows ra, rb, and their first nonzeros
    int64_t sa = 0, sb = 0;              // their starts in the pool
    if (has_a) {
      fa = __ldcg(p.loff + ra);
      sa = __ldcg(p.in.start + ra);
      la = __ldcg(p.in.len + ra);
    }
    if (two) {
      fb = __ldcg(p.loff + rb);
      sb = __ldcg(p.in.start + rb);
      lb = __ldcg(p.in.len + rb);
    }
    fsh[tid][0] = fsh[tid][1] = SweepScale{0ull, 0, 1};
    if (has_a) {
      q0.kh = ra;
      fa += ioff[ra / PT];
      fb += ioff[rb / PT];
      q0.ca = __ldcg(p.in.col + sa + (e0 + pos - fa));
      if (has_b)
        q0.cb = __ldcg(p.in.col + (two ? sb + (e0 + pos + 1 - fb) : sa + (e0 + pos + 1 - fa)));
      fsh[tid][0] = p.recip[la];
      if (two) {
        q0.kt = rb;
        fsh[tid][1] = p.recip[lb];
      }
    }
    V xa = V(0), xb = V(0);
    if (q0.ca >= 0) xa = sI[q0.ca];
    if (q0.cb >= 0) xb = sI[q0.cb];
    pair_pattern(q0);
    if (has_a) q0.fl |= flow_weight(fa, la, e0, per, inv_per) << 16;
    if (two) q0.fl |= flow_weight(fb, lb, e0, per, inv_per) << 24;
    __syncthreads();  // rowmap
    const int w0 = 32 * E * warp, w1 = min(cnt, w0 + 32 * E);  // the warp's positions
    if (w0 < cnt) {
      const int rf = rowmap[w0], rl = rowmap[w1 - 1];
      const bool from = w0 > 0 && rowmap[w0 - 1] == rf;
      give = from && lane == 0;
      if (w1 < cnt && rowmap[w1] == rl && !(from && rf == rl)) {
        // the run of rl ends this warp and goes on: whoever emits it waits
        const bool mine_h = (q0.fl & (1u << 6)) && q0.kh == rl;
        const bool mine_t = (q0.fl & (1u << 7)) && q0.kt == rl;
        if (mine_h || mine_t) {
          wait_tail = mine_t;
          for (int x = w1; x < cnt && rowmap[x] == rl; x += 32 * E) ++wait_w;
        }
      }
    }
    // w = Q sI: the parts of each row's mean, in units of 2^(eI - 56), into Y
    I2 h{0, 0}, t{0, 0};
    if (q0.ca >= 0) h.x = fixed_of(xa, eI);
    if (q0.cb >= 0) {
      const long long v = fixed_of(xb, eI);
      if (q0.kt >= 0) t.x = v; else h.x += v;
    }
    flow_sum(q0, h, t);
    if (q0.fl & (1u << 6)) {
      h.x = fixed_scale(h.x, fsh[tid][0]);
      if (give)
        dep[1][warp].x = h.x;
      else if (wait_w == 0 || wait_tail)
        put_flow1(p.Y + q0.kh, h.x, w_head());
    }
    if (q0.fl & (1u << 7)) {
      t.x = fixed_scale(t.x, fsh[tid][1]);
      if (!wait_tail) put_flow1(p.Y + q0.kt, t.x, w_tail());
    }
    __syncthreads();
    if (wait_w) {
      long long v = wait_tail ? t.x : h.x;
      for (int x = 1; x <= wait_w; ++x) v += dep[1][warp + x].x;
      put_flow1(p.Y + (wait_tail ? q0.kt : q0.kh), v, wait_tail ? w_tail() : w_head());
    }
  } else if (alive) {
    my_items = s_div;
    if (flat) {  // set up for the flow form above
      zero_w();
      alive = prep_barrier(p.bar, ++nb * G, p.limit, &s_ok);
    }
    int cbase = 0;
    for (int u = 0; u < my_items; ++u) {
      PrepItem& it = items[min(u, MAXI)];
      item_locate(p.in, ioff, nT, blockIdx.x + u * G, p.item, it);
      if (u < MAXI) {
        const int clen = max(0, min(it.e1 - it.e0, p.cap - cbase));
        // cache the column indices of [e0, e0 + clen), one nonzero per thread
        // (a row of the item may hold all of them)
#pragma unroll 2
        for (int e = it.e0 + tid; e < it.e0 + clen; e += PG) {
          int lo = 0, hi = PT;
          while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (it.off[mid] <= e) lo = mid; else hi = mid;
          }
          cc[cbase + (e - it.e0)] = __ldcg(p.in.col + it.start[lo] + (e - it.off[lo]));
        }
        __syncthreads();
        if (tid == 0) {
          it.cbase = cbase;
          it.clen = clen;
        }
        cbase += clen;
        __syncthreads();
      }
      const int64_t rb = (int64_t)it.T * PT;
      item_gather<V>(it, item_run(it), cc, p.in.col, [&](int b) { return V2<V>{sI[b], V(0)}; },
                     [&](int r, V a, V) { red_add(&W[rb + r].x, a); });
      __syncthreads();
    }
    alive = prep_barrier(p.bar, ++nb * G, p.limit, &s_ok);
  }

  // Waits of the flow form: a warp reads its entries of W[k] again until all of
  // them hold their parts (together: lanes that waited on their own would read
  // one after the other).  Bounded: a wait that runs out sets the status word,
  // and one that sees it set gives up as well (the steps then stop in the whole
  // CTA).  True to go on waiting.
  bool stop = false;
  auto flow_again = [&](bool there, long long& it) -> bool {
    if (__all_sync(0xffffffffu, there)) return false;
    ++it;
    bool out = it > p.limit;
    if ((it & 255) == 0)
      out |= __any_sync(0xffffffffu,
                        *(volatile unsigned long long*)(p.counters + CNT_STATUS) != 0ull);
    if (out) {
      if (lane == 0)
        atomicExch(&p.counters[CNT_STATUS], (unsigned long long)SR_ERR_TIMEOUT);
      stop = true;
    }
    return !out;
  };
  // ---- phase 1b: gamma per row (tiles round-robin); W[0] = (xi_0, eta_0)
  if (alive) {
    for (int t = 0; t < mt; ++t) {
      const int T = blockIdx.x + t * G;
      if (T >= nT) break;
      int pe = 0;
      if (tid < PT) {
        const int64_t a = (int64_t)T * PT + tid;
        const int len = __ldcg(p.in.len + a);
        // the factors of row a of Q on the new graph, for every step below
        const V inv = len > 0 && !flow ? V(1) / (V)len : V(0);
        long long yw = 0;
        if (flow) {
          // the mean, once its parts are there
          yw = ld_flow1(p.Y + a);
          for (long long it = 0; flow_again(flow_there(yw), it);)
            if (!flow_there(yw)) yw = ld_flow1(p.Y + a);
          yw -= FLOW_DONE;
        }
        // sum (item form) or mean (flow form) of sI over the new in-neighbours
        const V y = flow ? fixed_value<V>(yw, eI - 56) : __ldcg(&W[a].x);
        V g;
        if (a == p.j) {
          // row j: lambda (Eq. 29b) and w_j on the old row j, in FP64
          double S_II = 0.0;
          for (int u = 0; u < p.delta; ++u) S_II += (double)__ldcg(sI + p.I[u]);
          const double S_jj = (double)__ldcg(sJ + p.j);
          const double ys =
              flow ? fixed_value<double>(yw, eI - 56) * (double)len : (double)y;
          const double wj = (ys - (double)p.op * S_II) * p.inv_ddj;  // 0 when d_j = 0
          const double id = p.inv_delta, iC = p.inv_C;
          const double lam = S_II * id * id + S_jj * iC - 2.0 * wj - iC + 1.0;
          // gq = delta / (d_j + op delta)
          const double gj = p.gq * (wj - S_jj * iC + iC - 1.0), gl = 0.5 * p.gq * p.gq * lam;
          double gd;
          if (p.op > 0)
            gd = p.d_j == 0 ? wj + 0.5 * S_II * id * id : gj + gl;
          else
            gd = p.d_j == p.delta ? -wj + 0.5 * S_II * id * id : gl - gj;
          g = (V)gd;
        } else {
          const V w = flow ? y * (V)p.inv_delta : y * inv * (V)p.inv_delta;
          const V sJa = __ldcg(sJ + a);
          const V sc = sJa * (V)p.inv_C;
          if (p.op > 0) {
            g = (p.d_j == 0) ? w : (V)p.gq * (w - sc);
          } else {
            g = (p.d_j == p.delta) ? -w : (V)p.gq * (sc - w);
          }
        }
        const V x0 = (a == p.j) ? Cv : V(0);
        if (flow) {
          put_flow(F + a, I2{a == p.j ? 1ll << 56 : 0ll, fixed_of(g, eG)}, FLOW_FULL);
        } else {
          W[a] = V2<V>{x0, g};
          rinv[a] = V2<V>{Cv * inv, inv};
        }
        P[pidx(a, 0, koff)] = (TS)x0;
        P[pidx(a, 1, koff)] = (TS)g;
        pe = nz(g);
      }
      const int any_e = __syncthreads_or(pe);
      if (tid == 0) {
        mk[t][0] = (T == p.j / PT) ? 1ull : 0ull;
        mk[t][1] = any_e ? 1ull : 0ull;
      }
    }
    if (flow && __syncthreads_or(stop)) alive = false;
    if (K > 0 && !flow) alive = prep_barrier(p.bar, ++nb * G, p.limit, &s_ok);
  }

  // ---- phase 2: K steps
  // the CTA's first item takes the fixed per-thread form when it can
  const bool pair0 = !flow && my_items > 0 && items[0].e1 - items[0].e0 <= 2 * PG;
  int64_t rb0 = 0;
  if (pair0) {
    q0 = pair_setup<V>(items[0], cc, p.in.col);
    rb0 = (int64_t)items[0].T * PT;
    if (tid < PT) {
      const V2<V> f = ld_v2cg(rinv + rb0 + tid);
      rrc[tid] = f.x;
      rri[tid] = f.y;
    }
    __syncthreads();
  }
  if (alive && flow) {
    for (int k = 0; k < K; ++k) {
      const I2* Fk = F + (int64_t)k * p.n_pad;
      I2* Fn = F + (int64_t)(k + 1) * p.n_pad;
      I2 h{0, 0}, t{0, 0}, u{0, 0};
      // both loads are on their way before the first is looked at
      if (q0.ca >= 0) h = look_flow(Fk + q0.ca);
      if (q0.cb >= 0) u = look_flow(Fk + q0.cb);
      for (long long it = 0;;) {
        const bool wa = q0.ca >= 0 && !flow_there(h), wb = q0.cb >= 0 && !flow_there(u);
        if (!flow_again(!(wa || wb), it)) break;
        if (wa) h = ld_flow(Fk + q0.ca);
        if (wb) u = ld_flow(Fk + q0.cb);
      }
      if (q0.ca >= 0) flow_strip(h);
      if (q0.cb >= 0) flow_strip(u);
      if (q0.kt >= 0) {
        t = u;
      } else {
        h.x += u.x;
        h.y += u.y;
      }
      flow_sum(q0, h, t);
      if (q0.fl & (1u << 6)) {
        const SweepScale f = fsh[tid][0];
        h.x = fixed_scale(h.x, f);
        h.y = fixed_scale(h.y, f);
        if (give)
          dep[k & 1][warp] = h;
        else if (wait_w == 0 || wait_tail)
          put_flow(Fn + q0.kh, h, w_head());
      }
      if (q0.fl & (1u << 7)) {
        const SweepScale f = fsh[tid][1];
        t.x = fixed_scale(t.x, f);
        t.y = fixed_scale(t.y, f);
        if (!wait_tail) put_flow(Fn + q0.kt, t, w_tail());
      }
      if (__syncthreads_or(stop)) {
        alive = false;  // on every thread of the CTA
        break;
      }
      if (wait_w) {
        if (wait_tail) h = t;
#pragma unroll 4
        for (int x = 1; x <= wait_w; ++x) {
          h.x += dep[k & 1][warp + x].x;
          h.y += dep[k & 1][warp + x].y;
        }
        put_flow(Fn + (wait_tail ? q0.kt : q0.kh), h, wait_tail ? w_tail() : w_head());
      }
    }
  }
  for (int k = 0; alive && !flow && k < K; ++k) {
    const V2<V>* Wk = W + (int64_t)k * p.n_pad;
    V2<V>* Wn = W + (int64_t)(k + 1) * p.n_pad;
    for (int u = 0; u < my_items; ++u) {
      if (u == 0 && pair0) {
        pair_step<V>(q0, [&](int b) { return ld_v2(Wk + b); },
                     [&](int r, V a, V b) { red_add2(Wn + rb0 + r, a * rrc[r], b * rri[r]); });
        continue;
      }
      PrepItem& it = items[min(u, MAXI)];
      if (u >= MAXI) item_locate(p.in, ioff, nT, blockIdx.x + u * G, p.item, it);
      const int64_t rb = (int64_t)it.T * PT;
      item_gather<V>(it, item_run(it), cc, p.in.col,
                     [&](int b) { return ld_v2(Wk + b); },
                     [&](int r, V a, V b) {
                       const V2<V> f = ld_v2cg(rinv + rb + r);
                       red_add2(Wn + rb + r, a * f.x, b * f.y);
                     });
      __syncthreads();
    }
    alive = prep_barrier(p.bar, ++nb * G, p.limit, &s_ok);
  }

  // ---- columns 1..K of the owned tiles into the panels, with their mask bits
  if (alive && K > 0) {
    for (int t = 0; t < mt; ++t) {
      const int T = blockIdx.x + t * G;
      if (T >= nT) break;
      // warp w copies columns k = 1 + w, 1 + w + 16, ...
      for (int k = 1 + warp; k <= K; k += PG / 32) {
        const V2<V>* Wk = W + (int64_t)k * p.n_pad;
        const I2* Fk = F + (int64_t)k * p.n_pad + T * PT + lane;
        const SweepScale ck = flow ? p.cpow[k] : SweepScale{0ull, 0, 0};
        I2 look[PT / 32];
#pragma unroll
        for (int q = 0; q < PT / 32; ++q) look[q] = flow ? ld_flow(Fk + q * 32) : I2{0, 0};
        if (flow)
          for (long long it = 0;;) {
            bool w = false;
#pragma unroll
            for (int q = 0; q < PT / 32; ++q) w |= !flow_there(look[q]);
            if (!flow_again(!w, it)) break;
#pragma unroll
            for (int q = 0; q < PT / 32; ++q)
              if (!flow_there(look[q])) look[q] = ld_flow(Fk + q * 32);
          }
        if (stop) break;  // the whole warp: parts are missing, the panel keeps its values
        bool nx = false, ne = false;
#pragma unroll
        for (int q = 0; q < PT / 32; ++q) {
          const int64_t a = (int64_t)T * PT + q * 32 + lane;
          // the mask bits follow the stored panel values (a value that rounds
          // to zero in the precision of S adds nothing to S)
          TS px, pe;
          if (flow) {
            // xi_k = C^(k+1) x 2^-56, C^(k+1) = r 2^-(63 + s)
            I2 v = look[q];
            flow_strip(v);
            px = fixed_value<TS>(__mul64hi(v.x << 6, (long long)ck.r), -61 - ck.sh);
            pe = fixed_value<TS>(v.y, eG - 56);
          } else {
            const V2<V> v = ld_v2(Wk + a);
            px = (TS)v.x;
            pe = (TS)v.y;
          }
          P[pidx(a, 0, koff + k)] = px;
          P[pidx(a, 1, koff + k)] = pe;
          nx |= nz(px);
          ne |= nz(pe);
        }
        const unsigned bx = __ballot_sync(0xffffffffu, nx), be = __ballot_sync(0xffffffffu, ne);
        const unsigned long long bit = 1ull << (k & 63);
        if (lane == 0) {
          if (bx) atomicOr(&mk[t][0], bit);
          if (be) atomicOr(&mk[t][1], bit);
        }
      }
    }
    if (flow && __syncthreads_or(stop)) alive = false;  // no masks, no list
  }

  // ---- phase 3: mask words and the affected tile pairs
  if (alive) {
    __syncthreads();
    if (tid == 0) {
      for (int t = 0; t < mt; ++t) {
        const int T = blockIdx.x + t * G;
        if (T >= nT) break;
        p.mXi[T] = mk[t][0];
        p.mEta[T] = mk[t][1];
        if (p.pXi) {
          if (mk[t][0]) p.pXi[T] = 1ull;
          if (mk[t][1]) p.pEta[T] = 1ull;
        }
      }
    }
    if (p.tiles) {
      alive = prep_barrier(p.bar, ++nb * G, p.limit, &s_ok);
      if (alive) {
        const unsigned long long* mx = reinterpret_cast<const unsigned long long*>(p.mXi);
        const unsigned long long* me = reinterpret_cast<const unsigned long long*>(p.mEta);
        for (int I = blockIdx.x; I < nT; I += G) {
          const unsigned long long xi = __ldcg(mx + I), ei = __ldcg(me + I);
          for (int J0 = I; J0 < nT; J0 += PG) {
            const int J = J0 + tid;
            bool act = false;
            if (J < nT)
              act = (p.tile_mode == 0) ||
                    (((xi & __ldcg(me + J)) | (ei & __ldcg(mx + J))) != 0ull);
            const unsigned mask = __ballot_sync(0xffffffffu, act);
            if (mask == 0) continue;
            const int leader = __ffs(mask) - 1;
            int base = 0;
            if (lane == leader) base = atomicAdd(p.ntiles, __popc(mask));
            base = __shfl_sync(0xffffffffu, base, leader);
            if (act)
              p.tiles[base + __popc(mask & ((1u << lane) - 1u))] =
                  ((uint32_t)I << 16) | (uint32_t)J;
          }
        }
      }
    }
  }

  // every CTA has left every barrier once all have arrived here: the last
  // one resets the barrier state for the next launch
  __syncthreads();
  if (tid == 0) {
    if (!alive) atomicExch(&p.counters[CNT_STATUS], (unsigned long long)SR_ERR_TIMEOUT);
    __threadfence();
    const unsigned int e = atomicAdd(p.bar + 1, 1u) + 1u;
    if (e == (unsigned int)G) {
      atomicExch(p.bar, 0u);
      atomicExch(p.bar + 1, 0u);
      atomicExch(p.bar + 2, 0u);
      atomicExch(p.bar + 3, 0u);
      atomicExch(p.bar + 4, 0u);
    }
  }
}

template <typename TS>
size_t prep_smem(int cap, int nT_cap, int npend_max) {
  return (size_t)(MAXI + 1) * sizeof(PrepItem) + (size_t)std::max(cap, FLOW_INTS) * sizeof(int) +
         (size_t)((nT_cap + 1 + 3) & ~3) * sizeof(int) + (size_t)4 * npend_max * sizeof(TS);
}

}  // namespace

void launch_flow_recip(SweepScale* out, int count, cudaStream_t st) {
  k_flow_recip<<<(count + 255) / 256, 256, 0, st>>>(out, count);
}

// The co-resident CTAs per SM of a kernel with smem bytes of dynamic shared
// memory into fit (see PrepFit).  False on an error.
static bool prep_resident(const void* fn, int which, size_t smem, PrepFit& fit) {
  if (fit.fn == fn && fit.smem == smem) return true;
  // the limit is the device's, not this launch's, so that no handle lowers
  // another's (per device: smem_attr_once)
  static std::atomic<unsigned long long> done[6];
  cudaFuncAttributes fa;
  int dev = 0, most = 0, per_sm = 0;
  if (cudaFuncGetAttributes(&fa, fn) != cudaSuccess || cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess)
    return false;
  if (smem_attr_once(fn, most - (int)fa.sharedSizeBytes, done[which]) != cudaSuccess) return false;
  if (smem > (size_t)most - fa.sharedSizeBytes) return false;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, PG, smem) != cudaSuccess)
    return false;
  fit = PrepFit{fn, smem, per_sm};
  return true;
}

int launch_prep(const PrepParams& prm, int s_prec, int vec64, int npend_max, int num_sms,
                int max_ctas, int64_t nnz, PrepFit (&fit)[2], cudaStream_t st) {
  if (prm.nT <= 0) return 0;
  if (prm.item < 0 || prm.cap < 0 || (prm.cap & 3)) return 1;
  const size_t smem = (s_prec == 64) ? prep_smem<double>(prm.cap, prm.nT_cap, npend_max)
                                     : prep_smem<float>(prm.cap, prm.nT_cap, npend_max);
  // item form, flow form
  static const void* const fns[3][2] = {
      {(const void*)k_prep<double, double, false>, (const void*)k_prep<double, double, true>},
      {(const void*)k_prep<double, float, false>, (const void*)k_prep<double, float, true>},
      {(const void*)k_prep<float, float, false>, (const void*)k_prep<float, float, true>}};
  const int which = s_prec == 64 ? 0 : vec64 ? 1 : 2;
  PrepParams a = prm;
  if (a.item == 0) a.item = 1024;
  const void* fn = nullptr;
  int grid = 0;
  for (int flow = prm.flat ? 1 : 0; flow >= 0; --flow) {
    fn = fns[which][flow];
    const bool fits = prep_resident(fn, 2 * which + flow, smem, fit[flow]);
    if (flow && !(fits && fit[flow].per_sm > 0)) continue;
    if (!fits) return 1;
    if (fit[flow].per_sm <= 0) return 2;
    // one CTA per item (at most nT + nnz / item of them), at most all
    // co-resident CTAs
    const int full = fit[flow].per_sm * num_sms;
    grid = (int)std::min<int64_t>((int64_t)prm.nT + nnz / (prm.item > 0 ? prm.item : FLOW_CTA) + 1,
                                  full);
    if (max_ctas > 0) grid = std::min(grid, max_ctas);
    grid = std::max(grid, 1);
    a.flat = flow;
    // more than two nonzeros a thread take the item form.  The flow form would
    // find that out behind its zero fill and fill W again: n = 24,000,
    // m = 340,000, K = 15, FP32 129 us an update before the S pass, here 111
    if (nnz <= (int64_t)2 * PG * grid) break;
  }
  if ((prm.nT + grid - 1) / grid > PREP_MT) return 2;
  if (prm.npend > npend_max) return 1;
  a.mt = (prm.nT + grid - 1) / grid;
  void* args[] = {&a};
  if (cudaLaunchCooperativeKernel(fn, grid, PG, args, smem, st) != cudaSuccess) return 1;
  return 0;
}

}  // namespace sr
