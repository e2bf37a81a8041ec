// The s-overlap walk (Section IV-B/C): for every active row e, count the
// wedges e -> v -> f with f > e per far end f, keep the f with count >= s and
// emit them in ascending f.  The count of f after the walk is |e ∩ f|
// exactly, because each vertex of e contributes one wedge to f when f
// contains it.  Rows are binned by their wedge work:
//
//   warp bin   (work <= 128):   a warp gathers the row's wedge ends in shared
//                               memory, sorts them and counts runs;
//   CTA bins   (work <= 4096):  a CTA counts in a shared-memory open-
//                               addressing table holding twice the row's work
//                               (it can never fill), then sorts the surviving
//                               pairs in shared memory;
//   dense bin  (slg_dense.cu):  rows with enough wedges for their id span are
//                               counted in windows of packed counters;
//   sparse bin (slg_sparse.cu): other rows with s >= 2, up to 65,536 wedges;
//   flat bin   (slg_sparse.cu): of these, rows of many short tails, up to
//                               16,384 wedges;
//   rows bin   (slg_sparse.cu): rows with s >= 2 and work <= 1024, a warp each
//                               (the warp and CTA bins keep the s = 1 rows);
//   giant bin  (the rest):      a CTA splits the row's far ends into f-range
//                               buckets through a per-CTA global scratch and
//                               counts each bucket, in ascending f, in the
//                               shared-memory table.
//
// Output modes: COUNT (pairs per row only), STAGE (each row's sorted pairs
// are appended to a staging area at an atomically reserved offset) and
// DIRECT (written to their final place, row_ptr known).
#include <algorithm>
#include <mutex>
#include <type_traits>

#include "slg_walk.cuh"

namespace slg {

// ------------------------------------------------------------- warp bin --

constexpr int kWarpNT = 256;
constexpr int kWarpBuf = kWarpMaxWork;  // 128 ints per warp

__global__ __launch_bounds__(kWarpNT) void k_walk_warp(Walk w, const int32_t *__restrict__ rows,
                                                       EmitArgs a) {
  const Meta *meta = a.meta;
  if (meta->err) return;
  __shared__ int32_t s_buf[kWarpNT / 32][kWarpBuf];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  int32_t *buf = s_buf[wib];
  const long long nrows = (long long)meta->rows_bin[kBinWarp];
  const long long gw = ((long long)blockIdx.x * kWarpNT + threadIdx.x) >> 5;
  const long long nw = ((long long)gridDim.x * kWarpNT) >> 5;
  for (long long r = gw; r < nrows; r += nw) {
    const int32_t e = rows[r];
    const int32_t k0 = w.r_off[e], k1 = w.r_off[e + 1];
    const int32_t smin = s_of(a.row_s, a.smin, e);
    // 1. gather the wedge ends (row work <= kWarpBuf by binning)
    int32_t filled = 0;
    for (int32_t base = k0; base < k1; base += 32) {
      const int32_t k = base + lane;
      int32_t b = 0, len = 0;
      if (k < k1) {
        b = __ldg(w.tail_beg + k);
        len = __ldg(w.tail_end + k) - b;
      }
      const int32_t inc = warp_inclusive_scan(len);
      const int32_t total = __shfl_sync(0xffffffffu, inc, 31);
      for (int32_t i0 = 0; i0 < total; i0 += 32) {
        const int32_t i = i0 + lane;
        int32_t j = 0;
#pragma unroll
        for (int step = 16; step > 0; step >>= 1) {
          const int32_t cand = j + step;
          if (__shfl_sync(0xffffffffu, inc, cand - 1) <= i) j = cand;
        }
        const int32_t seg_inc = __shfl_sync(0xffffffffu, inc, j);
        const int32_t seg_len = __shfl_sync(0xffffffffu, len, j);
        const int32_t seg_beg = __shfl_sync(0xffffffffu, b, j);
        if (i < total && filled + i < kWarpBuf)
          buf[filled + i] = __ldg(w.c_idx_s + seg_beg + (i - (seg_inc - seg_len)));
      }
      filled += total;
    }
    const int32_t n = filled < kWarpBuf ? filled : kWarpBuf;
    // 2. bitonic sort of the n ends, padded to a power of two
    int32_t n2 = 1;
    while (n2 < n) n2 <<= 1;
    for (int32_t i = n + lane; i < n2; i += 32) buf[i] = 0x7fffffff;
    __syncwarp();
    for (int32_t k = 2; k <= n2; k <<= 1) {
      for (int32_t jj = k >> 1; jj > 0; jj >>= 1) {
        for (int32_t i = lane; i < n2; i += 32) {
          const int32_t ixj = i ^ jj;
          if (ixj > i) {
            const int32_t x = buf[i], y = buf[ixj];
            const bool up = (i & k) == 0;
            if ((x > y) == up) {
              buf[i] = y;
              buf[ixj] = x;
            }
          }
        }
        __syncwarp();
      }
    }
    // 3. run starts with run length >= s, kept in order
    int32_t cnt_total = 0;
    for (int32_t p0 = 0; p0 < n; p0 += 32) {
      const int32_t p = p0 + lane;
      bool q = false;
      if (p < n && (p == 0 || buf[p - 1] != buf[p])) {
        int32_t end = p + 1;
        while (end < n && buf[end] == buf[p]) ++end;
        q = (end - p) >= smin;
      }
      cnt_total += __popc(__ballot_sync(0xffffffffu, q));
    }
    long long base = -1;
    if (lane == 0) base = reserve(a, e, cnt_total, kBinWarp);
    base = __shfl_sync(0xffffffffu, base, 0);
    if (a.mode != kCount && base >= 0) {
      int32_t t0 = 0;
      for (int32_t p0 = 0; p0 < n; p0 += 32) {
        const int32_t p = p0 + lane;
        bool q = false;
        int32_t c = 0;
        if (p < n && (p == 0 || buf[p - 1] != buf[p])) {
          int32_t end = p + 1;
          while (end < n && buf[end] == buf[p]) ++end;
          c = end - p;
          q = c >= smin;
        }
        const unsigned bal = __ballot_sync(0xffffffffu, q);
        if (q) put(a, base, t0 + __popc(bal & ((1u << lane) - 1)), e, buf[p], c);
        t0 += __popc(bal);
      }
    }
    __syncwarp();
  }
}

// -------------------------------------------------------------- CTA bins --

#ifndef SLG_CTA_LIST_SORT
#define SLG_CTA_LIST_SORT 1
#endif
template <int NT, int TMAX>
struct CtaCfg {
  static constexpr int kSPT = TMAX / NT;  // slots per thread at most
  static constexpr int kList = TMAX / 4;  // survivors of a row when s >= 2 (<= work / 2)
  static constexpr int kQ = (kList + NT - 1) / NT;
  // survivor sets ranked in the list area: ceil(n / 2) + n keys <= kList / 2
  static constexpr int kListSortMax = kList / 3;
  static_assert((16 + TMAX * 8 + (2 * NT + 1 + NT / 32 + 1) * 4) % 8 == 0,
                "the survivor list starts on an 8-byte boundary");
  // [s_base 16 B][table TMAX x 8 B][s_beg NT][s_pref NT+1][ws NT/32+1]
  // [list kList][list count 1]
  static constexpr size_t smem() {
    return 16 + (size_t)TMAX * 8 + (size_t)(2 * NT + 1 + NT / 32 + 1) * 4 +
           (size_t)(kList + 1) * 4;
  }
};

template <int NT, int TMAX, int BIN, int MINB>
__global__ __launch_bounds__(NT, MINB) void k_walk_cta(Walk w, const int32_t *__restrict__ rows,
                                                 const int32_t *__restrict__ row_work,
                                                 EmitArgs a) {
  using Cfg = CtaCfg<NT, TMAX>;
  Meta *meta = a.meta;
  if (meta->err) return;
  extern __shared__ __align__(16) unsigned char smem[];
  long long *s_base = reinterpret_cast<long long *>(smem);
  unsigned long long *tab = reinterpret_cast<unsigned long long *>(smem + 16);
  int32_t *s_beg = reinterpret_cast<int32_t *>(tab + TMAX);
  int32_t *s_pref = s_beg + NT;
  int32_t *ws = s_pref + NT + 1;
  const SurvList sl = {ws + NT / 32 + 1, ws + NT / 32 + 1 + Cfg::kList, Cfg::kList};
  constexpr int lg_max = (TMAX >= 2) ? 31 - __builtin_clz(TMAX) : 1;

  for (int i = threadIdx.x; i < TMAX; i += NT) tab[i] = kEmpty64;
  if (threadIdx.x == 0) *sl.n = 0;
  __syncthreads();
  const long long nrows = (long long)meta->rows_bin[BIN];
  const bool unweighted = a.unweighted != 0;
  const bool emit = a.mode != kCount;
  for (long long r = blockIdx.x; r < nrows; r += gridDim.x) {
    const int32_t e = rows[r];
    const int32_t smin = s_of(a.row_s, a.smin, e);
    const int lgT = table_lg(row_work[e - a.row_begin], lg_max);
    const int32_t T = 1 << lgT;
    const int32_t k0 = w.r_off[e], k1 = w.r_off[e + 1];
    int32_t at = 0, used = 0, total;
    // s >= 2: survivors are listed as they appear; s = 1: every key survives
    if (smin >= 2) {
      cta_walk<NT, 4>(w, k0, k1, s_beg, s_pref, ws, [&](int32_t f, int32_t) {
        table_insert<true>(tab, lgT, f, 1, smin, unweighted, meta, sl);
      });
#if SLG_CTA_LIST_SORT
      // as in the giant bin: survivors ranked in the list area while the
      // table is cleared, each written straight to its place
      __syncthreads();  // inserts done: the list is final
      const int32_t nl = min(*sl.n, sl.cap);
      if (emit && nl <= Cfg::kListSortMax) {  // uniform
        if (threadIdx.x == 0) *s_base = reserve(a, e, nl, BIN);
        unsigned long long *lk = reinterpret_cast<unsigned long long *>(sl.slot) + ((nl + 1) >> 1);
        for (int32_t i = threadIdx.x; i < nl; i += NT) lk[i] = tab[sl.slot[i]] + 1ull;
        __syncthreads();  // keys and base in place; every table and slot read done
        clear_slots<NT>(tab, T);
        if (threadIdx.x == 0) *sl.n = 0;
        const long long base = *s_base;
        if (base >= 0)
          rank_keys<NT, false>(lk, nl, [&](int32_t r, unsigned long long x) {
            put(a, base, r, e, (int32_t)(x >> 32), (int32_t)(uint32_t)x);
          });
        __syncthreads();  // keys and base read before the next row
        continue;
      }
#endif
      total = table_collect_list<NT, Cfg::kQ>(tab, T, sl, emit, &at, &used);
    } else {
      cta_walk<NT, 4>(w, k0, k1, s_beg, s_pref, ws, [&](int32_t f, int32_t) {
        table_insert<false>(tab, lgT, f, 1, smin, unweighted, meta, sl);
      });
      total = table_collect<NT, Cfg::kSPT>(tab, T, smin, emit, ws, &at, &used);
    }
    if (threadIdx.x == 0) *s_base = reserve(a, e, total, BIN);
    __syncthreads();
    const long long base = *s_base;
    if (emit && base >= 0) {
      for (int32_t i = threadIdx.x; i < total; i += NT) {
        const unsigned long long x = tab[at + i];
        put(a, base, i, e, (int32_t)(x >> 32), (int32_t)(uint32_t)x);
      }
    }
    table_reset_front<NT>(tab, used);
  }
}

// ------------------------------------------------------------- giant bin --
//
// A CTA takes one giant row at a time (dynamic ticket; rows above
// kGiantHugeWork wedges first, so that the schedule ends on small rows); two
// CTAs share an SM.  The row's far ends f lie in [f_lo, R) (f_lo = e + 1 for
// the upper-triangle walk, 0 for whole columns).  Rows of at most
// kGiantDirectMax wedges are counted in one table during the walk; the
// others are partitioned:
//   1. one load-balanced walk copies the row's far ends, in flattened wedge
//      order, to the CTA's global scratch `flat` (coalesced stores); a row
//      whose ids fit one super-chunk also counts its sub-range histogram
//      during this walk;
//   2. the id range is cut into super-chunks of at most kNSB sub-ranges of
//      2^shift ids each (2^shift <= kGiantTMax / 4).  Per super-chunk: a pass
//      over `flat` counts its wedges per sub-range (shared histogram), an
//      exclusive scan, and a second pass scatters them to `wl`, grouped by
//      sub-range;
//   3. consecutive sub-ranges form buckets of at most CAP wedges (a single
//      larger sub-range forms its own bucket: it holds at most 2^shift
//      distinct ids); bucket by bucket, in ascending f, the shared table
//      counts the far ends and the bucket's pairs (already in order) are
//      appended to the row's output.
// Core rows (tensor-core tile path) add their tile items (f, tile count) to
// the buckets of their id ranges.  Nothing is counted in global memory and
// the output comes out sorted.

// Geometry (compile-time; the defaults are the tuned values).
#ifndef SLG_GIANT_NT
#define SLG_GIANT_NT 512
#endif
#ifndef SLG_GIANT_TMAX
#define SLG_GIANT_TMAX 8192
#endif
#ifndef SLG_GIANT_MINB
#define SLG_GIANT_MINB 2
#endif
constexpr int kGiantNT = SLG_GIANT_NT;
constexpr int kGiantTMax = SLG_GIANT_TMAX;
constexpr int kNSBLog = 11;
constexpr int kNSB = 1 << kNSBLog;  // sub-ranges per super-chunk
constexpr int kShiftMax = 31 - __builtin_clz(kGiantTMax / 4);  // 2^shift <= kGiantTMax / 4
constexpr int kGiantSPT = kGiantTMax / kGiantNT;

constexpr int kGiantList = kGiantTMax / 2;  // survivors of a bucket (<= its distinct keys)
#ifndef SLG_GIANT_DIRECT_MAX
#define SLG_GIANT_DIRECT_MAX 6144
#endif
// Rows of at most this many wedges skip the partition: one table, filled to
// at most 3/4 (the survivor list holds work / 2 >= any s >= 2 survivor set).
constexpr int32_t kGiantDirectMax = SLG_GIANT_DIRECT_MAX;
constexpr int kGiantG = 6;  // wedges per thread per step of the giant bin's walk (4, 6, 8 swept)
static_assert(kGiantDirectMax <= kGiantTMax && kGiantDirectMax / 2 <= kGiantList,
              "a direct row fits the table and the survivor list");
constexpr int kGiantQ = kGiantList / kGiantNT;
static_assert(kNSB % kGiantNT == 0 && kGiantTMax % kGiantNT == 0 && kGiantList % kGiantNT == 0,
              "giant bin geometry: whole sub-ranges, slots and list entries per thread");
// Survivor sets of up to this many keys are ordered in the survivor-list
// area (kGiantList ints = kGiantList / 2 keys): the keys start past the
// slot indices (ceil(n / 2) keys) and their runs take 32 ceil(n / 32).
#ifndef SLG_GIANT_LIST_SORT
#define SLG_GIANT_LIST_SORT 1
#endif
constexpr int32_t kGiantListSortMax = kGiantList / 4;
static_assert((kGiantListSortMax + 1) / 2 + 32 * ((kGiantListSortMax + 31) / 32) <=
                  kGiantList / 2,
              "the list area holds the runs of kGiantListSortMax keys");
static_assert(kGiantListSortMax <= 8 * kGiantNT, "the run sort covers the list sort");

// [s_base 16][s_misc 16][table TMAX x 8][sub NSB][subt NSB+1][bstart NSB+1]
// [s_beg NT][s_pref NT+1][ws NT/32+1][list kGiantList][list count 1]
constexpr size_t giant_smem() {
  return 32 + (size_t)kGiantTMax * 8 + (size_t)(3 * kNSB + 2) * 4 +
         (size_t)(2 * kGiantNT + 1 + kGiantNT / 32 + 1) * 4 + (size_t)(kGiantList + 1) * 4;
}
// The survivor list starts on an 8-byte boundary (it also holds 64-bit keys).
static_assert((32 + (size_t)kGiantTMax * 8 + (size_t)(3 * kNSB + 2) * 4 +
               (size_t)(2 * kGiantNT + 1 + kGiantNT / 32 + 1) * 4) % 8 == 0,
              "survivor list alignment");

// Exclusive scan of the kNSB sub-range counters in place (P per thread);
// returns the total.
__device__ __forceinline__ int32_t scan_subranges(int32_t *a, int32_t *ws) {
  constexpr int P = kNSB / kGiantNT;
  int32_t v[P], t = 0;
#pragma unroll
  for (int q = 0; q < P; ++q) {
    v[q] = a[threadIdx.x * P + q];
    t += v[q];
  }
  int32_t total;
  const int32_t inc = block_inclusive_scan<kGiantNT>(t, ws, &total);
  int32_t run = inc - t;
#pragma unroll
  for (int q = 0; q < P; ++q) {
    a[threadIdx.x * P + q] = run;
    run += v[q];
  }
  __syncthreads();
  return total;
}

__global__ __launch_bounds__(kGiantNT, SLG_GIANT_MINB) void k_walk_giant(Walk w, const int32_t *__restrict__ rows,
                                                            EmitArgs a, int32_t *__restrict__ scratch,
                                                            long long scratch_stride, int32_t R,
                                                            int32_t list_len) {
  Meta *meta = a.meta;
  if (meta->err) return;
  extern __shared__ __align__(16) unsigned char smem[];
  long long *s_base = reinterpret_cast<long long *>(smem);
  int32_t *s_misc = reinterpret_cast<int32_t *>(smem + 16);  // [0] row, [1] buckets, [2,3] items
  unsigned long long *tab = reinterpret_cast<unsigned long long *>(smem + 32);
  int32_t *sub = reinterpret_cast<int32_t *>(tab + kGiantTMax);
  int32_t *subt = sub + kNSB;  // tile items per sub-range (core rows)
  int32_t *bstart = subt + kNSB + 1;
  int32_t *s_beg = bstart + kNSB + 1;
  int32_t *s_pref = s_beg + kGiantNT;
  int32_t *ws = s_pref + kGiantNT + 1;
  const SurvList sl = {ws + kGiantNT / 32 + 1, ws + kGiantNT / 32 + 1 + kGiantList, kGiantList};
  // per-CTA global scratch, 4 ints per wedge of the largest row:
  // flattened far ends, far ends grouped by sub-range, staged pairs (j, w)
  const long long q4 = scratch_stride / 4;
  int32_t *flat = scratch + (long long)blockIdx.x * scratch_stride;
  int32_t *wl = flat + q4;
  int32_t *tj = wl + q4;
  int32_t *tw = tj + q4;

  for (int i = threadIdx.x; i < kGiantTMax; i += kGiantNT) tab[i] = kEmpty64;
  if (threadIdx.x == 0) *sl.n = 0;
  const unsigned nrows = (unsigned)meta->rows_bin[kBinGiant];
  const unsigned nhuge = meta->giant_huge;  // rows[0, nhuge); the others end at rows[list_len)
  const bool unweighted = a.unweighted != 0;
  const bool emit = a.mode != kCount;
  constexpr int lg_max = 31 - __builtin_clz(kGiantTMax);
  for (;;) {
    __syncthreads();
    if (threadIdx.x == 0) {
      const unsigned t = atomicAdd(&meta->giant_ticket, 1u);
      s_misc[0] = t >= nrows ? -1 : rows[t < nhuge ? t : list_len - 1 - (t - nhuge)];
    }
    __syncthreads();
    const int32_t e = s_misc[0];
    if (e < 0) break;
    const int32_t smin = s_of(a.row_s, a.smin, e);
    const int32_t f_lo = a.full_rows ? 0 : e + 1;
    // far ends lie in [f_lo, f_hi): below R, or below the end of e's member
    // in a batched union
    const int32_t f_hi = a.row_fhi ? a.row_fhi[e] : R;
    const int32_t span = f_hi - f_lo;
    const int shift = min(kShiftMax, max(0, ceil_log2(span) - kNSBLog));
    const int32_t chunk_w = kNSB << shift;  // ids per super-chunk
    const int32_t cap = kGiantTMax / 2 - (1 << shift);
    const int32_t work = a.row_work[e - a.row_begin];
    if (work > q4) {  // the scratch is sized by the largest row: cannot happen
      if (threadIdx.x == 0) raise_error(meta, SLG_ERR_INVALID, kWhereGiant);
      break;
    }
    // Core rows also receive tile items (f, |e ∩ f ∩ C_c|) for every active
    // core row f > e with a non-zero tile count.
    const CoreInfo &ci = a.core;
    const bool core_row = ci.T && ci.row_rank[e + 1] != ci.row_rank[e];
    const int32_t ri = core_row ? ci.row_rank[e] : 0;
    const int32_t *Trow = core_row ? ci.T + (long long)ri * ci.Mp : nullptr;
    long long base = -1;
    if (a.mode == kDirect) base = a.row_ptr[e - a.row_begin];
    int32_t out = 0;  // pairs of the row so far
    if (work <= kGiantDirectMax && !core_row) {
      // A row this small is counted in one table during the walk, as in the
      // CTA bins (no flattened copy, no sub-ranges): its distinct far ends
      // fill at most kGiantDirectMax / kGiantTMax of the table.
      const int lgT = table_lg(work, lg_max);
      const int32_t T = 1 << lgT;
      int32_t at = 0, used = T;
      if (smin >= 2) {
        cta_walk<kGiantNT, kGiantG>(w, w.r_off[e], w.r_off[e + 1], s_beg, s_pref, ws,
                              [&](int32_t f, int32_t) {
                                table_insert<true>(tab, lgT, f, 1, smin, unweighted, meta, sl);
                              });
        out = table_collect_list<kGiantNT, kGiantQ>(tab, T, sl, emit, &at, &used);
      } else {
        cta_walk<kGiantNT, kGiantG>(w, w.r_off[e], w.r_off[e + 1], s_beg, s_pref, ws,
                              [&](int32_t f, int32_t) {
                                table_insert<false>(tab, lgT, f, 1, smin, unweighted, meta, sl);
                              });
        out = table_collect<kGiantNT, kGiantSPT>(tab, T, smin, emit, ws, &at, &used);
      }
      if (emit)
        for (int32_t i = threadIdx.x; i < out; i += kGiantNT) {
          const unsigned long long x = tab[at + i];
          const int32_t f = (int32_t)(x >> 32), n = (int32_t)(uint32_t)x;
          if (a.mode == kDirect) {
            put(a, base, i, e, f, n);
          } else {
            tj[i] = f;
            if (!unweighted) tw[i] = n;
          }
        }
      table_reset_front<kGiantNT>(tab, used);
    } else {
      long long clk0 = clock64();
      // 1. flattened far ends; a row within one super-chunk also counts its
      // sub-range histogram here (saving one pass over the copy)
      const bool single = f_hi - f_lo <= chunk_w;
      if (single) {
        for (int i = threadIdx.x; i < kNSB; i += kGiantNT) {
          sub[i] = 0;
          subt[i] = 0;
        }
        __syncthreads();
        cta_walk<kGiantNT, kGiantG>(w, w.r_off[e], w.r_off[e + 1], s_beg, s_pref, ws,
                              [&](int32_t f, int32_t i) {
                                flat[i] = f;
                                atomicAdd(sub + ((f - f_lo) >> shift), 1);
                              });
      } else {
        cta_walk<kGiantNT, kGiantG>(w, w.r_off[e], w.r_off[e + 1], s_beg, s_pref, ws,
                              [&](int32_t f, int32_t i) { flat[i] = f; });
      }
      long long clk_part = 0, clk_bucket = 0;
      if (threadIdx.x == 0) atomicAdd(&meta->giant_cycles[0], (unsigned long long)(clock64() - clk0));
      for (int32_t F0 = f_lo; F0 < f_hi; F0 += chunk_w) {
        // An empty bucket is skipped without a barrier, so threads may still
        // be reading the previous super-chunk's sub[] / bstart[] here: every
        // thread must be done with them before they are rewritten.
        __syncthreads();
        const long long c0 = clock64();
        const int32_t F1 = (f_hi - F0 > chunk_w) ? F0 + chunk_w : f_hi;
        const int32_t nsb = ((F1 - F0 - 1) >> shift) + 1;
        // 2. histograms of sub-ranges (wedges; tile items), scans, scatter
        if (!single) {
          for (int i = threadIdx.x; i < kNSB; i += kGiantNT) {
            sub[i] = 0;
            subt[i] = 0;
          }
          __syncthreads();
          for_each_batched<kGiantNT, 8>(flat, 0, work, [&](int32_t f) {
            if (f >= F0 && f < F1) atomicAdd(sub + ((f - F0) >> shift), 1);
          });
        }
        if (core_row)
          for (int32_t p = ri + 1 + (int32_t)threadIdx.x; p < ci.n_core; p += kGiantNT) {
            const int32_t f = ci.core_list[p];
            if (f >= F0 && f < F1 && w.r_off[f + 1] - w.r_off[f] >= smin && Trow[p] > 0)
              atomicAdd(subt + ((f - F0) >> shift), 1);
          }
        __syncthreads();
        const int32_t nw = scan_subranges(sub, ws);
        const int32_t items = core_row ? scan_subranges(subt, ws) : 0;
        if (nw == 0 && items == 0) continue;  // uniform: both totals are block-wide
        if (threadIdx.x == 0) subt[kNSB] = items;
        for_each_batched<kGiantNT, 8>(flat, 0, work, [&](int32_t f) {
          if (f >= F0 && f < F1) wl[atomicAdd(sub + ((f - F0) >> shift), 1)] = f;
        });
        __syncthreads();
        if (F1 == f_hi) l2_discard(flat, work);  // the flattened copy's last read
        // now sub[b] = end of the wedges of sub-range b; subt[b] = start of its
        // items.  3. bucket starts: sub-range b opens a bucket when its start
        // in the merged order (wedges + items before it) / cap changes.
        {
          constexpr int P = kNSB / kGiantNT;
          int32_t flag[P], t = 0;
  #pragma unroll
          for (int q = 0; q < P; ++q) {
            const int32_t b = threadIdx.x * P + q;
            flag[q] = 0;
            if (b < nsb) {
              const int32_t st = (b ? sub[b - 1] : 0) + (core_row ? subt[b] : 0);
              const int32_t sp = b ? (b > 1 ? sub[b - 2] : 0) + (core_row ? subt[b - 1] : 0) : 0;
              flag[q] = (b == 0) || (st / cap != sp / cap);
            }
            t += flag[q];
          }
          int32_t total;
          const int32_t inc = block_inclusive_scan<kGiantNT>(t, ws, &total);
          int32_t pos = inc - t;
  #pragma unroll
          for (int q = 0; q < P; ++q)
            if (flag[q]) bstart[pos++] = threadIdx.x * P + q;
          if (threadIdx.x == 0) {
            bstart[total] = nsb;
            s_misc[1] = total;
          }
          __syncthreads();
        }
        const int32_t nb = s_misc[1];
        const long long c1 = clock64();
        clk_part += c1 - c0;
        for (int32_t c = 0; c < nb; ++c) {
          const int32_t b0 = bstart[c], b1 = bstart[c + 1];
          const int32_t lo = b0 ? sub[b0 - 1] : 0, hi = sub[b1 - 1];
          int32_t nit = 0;
          if (core_row) {
            nit = (b1 < nsb ? subt[b1] : subt[kNSB]) - subt[b0];
            if (threadIdx.x == 0) {
              // core positions of the bucket's id range, after row e itself
              const int32_t flo = F0 + (b0 << shift);
              const int32_t fhi = b1 < nsb ? F0 + (b1 << shift) : F1;
              s_misc[2] = max(core_lower(ci.core_list, ci.n_core, flo), ri + 1);
              s_misc[3] = core_lower(ci.core_list, ci.n_core, fhi);
            }
            __syncthreads();
          }
          if (hi - lo + nit == 0) continue;  // uniform
          // the sorted pairs tab[at, at + total) of a bucket go to the row's
          // output; false (uniform) when they would not fit the scratch
          auto emit_sorted = [&](int32_t at, int32_t total, int32_t used) -> bool {
            if (a.mode == kStage && out + total > q4) {
              // staged pairs would not fit the scratch (sized by wedges +
              // core items): report instead of writing past it
              if (threadIdx.x == 0) raise_error(meta, SLG_ERR_INVALID, kWhereGiant);
              table_reset_front<kGiantNT>(tab, used);
              return false;
            }
            if (emit && total > 0) {
              for (int32_t i = threadIdx.x; i < total; i += kGiantNT) {
                const unsigned long long x = tab[at + i];
                const int32_t f = (int32_t)(x >> 32), n = (int32_t)(uint32_t)x;
                if (a.mode == kDirect) {
                  put(a, base, out + i, e, f, n);
                } else {
                  tj[out + i] = f;
                  if (!unweighted) tw[out + i] = n;
                }
              }
            }
            out += total;
            table_reset_front<kGiantNT>(tab, used);
            return true;
          };
          // sub-ranges [h0, h1) (wedges wl[hlo, hhi), tile items `hnit`)
          // counted in the hash table
          auto hash_bucket = [&](int32_t h0, int32_t h1, int32_t hlo, int32_t hhi,
                                 int32_t hnit) -> bool {
            const int32_t width = (h1 - h0) << shift;
            const int lgT = table_lg(min(hhi - hlo + hnit, width), lg_max);
            const int32_t T = 1 << lgT;
            // s >= 2: survivors listed as they appear; s = 1: every key survives
            const bool list = smin >= 2;
            auto insert_all = [&](auto list_tag) {
              constexpr bool L = decltype(list_tag)::value;
              for_each_batched<kGiantNT, 8>(wl, hlo, hhi, [&](int32_t f) {
                table_insert<L>(tab, lgT, f, 1, smin, unweighted, meta, sl);
              });
              if (core_row && hnit > 0)
                for (int32_t p = s_misc[2] + (int32_t)threadIdx.x; p < s_misc[3];
                     p += kGiantNT) {
                  const int32_t f = ci.core_list[p];
                  const int32_t wt = Trow[p];
                  if (wt > 0 && w.r_off[f + 1] - w.r_off[f] >= smin)
                    table_insert<L>(tab, lgT, f, wt, smin, unweighted, meta, sl);
                }
            };
            int32_t at = 0, used = T, total;
            if (list) {
              insert_all(std::true_type{});
#if SLG_GIANT_LIST_SORT
              // Survivors ordered in the survivor-list area, past their slot
              // indices, while the table is cleared: no front region of the
              // table to clear afterwards, two block barriers fewer per bucket.
              __syncthreads();  // inserts done: the list is final
              const int32_t nl = min(*sl.n, sl.cap);
              if (emit && nl <= kGiantListSortMax) {  // uniform
                unsigned long long *lk =
                    reinterpret_cast<unsigned long long *>(sl.slot) + ((nl + 1) >> 1);
                for (int32_t i = threadIdx.x; i < nl; i += kGiantNT)
                  lk[i] = tab[sl.slot[i]] + 1ull;  // the count word holds count - 1
                __syncthreads();  // keys in place; every table and slot read done
                clear_slots<kGiantNT>(tab, T);
                if (threadIdx.x == 0) *sl.n = 0;
                if (a.mode == kStage && out + nl > q4) {  // uniform
                  if (threadIdx.x == 0) raise_error(meta, SLG_ERR_INVALID, kWhereGiant);
                  __syncthreads();
                  return false;
                }
                // each key goes straight to its ranked place in the row's output
                rank_keys<kGiantNT>(lk, nl, [&](int32_t r, unsigned long long x) {
                  const int32_t f = (int32_t)(x >> 32), n = (int32_t)(uint32_t)x;
                  if (a.mode == kDirect) {
                    put(a, base, out + r, e, f, n);
                  } else {
                    tj[out + r] = f;
                    if (!unweighted) tw[out + r] = n;
                  }
                });
                out += nl;
                __syncthreads();  // the keys are read before the next bucket fills the list
                return true;
              }
#endif
              total = table_collect_list<kGiantNT, kGiantQ>(tab, T, sl, emit, &at, &used);
            } else {
              insert_all(std::false_type{});
              __syncthreads();
              total = table_collect<kGiantNT, kGiantSPT>(tab, T, smin, emit, ws, &at, &used);
            }
            return emit_sorted(at, total, used);
          };
          if (!hash_bucket(b0, b1, lo, hi, nit)) break;
        }
        __syncthreads();
        l2_discard(wl, nw);  // the super-chunk's grouped far ends are consumed
        clk_bucket += clock64() - c1;
      }
      if (threadIdx.x == 0) {
        atomicAdd(&meta->giant_cycles[1], (unsigned long long)clk_part);
        atomicAdd(&meta->giant_cycles[2], (unsigned long long)clk_bucket);
      }
    }  // partitioned row
    if (threadIdx.x == 0) *s_base = reserve(a, e, out, kBinGiant);
    __syncthreads();
    if (a.mode == kStage) {
      const long long b = *s_base;
      if (b >= 0)
        for (int32_t i = threadIdx.x; i < out; i += kGiantNT) {
          a.stage_j[b + i] = tj[i];
          if (!unweighted) a.stage_w[b + i] = tw[i];
        }
      __syncthreads();
      l2_discard(tj, out);  // the row's pairs are in the staging area
      if (!unweighted) l2_discard(tw, out);
    }
  }
}

// --------------------------------------------------------------- launch --

namespace {

using CfgS = CtaCfg<256, 2 * kCtaSMaxWork>;
using CfgL = CtaCfg<256, 2 * kCtaLMaxWork>;
#define K_CTA_S k_walk_cta<256, 2 * kCtaSMaxWork, kBinCtaS, 4>
#define K_CTA_L k_walk_cta<256, 2 * kCtaLMaxWork, kBinCtaL, 3>

struct Occ {
  int sms = 0, warp_blocks = 0, s_blocks = 0, l_blocks = 0, g_blocks = 0;
  int dev = -1;
};

Occ &occ_for_device() {
  static Occ occ[64];
  static std::mutex mu;
  int dev = 0;
  cudaGetDevice(&dev);
  Occ &o = occ[dev & 63];
  std::lock_guard<std::mutex> lock(mu);
  if (o.dev != dev) {
    cudaDeviceGetAttribute(&o.sms, cudaDevAttrMultiProcessorCount, dev);
    cudaFuncSetAttribute(K_CTA_S, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)CfgS::smem());
    cudaFuncSetAttribute(K_CTA_L, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)CfgL::smem());
    cudaFuncSetAttribute(k_walk_giant, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)giant_smem());
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o.warp_blocks, k_walk_warp, kWarpNT, 0);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o.s_blocks, K_CTA_S, 256, CfgS::smem());
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o.l_blocks, K_CTA_L, 256, CfgL::smem());
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o.g_blocks, k_walk_giant, kGiantNT,
                                                  giant_smem());
    if (o.g_blocks < 1) o.g_blocks = 1;
    o.dev = dev;
  }
  return o;
}

}  // namespace

int giant_ctas_for_device() {
  Occ &o = occ_for_device();
  return o.sms * o.g_blocks;
}

int giant_ctas() { return giant_ctas_for_device(); }

namespace {

// Two streams beside the caller's for the bins' kernels, of the same priority, and
// the events that order them: this host thread's, made on first use on a device
// (one set per thread and priority; given back when the thread ends or turns to
// another device).
constexpr int kPriorities = 8;  // 0 (the least) to -5 on this GPU

// The index of the stream's priority, or -1.
int priority_index(cudaStream_t st, int *priority) {
  *priority = 0;
  if (cudaStreamGetPriority(st, priority) != cudaSuccess) return cudaGetLastError(), -1;
  return *priority <= 0 && *priority > -kPriorities ? -*priority : -1;
}

struct SideStreams {
  int dev = -1;
  bool ok = false;
  cudaStream_t s[2] = {nullptr, nullptr};
  cudaEvent_t fork = nullptr, done[2] = {nullptr, nullptr};

  void drop() {
    for (cudaStream_t &x : s)
      if (x) cudaStreamDestroy(x), x = nullptr;
    for (cudaEvent_t *x : {&fork, &done[0], &done[1]})
      if (*x) cudaEventDestroy(*x), *x = nullptr;
    ok = false;
  }
  ~SideStreams() { drop(); }

  // Whether they can be forked from st.  A stream that was forked into a
  // capture stays in it until the capture ends, so in the meantime they serve
  // that capture only.
  bool ready(cudaStream_t st, int priority) {
    int d = 0;
    if (cudaGetDevice(&d) != cudaSuccess) return false;
    if (d != dev) {
      drop();
      dev = d;
      ok = true;
      cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
      cudaThreadExchangeStreamCaptureMode(&mode);
      for (cudaStream_t &x : s)
        ok &= cudaStreamCreateWithPriority(&x, cudaStreamNonBlocking, priority) == cudaSuccess;
      for (cudaEvent_t *x : {&fork, &done[0], &done[1]})
        ok &= cudaEventCreateWithFlags(x, cudaEventDisableTiming) == cudaSuccess;
      cudaThreadExchangeStreamCaptureMode(&mode);
      if (!ok) {
        drop();
        cudaGetLastError();
      }
    }
    for (int i = 0; ok && i < 2; ++i) {
      cudaStreamCaptureStatus a = cudaStreamCaptureStatusNone, b = a;
      unsigned long long ia = 0, ib = 0;
      if (cudaStreamGetCaptureInfo(s[i], &a, &ia) != cudaSuccess) return cudaGetLastError(), false;
      if (a == cudaStreamCaptureStatusNone) continue;
      if (cudaStreamGetCaptureInfo(st, &b, &ib) != cudaSuccess) return cudaGetLastError(), false;
      if (a != cudaStreamCaptureStatusActive || b != a || ia != ib) return false;
    }
    return ok;
  }
};

}  // namespace

// The bins' kernels are independent of each other (each keeps its rows, its
// tickets and its part of the scratch; the totals are atomic), except the
// giant kernel, which also takes the rows that others handed over.  Each is
// sized to fill the device, but the long rows of DnBig (a CTA per SM) leave
// most of it idle at the end, and on a mid-size graph from the start: so where
// that bin has rows, the sparse bin and DnSmall run beside it on one stream
// and the other bins on a second.  One after the other -> so: counting pass of
// 120K x 240K 1,057 -> 800 us, host builds of 200K x 400K 4,157 -> 3,464,
// 16-member batch 2,505 -> 2,150..2,198, L_3 of 500K x 1M in row form 6,092 ->
// 5,777, L_1 of 100K x 200K 2,499 -> 2,287; chung_lu_1m's four lists 105.7 ms
// both ways.  DnSmall beside the sparse bin costs more than it fills (L_2
// sweep of 150K x 300K 10,190 -> 10,711 us), as does a fork without DnBig (L_3
// of a dual of 30K x 60K 1,346 -> 1,362), but for the flat bin's kernels, which last
// as long as their longest rows too.  With per-bin timing (ev) they run
// one after the other.
cudaError_t launch_walk(const WalkLaunch &L, cudaStream_t st, int32_t *launches,
                        cudaEvent_t *ev) {
  Occ &o = occ_for_device();
  const int32_t *lists = L.bin_rows;
  const int64_t stride = L.rows;
  int n = 0;
  cudaError_t err = cudaSuccess;
  auto keep = [&](cudaError_t e) {
    if (err == cudaSuccess) err = e;
  };
  auto empty = [&](int bin) { return (L.skip >> bin) & 1u; };
  static thread_local SideStreams sides[kPriorities];
  constexpr unsigned kSkipSparse =
      kSkipSparseBig | kSkipSparseSmall | kSkipFlatBig | kSkipFlatSmall;
  const bool has_sparse = L.sparse_scratch && (L.skip & kSkipSparse) != kSkipSparse;
  const bool dense_big = L.dense_pairs[0] > 0, dense_small = L.dense_pairs[1] > 0;
  const bool chain = has_sparse || dense_small;
  const bool ctas = !empty(kBinWarp) || !empty(kBinCtaS) || !empty(kBinCtaL) ||
                    !empty(kBinRows);
  const bool has_flat =
      has_sparse && (L.skip & (kSkipFlatBig | kSkipFlatSmall)) != (kSkipFlatBig | kSkipFlatSmall);
  const bool may_fork = !ev && (dense_big || (has_flat && ctas)) && (chain || ctas);
  int priority = 0;
  const int pi = may_fork ? priority_index(st, &priority) : -1;
  SideStreams &side = sides[pi < 0 ? 0 : pi];
  const bool fork = pi >= 0 && side.ready(st, priority);
  const bool use[2] = {fork && chain, fork && ctas};
  cudaStream_t s1 = use[0] ? side.s[0] : st, s2 = use[1] ? side.s[1] : st;
  if (fork) keep(cudaEventRecord(side.fork, st));
  for (int i = 0; i < 2; ++i)
    if (use[i]) keep(cudaStreamWaitEvent(side.s[i], side.fork, 0));
  if (err != cudaSuccess) return err;  // nothing was launched
  if (ev) cudaEventRecord(ev[0], st);
  // rows with the longest run first
  if (!ev && dense_big) {
    keep(launch_walk_dense(L, 0, st));
    ++n;
  }
  if (!ev && has_sparse) keep(launch_walk_sparse(L, s1, &n));
  if (!empty(kBinWarp)) {
    k_walk_warp<<<o.sms * (o.warp_blocks > 0 ? o.warp_blocks : 1), kWarpNT, 0, s2>>>(
        L.w, lists + 0 * stride, L.a);
    ++n;
  }
  if (ev) cudaEventRecord(ev[1], st);
  if (!empty(kBinRows)) {
    keep(launch_walk_rows(L, s2));
    ++n;
  }
  if (!empty(kBinCtaS)) {
    K_CTA_S<<<o.sms * (o.s_blocks > 0 ? o.s_blocks : 1), 256, CfgS::smem(), s2>>>(
        L.w, lists + 1 * stride, L.row_work, L.a);
    ++n;
  }
  if (ev) cudaEventRecord(ev[2], st);
  if (!empty(kBinCtaL)) {
    K_CTA_L<<<o.sms * (o.l_blocks > 0 ? o.l_blocks : 1), 256, CfgL::smem(), s2>>>(
        L.w, lists + 2 * stride, L.row_work, L.a);
    ++n;
  }
  if (ev) cudaEventRecord(ev[3], st);
  if (ev && has_sparse) keep(launch_walk_sparse(L, st, &n));
  if (ev) cudaEventRecord(ev[4], st);
  if (ev && dense_big) {
    keep(launch_walk_dense(L, 0, st));
    ++n;
  }
  if (dense_small) {
    keep(launch_walk_dense(L, 1, s1));
    ++n;
  }
  keep(cudaGetLastError());
  for (int i = 0; i < 2; ++i) {
    if (!use[i]) continue;
    // joined also after an error: nothing may run on when the call returns
    cudaError_t e = cudaEventRecord(side.done[i], side.s[i]);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(st, side.done[i], 0);
    if (e != cudaSuccess) cudaStreamSynchronize(side.s[i]);
    keep(e);
  }
  if (err != cudaSuccess) return err;
  if (L.giant_scratch && L.giant_stride > 0 && !empty(kBinGiant)) {
    k_walk_giant<<<o.sms * o.g_blocks, kGiantNT, giant_smem(), st>>>(
        L.w, lists + 3 * stride, L.a, L.giant_scratch, L.giant_stride, L.R, (int32_t)stride);
    ++n;
  }
  if (ev) cudaEventRecord(ev[5], st);
  if (launches) *launches += n;
  return cudaGetLastError();
}

}  // namespace slg
