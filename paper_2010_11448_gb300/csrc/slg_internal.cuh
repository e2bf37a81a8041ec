// Internal declarations of the slg CUDA library (not part of the C ABI).
//
// Terminology.  The side being computed (H, or H* with SLG_DUAL) has R rows
// (its hyperedges) and C columns (its vertices).  CSR = (r_off, r_idx) lists
// the columns of every row, CSC = (c_off, c_idx) the rows of every column;
// both strictly ascending.  A wedge is a path e -> v -> f with v in e and f in
// N(v) (Section IV-B, the two inner loops of Algorithm 2).  Only wedges with
// f > e are walked (the strict upper triangle of Algorithm 3) and only rows
// with |row| >= s take part (degree-based pruning of Algorithm 3).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/slg.h"

namespace slg {

constexpr int kWarp = 32;
constexpr int32_t kEmpty = -1;

// Row bins by wedge work (the degree-binned scheduler).  Rows above
// kDenseMinWork wedges whose far ends are dense in their id span (is_dense)
// go to the dense bin; of the others, rows with s >= 2 from Bins::bloom up to
// Bins::sparse wedges go to the sparse bin (the flat bin, if their tails are
// short: short_tails) and the rest above the CTA bins to
// the giant bin.  Rows with s >= 2 of at most Bins::ctas
// wedges take the rows bin (a warp each; of more than kRowsMaxSize vertices the
// small CTA bin), s = 1 ones the warp and CTA bins.
// The statistics count the dense bin's rows as giant ones, the rows bin's as
// the small CTA bin's and the flat bin's as sparse ones (kNumBins bins are
// reported, kNumLists lists kept).
enum Bin : int {
  kBinWarp = 0, kBinCtaS = 1, kBinCtaL = 2, kBinGiant = 3, kBinSparse = 4, kNumBins = 5,
  kBinDense = 5, kBinFlat = 6, kBinRows = 7, kNumLists = 8
};

// Upper bounds on a row's wedge count for each non-giant bin.  The hash tables
// hold twice the bound, so a row can never fill its table (distinct
// neighbours <= wedges).
#ifndef SLG_WARP_MAX_WORK
#define SLG_WARP_MAX_WORK 128
#endif
constexpr int32_t kWarpMaxWork = SLG_WARP_MAX_WORK;
constexpr int32_t kCtaSMaxWork = 1024;
constexpr int32_t kCtaLMaxWork = 4096;
// Giant rows above this work are handed out first (largest-first order
// bounds the tail of the dynamic schedule by the largest remaining row).
#ifndef SLG_GIANT_HUGE_WORK
#define SLG_GIANT_HUGE_WORK 32768
#endif
constexpr int32_t kGiantHugeWork = SLG_GIANT_HUGE_WORK;
// Sparse and flat rows above this work take the instance of their kernel with
// the larger table.
#ifndef SLG_SP_BIG_WORK
#define SLG_SP_BIG_WORK 8192
#endif
constexpr int32_t kSparseBigWork = SLG_SP_BIG_WORK;
// Largest row of the sparse bin (Bins::sparse is at most this).
#ifndef SLG_SPARSE_MAX_WORK
#define SLG_SPARSE_MAX_WORK 65536
#endif
constexpr int32_t kSparseMaxWork = SLG_SPARSE_MAX_WORK;
// Rows of the flat bin, of up to kFlatMaxWork wedges: many vertices whose tails are
// mostly short, or tails alike, of which the longest is no eighth of the row, so that
// setting it aside gains little (400K rows of 40 vertices with 40 far ends per tail,
// counting pass 6.0 -> 4.3 ms, of 100 with 50 14.5 -> 10.8).  Larger such rows go to
// the giant bin: the sparse bin's ranges search every tail (1M rows of 400 with 40
// 267 -> 221 ms; alike is a 32nd there, to leave the others in the sparse bin).
constexpr int32_t kFlatMaxWork = 16384;
__host__ __device__ __forceinline__ bool short_tails(int32_t work, int32_t size, int32_t longest) {
  return (size > 48 && work < 32ll * size) ||
         (size > 32 && work < 128ll * size &&
          (work <= kFlatMaxWork ? 8ll : 32ll) * longest <= work);
}
// Whether the flat bin's kernels run, by its wedges and the sparse bin's; else
// its rows are given to the sparse bin (launch_join_flat).  A kernel lasts as long
// as its longest row, so a few such rows are better taken along with the others
// (counting pass of 120K x 240K, host builds of 200K x 400K: 800 and 3,470 us so,
// 870 and 3,570 with kernels of their own; chung_lu_1m the same both ways).
__host__ __device__ __forceinline__ bool flat_kernels(long long flat, long long sparse) {
  return flat > 0 && (flat >= 2 * sparse || flat >= 1ll << 28);
}
// Rows of more vertices leave the rows bin to the small CTA bin: the kernel lasts
// as long as its longest row, and a warp there walks 32 tails at a time, a CTA 256
// (rows of few wedges: late ids, or vertices that few other rows hold).  4 rows of
// 100,000 vertices and 500 wedges 2.65 -> 0.85 ms, 50 of 20,000 0.84 -> 0.51; with
// many such rows the warps do better (10,000 of 1,000 vertices 0.20 instead of
// 0.67), and a few large rows are no reason to run the CTA bin's kernel (lines at
// 256 to 1,024: counting pass of 120K x 240K 805 -> 853 us, batch of 16 5 % more).
constexpr int32_t kRowsMaxSize = 16384;
#ifndef SLG_DENSE_MIN_WORK
#define SLG_DENSE_MIN_WORK 256
#endif
constexpr int32_t kDenseMinWork = SLG_DENSE_MIN_WORK;
// Dense rows of more vertices (16-bit counters and up) take the instance of
// the dense kernel with the larger windows.
constexpr int32_t kDenseBigSize = 255;

// log2 of the dense bin's counter width for a row of `size` vertices: a
// count |e ∩ f| is at most `size`.
__host__ __device__ __forceinline__ int dense_lg_bits(int32_t size) {
  return size <= 15 ? 2 : size <= 255 ? 3 : size <= 65535 ? 4 : 5;
}

// Counter words of a window of the dense bin's two instances.
#ifndef SLG_DN_WORDS
#define SLG_DN_WORDS 10240
#endif
#ifndef SLG_DN_BIG_WORDS
#define SLG_DN_BIG_WORDS 48128
#endif
// Wedges per window and row from which a row is dense, by what else would
// count it (see is_dense): s = 1 (CTA bins or giant bin; L_1 of 100K x 200K
// 4.12, 3.84, 3.15 ms with 700, 200 from 1,024 wedges and 200 from 256); rows
// of up to kDenseFew vertices per vertex beyond two of the threshold, whose
// wedges the sparse bin mostly sets aside (L_8 of a 300K x 600K dual 7.48,
// 6.83, 7.06 ms with 2,000, 3,000, 4,500; 10.0 with one line for all s); the
// other rows (L_2 and more of a 150K x 300K dual 14.1, 13.8, 13.2 ms, step of
// chung_lu_1m 118.5, 118.4, 120.0 with 1,000, 1,300, 1,800); rows of the
// large-window instance (118.5, 117.8, 121.9 ms with 5,000, 3,500, 8,000,
// and 115.0, 115.3 with 2,500, 1,500 and the rest as here).
#ifndef SLG_DENSE_T1
#define SLG_DENSE_T1 200
#endif
#ifndef SLG_DENSE_T2
#define SLG_DENSE_T2 1300
#endif
#ifndef SLG_DENSE_T4
#define SLG_DENSE_T4 3000
#endif
#ifndef SLG_DENSE_KF
#define SLG_DENSE_KF 10
#endif
constexpr int32_t kDenseFew = SLG_DENSE_KF;
#ifndef SLG_DENSE_TB
#define SLG_DENSE_TB 2000
#endif
constexpr int kDenseRatio = 16;

// Dense rows: the dense bin's cost per row is its wedges plus so much per
// window (sweep latency, survivors, clear), the other bins' is their cost per
// wedge; so the line is drawn at a number of wedges per window.  A window also
// visits every tail, which the other bins read once: in the large-window
// instance, whose rows can have more tails than wedges per window, a visit after
// the first counts as 2.5 wedges (a quarter where hash tables would count the
// row: at s = 1, and core rows).  400K rows of 1,500 of 67M vertices, counting pass at s = 2
// 112.7, 95.3, 90.6 ms with 0.25, 1, 2.5 (125.3 without), at s = 1 117.6, 119.6,
// 121.3; rows of up to 100,000 vertices over 4M ids (web-shaped input with the
// tile path) 4.6 -> 1.75 ms; step of chung_lu_1m the same all ways.
__host__ __device__ __forceinline__ bool is_dense(int32_t work, int32_t size, int32_t s,
                                                  int32_t span, int32_t ratio,
                                                  bool core = false) {
  const int lw = 5 - dense_lg_bits(size);
  const bool big = size > kDenseBigSize;
  const int32_t nwin = span / ((big ? SLG_DN_BIG_WORDS : SLG_DN_WORDS) << lw) + 1;
  const int32_t per = big                                          ? SLG_DENSE_TB
                      : s == 1                                     ? SLG_DENSE_T1
                      : size <= (long long)kDenseFew * (s - 2) ? SLG_DENSE_T4
                                                                   : SLG_DENSE_T2;
  const long long visits = big ? (nwin - 1ll) * size * (s == 1 || core ? 4 : 40) : 0;
  return (long long)work * ratio >= (long long)per * 16 * nwin + visits;
}

// Counters the device writes and the host reads once per call.
struct Meta {
  int32_t err;                         // first slg_status raised on the device
  int32_t err_where;                   // which check raised it
  unsigned long long rows_bin[kNumLists];
  unsigned long long wedges_bin[kNumLists];
  unsigned long long incid_bin[kNumLists];
  unsigned long long pairs_bin[kNumLists];
  unsigned long long wedges;           // W_s
  unsigned long long active;           // rows with size >= s in range
  unsigned long long pairs;            // |L_s| over the row range
  unsigned int giant_ticket;           // dynamic giant-row scheduling
  unsigned int giant_huge;             // giant rows above kGiantHugeWork (front of the list)
  unsigned int giant_rest;             // the other giant rows (back of the list)
  unsigned int sparse_ticket;          // the same three for the sparse bin
  unsigned int sparse_ticket_rest;
  unsigned int sparse_huge;
  unsigned int sparse_rest;
  unsigned int flat_ticket;            // the same four for the flat bin
  unsigned int flat_ticket_rest;
  unsigned int flat_huge;
  unsigned int flat_rest;
  unsigned int dense_ticket;           // the same four for the dense bin (huge: kDenseBigSize)
  unsigned int dense_ticket_rest;
  unsigned int dense_huge;
  unsigned int dense_rest;
  int32_t max_dense_work[2];           // largest work of a dense-bin row: big instance, other
  int32_t max_dense_size;              // most vertices of a dense-bin row
  int32_t max_row_size;                // most vertices of a row with work
  int32_t longest_row;                 // most vertices of a row (k_validate)
  // Of a side with thresholds per row (a plan sizes its scratch by these, whatever
  // its bins): most pairs a dense-bin row can have, big instance and other, and
  // largest work of a row that the sparse bin could take.
  int32_t plan_pairs[2];
  int32_t plan_sparse;
  int32_t max_sparse_work;             // largest work of a sparse- or flat-bin row
  int32_t kept;                        // entries of the filtered CSC
  int32_t max_giant_work;              // largest work of a giant-bin row
  unsigned long long nnz_core;         // incidences of the dense core
  int32_t max_row_work;                // largest work of any row
  unsigned long long giant_cycles[4];  // giant bin: SM cycles in walk, partition, buckets; dense bin
  unsigned long long sparse_cycles[5]; // sparse bin: row set-up, walk, collect, emit, staging
  // Every row that emits adds to pairs_bin and to stage_cursor, so they lie more
  // than an L2 line apart (in one line, k_walk_rows of an L_2 of 200K x 400K took
  // 0.41 instead of 0.32 ms).
  unsigned long long stage_cursor;     // staging allocator
  unsigned long long stage_overflow;   // rows that did not fit the staging
};

// Where a device-side check fired (for error reports).
enum Where : int32_t {
  kWhereNone = 0, kWhereRowOffsets = 1, kWhereRowIds = 2, kWhereColOffsets = 3,
  kWhereColIds = 4, kWhereMismatch = 5, kWhereHash = 6, kWhereGiant = 7, kWhereStage = 8,
};

__device__ __forceinline__ void raise_error(Meta *meta, int32_t status, int32_t where) {
  if (atomicCAS(&meta->err, 0, status) == 0) meta->err_where = where;
}

// ------------------------------------------------------------------ scans --

__device__ __forceinline__ int32_t warp_inclusive_scan(int32_t x) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    int32_t y = __shfl_up_sync(0xffffffffu, x, d);
    if (lane >= d) x += y;
  }
  return x;
}

__device__ __forceinline__ long long warp_inclusive_scan64(long long x) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    long long y = __shfl_up_sync(0xffffffffu, x, d);
    if (lane >= d) x += y;
  }
  return x;
}

// Block-wide inclusive scan; `ws` is shared scratch of NT/32 + 1 ints.
// Returns the thread's inclusive prefix, writes the block total to *total.
template <int NT>
__device__ __forceinline__ int32_t block_inclusive_scan(int32_t x, int32_t *ws,
                                                        int32_t *total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  constexpr int NW = NT / 32;
  int32_t inc = warp_inclusive_scan(x);
  if (lane == 31) ws[warp] = inc;
  __syncthreads();
  if (warp == 0) {
    int32_t v = lane < NW ? ws[lane] : 0;
    int32_t vi = warp_inclusive_scan(v);
    if (lane < NW) ws[lane] = vi - v;  // exclusive warp offsets
    if (lane == NW - 1) ws[NW] = vi;
  }
  __syncthreads();
  inc += ws[warp];
  *total = ws[NW];
  __syncthreads();  // ws may be reused right after
  return inc;
}

template <int NT>
__device__ __forceinline__ long long block_inclusive_scan64(long long x, long long *ws,
                                                            long long *total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  constexpr int NW = NT / 32;
  long long inc = warp_inclusive_scan64(x);
  if (lane == 31) ws[warp] = inc;
  __syncthreads();
  if (warp == 0) {
    long long v = lane < NW ? ws[lane] : 0;
    long long vi = warp_inclusive_scan64(v);
    if (lane < NW) ws[lane] = vi - v;
    if (lane == NW - 1) ws[NW] = vi;
  }
  __syncthreads();
  inc += ws[warp];
  *total = ws[NW];
  __syncthreads();
  return inc;
}

// Position of `key` in the ascending array a[lo, hi), or -1.
__device__ __forceinline__ int32_t find_sorted(const int32_t *__restrict__ a, int32_t lo,
                                               int32_t hi, int32_t key) {
  while (lo < hi) {
    int32_t mid = lo + ((hi - lo) >> 1);
    int32_t x = __ldg(a + mid);
    if (x < key) lo = mid + 1;
    else if (x > key) hi = mid;
    else return mid;
  }
  return -1;
}

// The row r with off[r] <= k < off[r + 1] (off ascending, off[0] <= k <
// off[rows]), starting from a row `r` known not to be past it: a few steps
// forward, else a binary search.
__device__ __forceinline__ int32_t row_of(const int32_t *__restrict__ off, int32_t rows, int32_t r,
                                          int32_t k) {
  for (int step = 0; step < 4; ++step) {
    if (__ldg(off + r + 1) > k) return r;
    if (++r >= rows) return rows - 1;
  }
  int32_t lo = r, hi = rows;  // off[lo] <= k < off[hi]
  while (hi - lo > 1) {
    const int32_t mid = lo + ((hi - lo) >> 1);
    if (__ldg(off + mid) <= k) lo = mid;
    else hi = mid;
  }
  return lo;
}

// Multiplicative hash onto [0, T) (Fibonacci hashing + fast range).
__device__ __forceinline__ uint32_t hash_slot(int32_t f, uint32_t T) {
  return __umulhi((uint32_t)f * 0x9E3779B1u, T);
}

// --------------------------------------------------------- wedge walking --
//
// The rows's incidences k in [k0, k1) each own a "tail": the entries after the
// row in the filtered CSC of their column, c_idx_s[tail_beg[k], c_off_s[v+1]).
// The union of the tails (as a multiset) is the row's wedge list.  The walkers
// below flatten the tails and hand every wedge's far end f to `fn`, with the
// work of a batch spread evenly over the threads (load-balanced search over
// the prefix sums of the tail lengths) and coalesced reads of c_idx_s.

struct Walk {
  const int32_t *r_off, *r_idx;      // CSR of the side
  const int32_t *c_idx_s;            // far ends: CSC filtered to rows of size >= s
  const int32_t *tail_beg;           // per CSR incidence: its tail [beg, end)
  const int32_t *tail_end;
};

// CTA-wide walker.  Shared scratch: s_beg[NT], s_pref[NT + 1], ws[NT/32 + 1].
// fn(f, i) receives every wedge's far end f and its index i in the row's
// flattened wedge list (0 .. work-1).
//
// A batch's flattened wedges are cut into chunks
// of 32 G; warp w takes chunks w, w + NT/32, ...; in a chunk, lane l takes
// wedges c0 + 32 g + l (g < G), so every warp-wide load of far ends reads
// 32 consecutive wedges (a few tails) and is coalesced.  The chunk's first
// incidence is found by one binary search (the same address in every lane);
// each lane then steps forward over the incidences its wedges cross.
template <int NT, int G, class Fn>
__device__ __forceinline__ void cta_walk(const Walk &w, int32_t k0, int32_t k1, int32_t *s_beg,
                                         int32_t *s_pref, int32_t *ws, Fn &&fn) {
  const int32_t lane = (int32_t)(threadIdx.x & 31);
  int32_t done = 0;  // wedges of earlier batches
  for (int32_t base = k0; base < k1; base += NT) {
    const int32_t k = base + (int32_t)threadIdx.x;
    int32_t b = 0, len = 0;
    if (k < k1) {
      b = __ldg(w.tail_beg + k);
      len = __ldg(w.tail_end + k) - b;
    }
    int32_t total;
    const int32_t inc = block_inclusive_scan<NT>(len, ws, &total);
    s_beg[threadIdx.x] = b;
    s_pref[threadIdx.x + 1] = inc;
    if (threadIdx.x == 0) s_pref[0] = 0;
    __syncthreads();
    for (int32_t c0 = (int32_t)(threadIdx.x >> 5) * 32 * G; c0 < total; c0 += NT * G) {
      int32_t lo = 0, hi = NT;  // invariant: s_pref[lo] <= c0 < s_pref[hi]
      while (hi - lo > 1) {
        const int32_t mid = (lo + hi) >> 1;
        if (s_pref[mid] <= c0) lo = mid;
        else hi = mid;
      }
      int32_t src[G];
      int32_t j = lo;
#pragma unroll
      for (int g = 0; g < G; ++g) {
        const int32_t i = c0 + 32 * g + lane;
        src[g] = -1;
        if (i < total) {
          while (s_pref[j + 1] <= i) ++j;
          src[g] = s_beg[j] + (i - s_pref[j]);
        }
      }
      int32_t f[G];
#pragma unroll
      for (int g = 0; g < G; ++g) f[g] = src[g] >= 0 ? __ldg(w.c_idx_s + src[g]) : -1;
#pragma unroll
      for (int g = 0; g < G; ++g)
        if (src[g] >= 0) fn(f[g], done + c0 + 32 * g + lane);
    }
    done += total;
    __syncthreads();
  }
}

// ------------------------------------------------------------- launchers --
// All launchers enqueue on `st` and return the first CUDA error, if any.

struct Side {
  int32_t R, C;     // rows (hyperedges of the side), columns (its vertices)
  int64_t nnz;
  const int32_t *r_off, *r_idx, *c_off, *c_idx;
  const int32_t *row_s = nullptr;  // per-row threshold (batched form), else null
  // per-row bound on far ends (batched form: a row's far ends lie below the
  // end of its member's rows), else null: R
  const int32_t *row_fhi = nullptr;
};

// Threshold of row e: its own (batched form) or the call's s.
__device__ __forceinline__ int32_t s_of(const int32_t *row_s, int32_t smin, int32_t e) {
  return row_s ? __ldg(row_s + e) : smin;
}

// Wedge-work thresholds of the bins (runtime; each at most the capacity the
// bin's kernel is compiled for: kWarpMaxWork, kCtaSMaxWork, kCtaLMaxWork).
// `sparse`: rows with s >= 2 that are not dense take the sparse bin up to this
// work (larger ones the giant bin); 0 turns the bin off.  `bloom`: the least
// work of its rows (those of at most `ctas` wedges take the rows bin).
#ifndef SLG_BLOOM_MIN_WORK
#define SLG_BLOOM_MIN_WORK 1024
#endif
// `dense`: scales the dense bin's threshold (see is_dense; 16: as stated there,
// more: more rows are dense).
struct Bins {
  int32_t warp = kWarpMaxWork, ctas = kCtaSMaxWork, ctal = kCtaLMaxWork;
  int32_t sparse = kSparseMaxWork;
  int32_t bloom = SLG_BLOOM_MIN_WORK;
  int32_t dense = kDenseRatio;
  bool flat = true;  // the flat bin is on
};

// Dense core for the tensor-core tile path (all null / 0 when unused).
// Core rows form an ascending list; row_rank / col_rank are exclusive scans
// of the core flags (rank[x+1] != rank[x] marks a core member).  For core
// columns, the entries of the filtered CSC that are not core rows are stored
// at c_idx_s[x_base + x_off[rank] .. x_base + x_off[rank + 1]).  T holds the
// tile counts |e ∩ f ∩ C_c| of core rows, row-major with stride Mp.
struct CoreInfo {
  const int32_t *row_rank, *col_rank;
  const int32_t *x_off;
  int32_t x_base;
  const int32_t *core_list;
  int32_t n_core;
  const int32_t *T;
  int32_t Mp;
};

// Per-call device buffers (carved out of one pool allocation).
struct Work {
  int32_t *csr2csc;    // [nnz] CSC position of every CSR incidence
  int32_t *qs;         // [nnz + 1] exclusive scan of "row of this CSC entry kept"
  int32_t *c_idx_s;    // [nnz] filtered CSC ids
  int32_t *c_off_s;    // [C + 1] filtered CSC offsets
  int32_t *tail_beg;   // [nnz] tail of each incidence: [tail_beg, tail_end)
  int32_t *tail_end;   // [nnz]
  int32_t *tile;       // [ntiles + 1] scan scratch
  int32_t *bin_rows;   // [kNumLists][R] row lists
  int32_t *n_e;        // [R] pairs per row
  int32_t *row_work;   // [R] wedges per row
  long long *stage_pos;// [R] staging offset per row, -1 = not staged
  long long *row_ptr;  // [R + 1] output offsets (relative to row_begin)
  long long *tile64;   // [ntiles64 + 1]
  int32_t *stage_j, *stage_w;  // [stage_cap]
  long long stage_cap;
  Meta *meta;
};

cudaError_t launch_validate(const Side &s, Meta *meta, cudaStream_t st);
cudaError_t launch_csr2csc(const Side &s, int32_t *csr2csc, Meta *meta, cudaStream_t st);
// inv[map[k]] = k (k < n): a permutation's inverse.
cudaError_t launch_invert(const int32_t *map, int64_t n, int32_t *inv, cudaStream_t st);
cudaError_t launch_filter(const Side &s, int32_t smin, const Work &w, cudaStream_t st);
cudaError_t launch_rows_work(const Side &s, int32_t smin, int32_t row_begin, int32_t row_end,
                             const Work &w, const CoreInfo &core, const Bins &bins,
                             cudaStream_t st);

// Dense-core detection / packing (slg_core.cu).
int64_t xscan_tiles(int64_t n);
cudaError_t launch_xscan(const int32_t *in, int32_t *out, int64_t n, int32_t *tile,
                         cudaStream_t st);
cudaError_t launch_core_cols(const Side &s, int32_t tau_c, int32_t *core_col, const Meta *meta,
                             cudaStream_t st);
cudaError_t launch_core_rows(const Side &s, int32_t tau_r, const int32_t *col_rank,
                             int32_t *core_row, unsigned long long *nnz_core, const Meta *meta,
                             cudaStream_t st);
cudaError_t launch_core_list(int32_t R, const int32_t *row_rank, int32_t *core_list,
                             cudaStream_t st);
cudaError_t launch_core_refine(const Side &s, const int32_t *row_rank, int32_t *col_cnt,
                               int32_t tau, int32_t *core_col, const Meta *meta,
                               cudaStream_t st);
cudaError_t launch_core_pack(const Side &s, const int32_t *row_rank, const int32_t *col_rank,
                             uint8_t *A, int32_t Kp, const Meta *meta, cudaStream_t st);
cudaError_t launch_core_xcount(int32_t C, const int32_t *col_rank, const int32_t *c_off_s,
                               const int32_t *c_idx_s, const int32_t *row_rank, int32_t *x_cnt,
                               const Meta *meta, cudaStream_t st);
cudaError_t launch_core_xcsc(int32_t C, const int32_t *col_rank, const int32_t *c_off_s,
                             const int32_t *c_idx_s, const int32_t *row_rank,
                             const int32_t *x_off, int32_t *x_idx, const Meta *meta,
                             cudaStream_t st);
// Output modes of the walk: COUNT (pairs per row only), STAGE (each row's
// sorted pairs appended to a staging area at an atomically reserved offset),
// DIRECT (written to their final place; row_ptr known).
enum Mode : int { kCount = 0, kStage = 1, kDirect = 2 };

struct EmitArgs {
  int mode;
  int unweighted;
  const int32_t *row_s;               // per-row threshold, or null: smin
  const int32_t *row_fhi;             // per-row far-end bound, or null: R
  int full_rows;                      // 1: tails are whole columns, far ends in [0, R)
  const int32_t *row_work;            // [rows] wedges per row (giant bin)
  CoreInfo core;                      // dense core (tile counts added by the giant bin)
  int32_t smin;
  int32_t row_begin;
  int32_t *n_e;                       // [rows] pairs per row
  long long *stage_pos;               // [rows] staging offset, -1 = none
  int32_t *stage_j, *stage_w;         // STAGE
  long long stage_cap;
  const long long *row_ptr;           // DIRECT
  int32_t *out_i, *out_j, *out_w;     // DIRECT
  Meta *meta;
};

struct WalkLaunch {
  Walk w;
  EmitArgs a;
  const int32_t *bin_rows;  // [kNumLists][rows] row lists
  const int32_t *row_work;  // [rows] wedges per row
  int32_t rows;             // rows in the range (list stride)
  int32_t *giant_scratch;   // [giant_ctas][4 * max giant work] wedge ends + pairs; before the
                            // giant kernel, the other bins' scratch one behind the other
  long long giant_stride;   // ints per giant CTA
  int32_t R;                // rows of the side (far ends lie in [0, R))
  int32_t *dense_scratch[2], *sparse_scratch;  // in giant_scratch
  long long sparse_ints;    // of sparse_scratch (the flat kernels' as well: they follow)
  long long dense_pairs[2]; // most pairs a dense-bin row can have: big instance, other (0: no row)
  int32_t dense_size;       // most vertices of a dense-bin row
  unsigned skip;            // bit b: bin b is known to be empty (kSkipSparseBig, ...)
};
// Further bits of WalkLaunch::skip: the two instances of the sparse and flat bins.
constexpr unsigned kSkipSparseBig = 1u << 8, kSkipSparseSmall = 1u << 9;
constexpr unsigned kSkipFlatBig = 1u << 10, kSkipFlatSmall = 1u << 11;

// Sides of at most this many rows take the short path (slg_small.cu).
#ifndef SLG_SMALL_ROWS
#define SLG_SMALL_ROWS 16384
#endif
constexpr int32_t kSmallRows = SLG_SMALL_ROWS;
struct SmallCall {
  Side s;
  int32_t s_prune;               // size from which rows take part
  int32_t row_begin, row_end;
  int32_t *map;                  // [nnz] CSC positions (made unless !validate)
  bool validate;
  uint32_t *active;              // [(R + 31) / 32], zeroed
  EmitArgs a;                    // n_e zeroed; stage_cap = the output's capacity
  int32_t *out_i, *out_j, *out_w;
  long long *row_ptr;            // [rows + 1] or null
  Meta *host;                    // mapped host memory, receives the Meta
  bool hold;                     // the outputs come later (launch_small_emit)
};
cudaError_t launch_small_emit(const SmallCall &c, cudaStream_t st, int32_t *launches);
cudaError_t launch_small(const SmallCall &c, cudaStream_t st, int32_t *launches, cudaEvent_t walk0,
                         cudaEvent_t walk1);

// CTAs of the giant kernel (two per SM); scratch ints of the sparse (and flat) and
// dense kernels.
int giant_ctas();
long long sparse_ints(int32_t max_work);
long long dense_ints(int small, long long pairs, int32_t size_big);
// The largest side (rows) a build supports: row ids and the giant bin's
// super-chunk bounds stay below 2^31.
constexpr int32_t kMaxRows = (int32_t)((1u << 31) - (1u << 23));
// The largest id space of slg_components (its bounded union-find loop).
constexpr int32_t kComponentsMaxR = 1 << 24;

// ev (optional): kNumBins + 1 events recorded before the first and after
// every bin kernel, in launch order (warp, CTA small, CTA large, sparse,
// giant); bin b runs from ev[kWalkEv[b]] to ev[kWalkEv[b] + 1].
constexpr int kWalkEv[kNumBins] = {0, 1, 2, 4, 3};
cudaError_t launch_walk(const WalkLaunch &L, cudaStream_t st, int32_t *launches,
                        cudaEvent_t *ev = nullptr);
cudaError_t launch_walk_rows(const WalkLaunch &L, cudaStream_t st);
cudaError_t launch_walk_sparse(const WalkLaunch &L, cudaStream_t st, int32_t *launches);
cudaError_t launch_join_flat(int32_t *bin_rows, int32_t rows, const Meta &m, Meta *meta,
                             cudaStream_t st);
cudaError_t launch_walk_dense(const WalkLaunch &L, int small, cudaStream_t st);
cudaError_t launch_row_scan(int32_t rows, const Work &w, cudaStream_t st);
// The device Meta into host memory the device can address (mapped pinned
// memory), by a kernel: no copy engine involved.
cudaError_t launch_meta_copy(const Meta *src, Meta *dst, cudaStream_t st);
// w16[i] = w[i] (i < n); *bad = 1 if a weight is above 65,535.
cudaError_t launch_pack_w16(const int32_t *w, int64_t n, uint16_t *w16, int32_t *bad,
                            cudaStream_t st);
// out_cap: entries of the output arrays (with more pairs, or rows that found
// no staging room, nothing is written; strict: that is an error).
cudaError_t launch_gather(int32_t row_begin, int32_t rows, const Work &w, int32_t *out_i,
                          int32_t *out_j, int32_t *out_w, int unweighted, long long out_cap,
                          int strict, cudaStream_t st);

// Batched form (slg_plan.cu): union of many hypergraphs.
struct BatchGraph {            // one member, device pointers
  const int32_t *e_off, *e_idx, *v_off, *v_idx;
  int32_t m, n;
  int64_t nnz;
  int32_t e_base, v_base;      // id offsets in the union
  int64_t k_base;              // incidence offset in the union
  int32_t s;
};
cudaError_t launch_concat(const BatchGraph *g, int32_t count, int32_t max_len, int32_t *e_off,
                          int32_t *e_idx, int32_t *v_off, int32_t *v_idx, int32_t *row_s_e,
                          int32_t *row_s_v, int32_t *row_fhi_e, int32_t *row_fhi_v,
                          cudaStream_t st);
cudaError_t launch_localize(int32_t *out_i, int32_t *out_j, long long pairs,
                            const int32_t *row_base, int32_t count, const long long *row_ptr,
                            long long *offsets, cudaStream_t st);

int giant_ctas_for_device();

// Plain per-hyperedge kernel (comparison): `warps` warps, each with R_pad
// counters in `scratch` and R_pad/1024 bitmap words in `summ`, all zero.
cudaError_t launch_plain(const Side &sd, int32_t smin, int32_t row_begin, int32_t row_end,
                         const EmitArgs &a, int32_t *scratch, uint32_t *summ, int32_t R_pad,
                         int32_t warps, cudaStream_t st);

// Dense-core tile path (tcgen05): C = A·Aᵀ on the upper-triangle 128 x 128
// tiles of an Mp x Kp byte matrix A (0x38 = 1.0).  `tasks` holds room for
// nt (nt + 1) / 2 tile pairs (nt = Mp / 128), `err` one device int.
cudaError_t launch_tile_overlap(const uint8_t *A, int32_t Mp, int32_t Kp, int32_t *C,
                                void *tasks, int32_t *err, cudaStream_t st);
size_t tile_overlap_smem();

// Stable LSD radix sort (slg_sort.cu) by bits [begin_bit, end_bit) of the
// keys, values alongside (vals may be null); tmp buffers of n entries,
// hist of radix_sort_scratch_ints(n) ints; the result ends in keys / vals.
// `launches` (optional) counts the kernels launched.
size_t radix_sort_scratch_ints(int64_t n);
cudaError_t launch_radix_sort(unsigned long long *keys, unsigned long long *keys_tmp,
                              int32_t *vals, int32_t *vals_tmp, int64_t n, int begin_bit,
                              int end_bit, int32_t *hist, cudaStream_t st,
                              int32_t *launches = nullptr);
cudaError_t launch_radix_sort(uint32_t *keys, uint32_t *keys_tmp, int32_t *vals,
                              int32_t *vals_tmp, int64_t n, int begin_bit, int end_bit,
                              int32_t *hist, cudaStream_t st, int32_t *launches = nullptr);

// Degree-ordered relabelling (slg_relabel.cu).
int relabel_row_bits(int32_t R);
size_t relabel_scratch_ints(int32_t R, int64_t nnz);
cudaError_t launch_relabel(const Side &sd, int descending, int32_t *perm, int32_t *r_off2,
                           int32_t *r_idx2, int32_t *c_idx2, int32_t *scratch, cudaStream_t st,
                           int32_t *launches);
cudaError_t launch_unrelabel(int64_t P, int32_t R, const int32_t *perm, int32_t *out_i,
                             int32_t *out_j, int32_t *out_w, unsigned long long *keys,
                             int32_t *vals, int32_t *hist, cudaStream_t st, int32_t *launches);

// Threshold filter of a canonical edge list (slg_sweep.cu): tile counts of
// the triples with w >= s and their exclusive scan in `tile` (keep_tiles(n)
// + 1 entries, tile[keep_tiles(n)] = total), then the ordered compaction.
int64_t keep_tiles(int64_t n);
cudaError_t launch_keep_count(const int32_t *w, int64_t n, int32_t s, long long *tile,
                              cudaStream_t st);
cudaError_t launch_keep_write(const int32_t *in_i, const int32_t *in_j, const int32_t *in_w,
                              int64_t n, int32_t s, const long long *tile, int32_t *out_i,
                              int32_t *out_j, int32_t *out_w, int64_t capacity,
                              cudaStream_t st);

// After the edge list (slg_post.cu): ID squeezing, adjacency, components.
// Each checks its pairs first; *err (zeroed by the caller) tells the result.
cudaError_t launch_squeeze(const int32_t *a, const int32_t *b, int64_t n, int32_t R,
                           uint32_t *bits, int32_t *cnt, int32_t *rank, void *word,
                           int32_t *tile, int32_t *oa, int32_t *ob, int32_t *old_of_new,
                           int32_t *err, cudaStream_t st);
int adjacency_passes(int32_t V);
size_t adjacency_scratch_ints(int64_t n);
cudaError_t launch_adjacency(const int32_t *a, const int32_t *b, const int32_t *w, int64_t n,
                             int32_t V, int32_t *first, int32_t *last, int32_t *U, int32_t *L,
                             int32_t *tile, uint32_t *const key[2], int32_t *const vi[2],
                             int32_t *const vw[2], int32_t *hist, long long *off, int32_t *adj,
                             int32_t *adj_w, int32_t *err, cudaStream_t st);
cudaError_t launch_components(const int32_t *a, const int32_t *b, int64_t n, int32_t R,
                              int32_t *labels, int32_t *child, unsigned long long *n_comp,
                              int32_t *err, cudaStream_t st);

// Filtered SpGEMM comparison: full-column tails / per-row work, filtration.
cudaError_t launch_rows_full(const Side &sd, int32_t row_begin, int32_t row_end,
                             int32_t list_base, int32_t *tail_beg, int32_t *tail_end,
                             int32_t *work_out,
                             int32_t *n_e, long long *stage_pos, int32_t *bin_rows,
                             int32_t list_stride, Meta *meta, cudaStream_t st);
cudaError_t launch_filter_count(int32_t row_begin, int32_t row_end, int32_t list_base,
                                const Work &w, int32_t smin, int32_t *kept, cudaStream_t st);
cudaError_t launch_filter_write(int32_t row_begin, int32_t row_end, int32_t list_base,
                                const Work &w, int32_t smin, const long long *row_ptr,
                                long long out_base, int unweighted, int32_t *out_i,
                                int32_t *out_j, int32_t *out_w, cudaStream_t st);

}  // namespace slg
