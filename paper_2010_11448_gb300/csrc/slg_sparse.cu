// The sparse bin of the s-overlap walk.
//
// Large rows whose far ends are sparse in their id span, with s >= 2.  Almost
// every far end of such a row occurs once (on the Chung-Lu workloads about
// 96 % of the wedges of these rows are the only wedge to their far end), and
// a far end with a single wedge can never reach s >= 2.  The row is counted
// in two passes with little shared memory, so that several rows are in
// flight on each SM (the walk's far-end gathers are latency-bound: a row at
// a time per SM leaves the memory system idle):
//   1. every wedge sets its far end's bit in a one-hash Bloom filter (one
//      shared atomicOr); a wedge that finds the bit already set makes f a
//      candidate: f is claimed in a small shared table (key, count 0) and
//      marked in a second filter.  Every f with two or more wedges becomes
//      a candidate (its second wedge finds the bit set); so may a few
//      single-wedge f whose bit another f had set;
//   2. a second pass counts, exactly, every wedge whose far end is a
//      candidate (the second filter screens out almost all others before
//      the table is probed).  The count of f is then |e ∩ f|.  It reads the
//      row's far ends from a copy the first walk wrote to global scratch
//      (or, for a row of at most kSpCache wedges, to shared memory), or
//      walks the tails again when there is no room for the copy.
// The candidates with count >= s are sorted and emitted.  A row whose
// candidates overflow the table (a probe sequence longer than kSpMaxProbe)
// is handed to the giant bin, which runs after this one.
// Two instances of the kernel share the bin: rows above kSparseBigWork go
// to one with a 2^SLG_SP_LGT-slot table, the rest to one with a
// 2^SLG_SP_SMALL_LGT-slot table, whose smaller shared memory leaves room for
// one more resident CTA per SM.  Rows of up to 8192 wedges seldom have more
// candidates or survivors than the smaller table holds (the overflow would
// send them to the giant bin); rows of up to 16384 do.

#include <algorithm>
#include <mutex>

#include "slg_walk.cuh"

namespace slg {

namespace {

#ifndef SLG_SP_NT
#define SLG_SP_NT 256
#endif
#ifndef SLG_SP_LOGB
#define SLG_SP_LOGB 17
#endif
#ifndef SLG_SP_LGT
#define SLG_SP_LGT 12
#endif
#ifndef SLG_SP_CACHE
#define SLG_SP_CACHE 0
#endif
#ifndef SLG_SP_MINB
#define SLG_SP_MINB 4
#endif
#ifndef SLG_SP_SMALL_LGT
#define SLG_SP_SMALL_LGT 11
#endif
#ifndef SLG_SP_SMALL_MINB
#define SLG_SP_SMALL_MINB 5
#endif
#ifndef SLG_SP_G
#define SLG_SP_G 6
#endif
#ifndef SLG_SP_RUNS
#define SLG_SP_RUNS 1  // order survivor sets above 64 by sorted warp runs
#endif
constexpr int kSpNT = SLG_SP_NT;
constexpr int kSpLogB = SLG_SP_LOGB;          // Bloom filter bits (log2)
constexpr int kSpWords = 1 << (kSpLogB - 5);
constexpr int kSpCWords = kSpWords / 4;       // candidate filter words
constexpr int kSpLgT = SLG_SP_LGT;            // candidate table slots (log2)
constexpr int kSpSmallLgT = SLG_SP_SMALL_LGT;  // the same, rows up to kSparseBigWork
constexpr int kSpCache = SLG_SP_CACHE;        // far ends kept of a small row
constexpr int kSpMaxProbe = 32;
constexpr int kSpG = SLG_SP_G;                // wedges per thread per walk step
static_assert((1 << kSpSmallLgT) >= kSpNT && kSpSmallLgT <= kSpLgT &&
                  kSpWords % (4 * kSpNT) == 0 && kSpCWords % 4 == 0,
              "sparse bin geometry");

// [s_base 8][s_ovf 4][s_row 4][pad 16][filter kSpWords x 4]
// [candidate filter kSpCWords x 4][table 2^lgt x 8][cache kSpCache x 4]
// [s_beg NT][s_pref NT+1][ws NT/32+1]
constexpr size_t sparse_smem(int lgt) {
  return 32 + (size_t)kSpWords * 4 + (size_t)kSpCWords * 4 + ((size_t)8 << lgt) +
         (size_t)kSpCache * 4 + (size_t)(2 * kSpNT + 1 + kSpNT / 32 + 1) * 4;
}

// A row's filter has 2^lgb bits (its candidate filter 2^(lgb - 2)) and its
// table 2^lgt slots, sized by the row's work (see sp_sizes).
__device__ __forceinline__ uint32_t sp_h1(int32_t f, int lgb) {  // Bloom filter bit
  return ((uint32_t)f * 0x9E3779B1u) >> (32 - lgb);
}
__device__ __forceinline__ uint32_t sp_h2(int32_t f, int lgb) {  // candidate filter bit
  return ((uint32_t)f * 0x85EBCA6Bu) >> (34 - lgb);
}
__device__ __forceinline__ uint32_t sp_ht(int32_t f, int lgt) {  // candidate table slot
  return ((uint32_t)f * 0xC2B2AE35u) >> (32 - lgt);
}

// Per-row sizes: a filter of >= 32 bits per wedge (so that a single-wedge
// far end finds its bit set by another with probability below 1/64 on
// average) and a table of >= one slot per wedge (every candidate has two
// wedges or is such a collision), within the shared-memory maxima (a table
// of at most 2^max_lgt slots).
__device__ __forceinline__ void sp_sizes(int32_t work, int max_lgt, int *lgb, int *lgt) {
  const int lw = ceil_log2(work > 1 ? work : 2);
  *lgb = min(max(lw + 5, 12), kSpLogB);
  *lgt = min(max(lw, 7), max_lgt);
}

// Pass 1: f is a candidate (its filter bit was already set).  Claims f's
// table slot (32-bit CAS on the key word; the count word stays 0) unless it
// is there already, and marks it in the candidate filter.  A probe sequence
// longer than kSpMaxProbe marks the row as overflowed.
__device__ __forceinline__ void sp_candidate(unsigned long long *tab, uint32_t *cand, int32_t f,
                                             int32_t *s_ovf, int lgb, int lgt) {
  if (*(volatile int32_t *)s_ovf) return;
  const uint32_t mask = (1u << lgt) - 1u;
  uint32_t h = sp_ht(f, lgt);
  for (int probe = 0; probe < kSpMaxProbe; ++probe) {
    const uint32_t k = atomicCAS(count_word(tab, h) + 1, 0xFFFFFFFFu, (uint32_t)f);
    if (k == 0xFFFFFFFFu) {
      const uint32_t c = sp_h2(f, lgb);
      atomicOr(cand + (c >> 5), 1u << (c & 31));
      return;
    }
    if (k == (uint32_t)f) return;
    h = (h + 1) & mask;
  }
  *(volatile int32_t *)s_ovf = 1;
}

// Pass 2, for an f that passed the candidate filter: counted if it is in
// the table.  Unweighted: a count that reached s is not raised further.
__device__ __forceinline__ void sp_count_listed(unsigned long long *tab, int32_t f, int32_t smin,
                                                bool unweighted, int lgt) {
  const uint32_t mask = (1u << lgt) - 1u;
  uint32_t h = sp_ht(f, lgt);
  for (int probe = 0; probe < kSpMaxProbe; ++probe) {
    uint32_t *cw = count_word(tab, h);
    const uint32_t k = cw[1];
    if (k == (uint32_t)f) {
      if (!unweighted || (int32_t)*(volatile uint32_t *)cw < smin) atomicAdd(cw, 1u);
      return;
    }
    if (k == 0xFFFFFFFFu) return;
    h = (h + 1) & mask;
  }
}

// Pass 2: one wedge to f; counted when f is a candidate.
__device__ __forceinline__ void sp_count(unsigned long long *tab, const uint32_t *cand,
                                         int32_t f, int32_t smin, bool unweighted, int lgb,
                                         int lgt) {
  const uint32_t c = sp_h2(f, lgb);
  if (!(cand[c >> 5] & (1u << (c & 31)))) return;
  sp_count_listed(tab, f, smin, unweighted, lgt);
}

// A lane's few wedges of a walk step that take the slow path (candidate
// claims in pass 1, counts in pass 2: a small fraction of the wedges) are
// gathered in registers and handled in rounds, the q-th round taking every
// lane's q-th one, so that a warp runs max over its lanes rounds instead of
// one round per wedge slot of the step with a lane or two active.
#ifndef SLG_SP_DEFER
#define SLG_SP_DEFER 1
#endif
template <int G>
__device__ __forceinline__ void pend_push(int32_t (&pend)[G], int &np, bool c, int32_t f, int g) {
#pragma unroll
  for (int q = 0; q < G; ++q)  // selects: no local memory
    if (q <= g) pend[q] = (c && q == np) ? f : pend[q];
  np += c;
}

// The first walk also copies the row's far ends (in flattened wedge order) to
// the CTA's part of the giant bin's scratch (free while this kernel runs:
// the giant bin runs after it), so that the second pass reads them in order
// instead of walking the tails again.  buf_stride: ints per CTA (0: none).
#ifndef SLG_SP_GBUF
#define SLG_SP_GBUF 1
#endif
// part: 0 every row of the bin, 1 the rows handed out first (the front of
// the list), 2 the others (the back of the list, on their own ticket).
template <int LGT, int MINB>
__global__ __launch_bounds__(kSpNT, MINB) void k_walk_sparse(
    Walk w, const int32_t *__restrict__ rows, EmitArgs a, int32_t *__restrict__ giant_rows,
    int32_t list_len, int32_t *__restrict__ buf, long long buf_stride, int part) {
  constexpr int kT = 1 << LGT;        // candidate table slots
  constexpr int kSPT = kT / kSpNT;    // table slots per thread
  Meta *meta = a.meta;
  if (meta->err) return;
  extern __shared__ __align__(16) unsigned char smem[];
  long long *s_base = reinterpret_cast<long long *>(smem);
  int32_t *s_ovf = reinterpret_cast<int32_t *>(smem + 8);
  int32_t *s_row = reinterpret_cast<int32_t *>(smem + 12);
  uint32_t *filt = reinterpret_cast<uint32_t *>(smem + 32);
  uint32_t *cand = filt + kSpWords;
  unsigned long long *tab = reinterpret_cast<unsigned long long *>(cand + kSpCWords);
  int32_t *cache = reinterpret_cast<int32_t *>(tab + kT);
  int32_t *s_beg = cache + kSpCache;
  int32_t *s_pref = s_beg + kSpNT;
  int32_t *ws = s_pref + kSpNT + 1;
  const int32_t tid = (int32_t)threadIdx.x;
  // clears the first 2^(lgb - 5) filter words and 2^(lgb - 7) candidate
  // filter words (>= 128 and 32: whole uint4 groups)
  auto clear_filters = [&](int lgb) {
    uint4 *f4 = reinterpret_cast<uint4 *>(filt);
    for (int i = tid; i < (1 << (lgb - 7)); i += kSpNT) f4[i] = make_uint4(0, 0, 0, 0);
    uint4 *c4 = reinterpret_cast<uint4 *>(cand);
    for (int i = tid; i < (1 << (lgb - 9)); i += kSpNT) c4[i] = make_uint4(0, 0, 0, 0);
  };
  clear_filters(kSpLogB);
  for (int i = tid; i < kT; i += kSpNT) tab[i] = kEmpty64;
  const unsigned nrows = (unsigned)meta->rows_bin[kBinSparse];
  const unsigned nhuge = meta->sparse_huge;
  unsigned *ticket = part == 2 ? &meta->sparse_ticket_rest : &meta->sparse_ticket;
  const unsigned t_first = part == 2 ? nhuge : 0u;
  const unsigned t_end = part == 1 ? nhuge : nrows;
  const bool unweighted = a.unweighted != 0;
  const bool emit = a.mode != kCount;
  // SM cycles of the CTA's first thread: row set-up, first walk, second
  // walk, collect and order, emit and clear
  long long cyc[5] = {0, 0, 0, 0, 0};
  for (;;) {
    long long t0 = clock64();
    __syncthreads();  // the previous row's clears done
    if (tid == 0) {
      const unsigned t = t_first + atomicAdd(ticket, 1u);
      *s_ovf = 0;
      *s_row = t >= t_end ? -1 : rows[t < nhuge ? t : list_len - 1 - (t - nhuge)];
    }
    __syncthreads();
    const int32_t e = *s_row;
    if (e < 0) break;
    const int32_t smin = s_of(a.row_s, a.smin, e);
    const int32_t work = a.row_work[e - a.row_begin];
    const int32_t k0 = w.r_off[e], k1 = w.r_off[e + 1];
    const bool cached = work <= kSpCache;
    // the far ends kept in global scratch for the second pass (uniform)
    int32_t *gbuf = (SLG_SP_GBUF && !cached && (long long)work <= buf_stride)
                        ? buf + (long long)blockIdx.x * buf_stride
                        : nullptr;
    int lgb, lgt;
    sp_sizes(work, LGT, &lgb, &lgt);
    const int32_t T = 1 << lgt;
    {
      const long long t1 = clock64();
      cyc[0] += t1 - t0;
      t0 = t1;
    }
    // 1. filter; candidates (a thread's G filter updates are in flight together)
    cta_walk_batched<kSpNT, kSpG>(
        w, k0, k1, s_beg, s_pref, ws, [&](const int32_t(&f)[kSpG], int32_t i0) {
          uint32_t old[kSpG], m[kSpG];
#pragma unroll
          for (int g = 0; g < kSpG; ++g) {
            if (cached && f[g] >= 0) cache[i0 + 32 * g] = f[g];
            if (gbuf && f[g] >= 0) gbuf[i0 + 32 * g] = f[g];
            const uint32_t h = sp_h1(f[g], lgb);
            m[g] = f[g] >= 0 ? 1u << (h & 31) : 0u;
            old[g] = f[g] >= 0 ? atomicOr(filt + (h >> 5), m[g]) : 0u;
          }
#if SLG_SP_DEFER
          int32_t pend[kSpG] = {};
          int np = 0;
#pragma unroll
          for (int g = 0; g < kSpG; ++g) pend_push(pend, np, (old[g] & m[g]) != 0, f[g], g);
#pragma unroll
          for (int q = 0; q < kSpG; ++q) {
            if (!__any_sync(0xffffffffu, q < np)) break;
            if (q < np) sp_candidate(tab, cand, pend[q], s_ovf, lgb, lgt);
          }
#else
#pragma unroll
          for (int g = 0; g < kSpG; ++g)
            if (old[g] & m[g]) sp_candidate(tab, cand, f[g], s_ovf, lgb, lgt);
#endif
        });
    __syncthreads();  // candidates final
    {
      const long long t1 = clock64();
      cyc[1] += t1 - t0;
      t0 = t1;
    }
    if (*s_ovf) {  // uniform: too many candidates for the table
      if (tid == 0) {
        // hand the row to the giant bin (launched after this kernel)
        const unsigned pos = atomicAdd(&meta->giant_rest, 1u);
        giant_rows[list_len - 1 - pos] = e;
        atomicAdd(&meta->rows_bin[kBinGiant], 1ull);
      }
      clear_filters(lgb);
      for (int i = tid; i < T; i += kSpNT) tab[i] = kEmpty64;
      continue;
    }
    // 2. exact counts of the candidates
    // (the deferred slow path, as in the walk below)
    auto count_step = [&](const int32_t(&f)[kSpG]) {
      uint32_t word[kSpG], bit[kSpG];
#pragma unroll
      for (int g = 0; g < kSpG; ++g) {  // the candidate filter, loads in flight together
        const uint32_t c = sp_h2(f[g], lgb);
        bit[g] = 1u << (c & 31);
        word[g] = f[g] >= 0 ? cand[c >> 5] : 0u;
      }
      int32_t pend[kSpG] = {};
      int np = 0;
#pragma unroll
      for (int g = 0; g < kSpG; ++g) pend_push(pend, np, (word[g] & bit[g]) != 0, f[g], g);
#pragma unroll
      for (int q = 0; q < kSpG; ++q) {
        if (!__any_sync(0xffffffffu, q < np)) break;
        if (q < np) sp_count_listed(tab, pend[q], smin, unweighted, lgt);
      }
    };
    if (gbuf) {
      // warp-uniform steps over the copy, 32 consecutive far ends per load
      const int32_t lane = tid & 31;
      for (int32_t b0 = (tid >> 5) * 32 * kSpG; b0 < work; b0 += kSpNT * kSpG) {
        int32_t f[kSpG];
#pragma unroll
        for (int g = 0; g < kSpG; ++g) {
          const int32_t i = b0 + 32 * g + lane;
          f[g] = i < work ? gbuf[i] : -1;
        }
        count_step(f);
      }
      __syncthreads();  // every read of the copy done
      l2_discard(gbuf, work);
    } else if (cached) {
      for (int32_t i = tid; i < work; i += kSpNT)
        sp_count(tab, cand, cache[i], smin, unweighted, lgb, lgt);
    } else {
      cta_walk_batched<kSpNT, kSpG>(
          w, k0, k1, s_beg, s_pref, ws, [&](const int32_t(&f)[kSpG], int32_t) {
#if SLG_SP_DEFER
            uint32_t word[kSpG], bit[kSpG];
#pragma unroll
            for (int g = 0; g < kSpG; ++g) {  // the candidate filter, loads in flight together
              const uint32_t c = sp_h2(f[g], lgb);
              bit[g] = 1u << (c & 31);
              word[g] = f[g] >= 0 ? cand[c >> 5] : 0u;
            }
            int32_t pend[kSpG] = {};
            int np = 0;
#pragma unroll
            for (int g = 0; g < kSpG; ++g) pend_push(pend, np, (word[g] & bit[g]) != 0, f[g], g);
#pragma unroll
            for (int q = 0; q < kSpG; ++q) {
              if (!__any_sync(0xffffffffu, q < np)) break;
              if (q < np) sp_count_listed(tab, pend[q], smin, unweighted, lgt);
            }
#else
#pragma unroll
            for (int g = 0; g < kSpG; ++g)
              if (f[g] >= 0) sp_count(tab, cand, f[g], smin, unweighted, lgb, lgt);
#endif
          });
    }
    __syncthreads();  // counts final
    {
      const long long t1 = clock64();
      cyc[2] += t1 - t0;
      t0 = t1;
    }
    // 3. candidates with count >= s, in ascending f at tab[at, at + n)
    int32_t at = 0, used = T;
    // (ordering n survivors needs 2 n + 32 slots of the table)
    const int32_t n = table_collect<kSpNT, kSPT, (SLG_SP_RUNS != 0)>(
        tab, T, smin, emit, ws, &at, &used, (T - 32) / 2);
    if (n < 0) {  // uniform: hand the row to the giant bin, as for an overflow
      __syncthreads();
      if (tid == 0) {
        const unsigned pos = atomicAdd(&meta->giant_rest, 1u);
        giant_rows[list_len - 1 - pos] = e;
        atomicAdd(&meta->rows_bin[kBinGiant], 1ull);
      }
      clear_filters(lgb);
      for (int i = tid; i < T; i += kSpNT) tab[i] = kEmpty64;
      continue;
    }
    if (tid == 0) *s_base = reserve(a, e, n, kBinSparse);
    __syncthreads();
    {
      const long long t1 = clock64();
      cyc[3] += t1 - t0;
      t0 = t1;
    }
    const long long base = *s_base;
    if (emit && base >= 0)
      for (int32_t i = tid; i < n; i += kSpNT) {
        const unsigned long long x = tab[at + i];
        const int32_t f = (int32_t)(x >> 32), c = (int32_t)(uint32_t)x;
        put(a, base, i, e, f, c);
      }
    clear_filters(lgb);  // nothing reads the filters after the second pass
    table_reset_front<kSpNT>(tab, used);
    cyc[4] += clock64() - t0;
  }
  if (tid == 0)
    for (int q = 0; q < 5; ++q) atomicAdd(&meta->sparse_cycles[q], (unsigned long long)cyc[q]);
}

#define K_SP_BIG k_walk_sparse<kSpLgT, SLG_SP_MINB>
#define K_SP_SMALL k_walk_sparse<kSpSmallLgT, SLG_SP_SMALL_MINB>

struct SpOcc {
  int big = 0, small = 0;  // CTAs
  int dev = -1;
};

SpOcc &sp_occ() {
  static SpOcc occ[64];
  static std::mutex mu;
  int dev = 0;
  cudaGetDevice(&dev);
  SpOcc &o = occ[dev & 63];
  std::lock_guard<std::mutex> lock(mu);
  if (o.dev != dev) {
    int sms = 0, nb = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaFuncSetAttribute(K_SP_BIG, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)sparse_smem(kSpLgT));
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, K_SP_BIG, kSpNT, sparse_smem(kSpLgT));
    o.big = sms * std::max(nb, 1);
    cudaFuncSetAttribute(K_SP_SMALL, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)sparse_smem(kSpSmallLgT));
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, K_SP_SMALL, kSpNT,
                                                  sparse_smem(kSpSmallLgT));
    o.small = sms * std::max(nb, 1);
    o.dev = dev;
  }
  return o;
}

}  // namespace

int sparse_ctas() { return std::max(sp_occ().big, sp_occ().small); }

cudaError_t launch_walk_sparse(const WalkLaunch &L, cudaStream_t st, int32_t *launches) {
  SpOcc &o = sp_occ();
  const int64_t stride = L.rows;
  // the CTAs share the giant bin's scratch out (it holds at least
  // 4 x max(giant, sparse row work) ints per giant CTA)
  auto buf_stride = [&](int ctas) -> long long {
    return L.giant_scratch ? (L.scratch_ints / (long long)ctas) & ~31ll : 0;
  };
  const int32_t *rows = L.bin_rows + (int64_t)kBinSparse * stride;
  int32_t *giant_list = const_cast<int32_t *>(L.bin_rows) + (int64_t)kBinGiant * stride;
  K_SP_BIG<<<o.big, kSpNT, sparse_smem(kSpLgT), st>>>(L.w, rows, L.a, giant_list, (int32_t)stride,
                                                      L.giant_scratch, buf_stride(o.big),
                                                      SLG_SP_BIG_WORK > 0 ? 1 : 0);
  ++*launches;
  if (SLG_SP_BIG_WORK > 0) {
    K_SP_SMALL<<<o.small, kSpNT, sparse_smem(kSpSmallLgT), st>>>(
        L.w, rows, L.a, giant_list, (int32_t)stride, L.giant_scratch, buf_stride(o.small), 2);
    ++*launches;
  }
  return cudaGetLastError();
}

}  // namespace slg
