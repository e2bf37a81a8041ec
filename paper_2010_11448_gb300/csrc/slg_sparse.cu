// The sparse bin of the s-overlap walk: rows with s >= 2 whose far ends are
// sparse in their id span.
//
// Almost every far end of such a row occurs once (on the Chung-Lu workloads
// about 96 % of the wedges are the only wedge to their far end), and a far
// end with a single wedge can never reach s >= 2.  Moreover a far end f with
// |e ∩ f| >= s meets e outside any s - 1 of e's vertices: with the row's t <=
// s - 1 longest tails set aside, f still has s - t wedges in the others.  The
// tails are very unequal (on L_8 of the dual of chung_lu_1m the six longest
// hold nine tenths of such a row's wedges), so most wedges are only looked
// up, never inserted anywhere:
//   1. every wedge of the inserted tails sets its far end's bit in a Bloom
//      filter `once` (one shared atomicOr); a wedge that finds the bit set
//      also sets it in a second filter `twice`;
//   2. s <= 3, one tail set aside: a far end of that tail whose bit is set
//      in `once` is marked in `twice` and counted in a small shared table
//      (a tail holds each far end at most once);
//   3. the inserted tails are read again; a far end whose bit is set in
//      `twice` is counted in the table.  s > 3, s - 2 tails set aside: theirs
//      are read too.  Every f with |e ∩ f| >= s passes in each of its wedges
//      (it has s - t >= 2 inserted wedges, or, s <= 3, one and one in the
//      tail set aside), so its count is exact;
//   4. the far ends whose count reached s, listed as they did, are ranked
//      and written.
// A warp takes a segment of a tail at a time (consecutive far ends: no
// search for a wedge's tail); the few far ends that pass a filter are queued
// and counted by whole warps.
//
// Rows above kSpChunk (s > 3: kSpChunkAside) wedges are processed in several ranges of ids, so that
// a range's far ends fit the filter and the table.  A range that overflows
// the table (a probe sequence longer than kSpMaxProbe) is repeated with the
// largest one; one that overflows that, or has more survivors than can be
// ordered, with half the ids (a row that still fails with 64 ids would be
// handed to the giant bin, which runs after this one).
//
// Rows of at most kCtaSMaxWork wedges are counted in the same way by one warp
// each (k_walk_rows), with nothing but warp-wide steps; rows of many short tails
// by a kernel that flattens them (k_walk_flat).
//
// Bound by instruction issue (70 % of issue slots) and the latency of the
// dependent steps of a row, with five rows in flight per SM.
#include <algorithm>
#include <mutex>

#include "slg_walk.cuh"

namespace slg {

namespace {

#ifndef SLG_SP_LOGB
#define SLG_SP_LOGB 16
#endif
#ifndef SLG_SP_NT
#define SLG_SP_NT 256
#endif
#ifndef SLG_SP_MINB
#define SLG_SP_MINB 5
#endif
#ifndef SLG_SP_LGT
#define SLG_SP_LGT 11
#endif
#ifndef SLG_SP_BIG_NT
#define SLG_SP_BIG_NT 512
#endif
#ifndef SLG_SP_BIG_MINB
#define SLG_SP_BIG_MINB 3
#endif
#ifndef SLG_SP_G
#define SLG_SP_G 4
#endif
#ifndef SLG_SP_CHUNK
#define SLG_SP_CHUNK 12288
#endif
#ifndef SLG_SP_CHUNK_ASIDE
#define SLG_SP_CHUNK_ASIDE 32768
#endif
#ifndef SLG_SP_DROP
#define SLG_SP_DROP 16
#endif
constexpr int kSpLogB = SLG_SP_LOGB;          // bits of each filter (log2)
constexpr int kSpWords = 1 << (kSpLogB - 5);
constexpr int kSpMaxProbe = 32;
constexpr int kSpG = SLG_SP_G;                // wedges per thread per step
constexpr int kSpSeg = 32 * kSpG;             // far ends per segment of a tail
constexpr int32_t kSpChunk = SLG_SP_CHUNK;    // a row's wedges per id range, about
constexpr int32_t kSpChunkAside = SLG_SP_CHUNK_ASIDE;  // s > 3 (most wedges are set aside)
constexpr int kSpDrop = SLG_SP_DROP;          // tails set aside, at most
constexpr int kSpQ = 32 + kSpSeg;             // queued far ends per warp
constexpr int kSpList = kSpWords;             // listed survivors, at most (in `once`)
constexpr int kSpSortMax = kSpWords / 2 - 32;  // of which ordered in `twice`
constexpr int kSpRegQ = 4;                    // more: ordered in the table, 4 per thread

// The two instances of the kernel: NT threads, tables of up to 2^LGT slots,
// MINB CTAs per SM, tails of up to MAXW wedges in all.
struct SpSmall {  // rows of at most kSparseBigWork wedges
  static constexpr int NT = SLG_SP_NT, LGT = SLG_SP_LGT, MINB = SLG_SP_MINB;
  static constexpr int32_t MAXW = kSparseBigWork;
};
struct SpBig {
  static constexpr int NT = SLG_SP_BIG_NT, LGT = 12, MINB = SLG_SP_BIG_MINB;
  static constexpr int32_t MAXW = kSparseMaxWork;
};
template <class C>
constexpr int sp_max_seg() {  // segments of a batch of NT tails
  return C::MAXW / kSpSeg + C::NT;
}

// [s_base 8][s_ovf 4][s_row 4][s_any 4][s_sum 4][s_nsurv 4][pad 4][s_cyc 6 x 8][once][twice]
// [table x 8][segments x 8][lengths NT][ws NT/32+1][queues]
template <class C>
constexpr size_t sparse_smem() {
  static_assert(kSpWords % (4 * C::NT) == 0 && sp_max_seg<C>() < 65536 &&
                    kSpList <= 2 * (1 << C::LGT) && 2 * C::NT * kSpRegQ <= (1 << C::LGT),
                "sparse bin geometry");
  return 80 + (size_t)kSpWords * 8 + (size_t)((1 << C::LGT) + 32) * 8 +
         (size_t)sp_max_seg<C>() * 8 +
         (size_t)(C::NT + C::NT / 32 + 1 + C::NT / 32 * kSpQ) * 4;
}

__device__ __forceinline__ uint32_t sp_bit(int32_t f, int lgb) {  // filter bit
  return ((uint32_t)f * 0x9E3779B1u) >> (32 - lgb);
}

// One wedge to f, counted in the table: the key word is claimed with a 32-bit
// CAS and the claim stands for one wedge (the count word holds count - 1).  A
// far end whose count reaches s (>= 2) appends its slot to the survivors.
// Unweighted: a count that reached s is not raised further.  A probe sequence
// longer than kSpMaxProbe marks the range as overflowed.
__device__ __forceinline__ void sp_insert(unsigned long long *tab, int32_t f, int32_t smin,
                                          bool unweighted, int lgt, int32_t *s_ovf,
                                          int32_t *list, int32_t list_cap, int32_t *s_nsurv) {
  const uint32_t mask = (1u << lgt) - 1u;
  uint32_t h = ((uint32_t)f * 0xC2B2AE35u) >> (32 - lgt);
  for (int probe = 0; probe < kSpMaxProbe; ++probe) {
    uint32_t *cw = count_word(tab, h);
    const uint32_t k = atomicCAS(cw + 1, 0xFFFFFFFFu, (uint32_t)f);
    if (k == 0xFFFFFFFFu) return;
    if (k == (uint32_t)f) {
      if (unweighted && (int32_t)*(volatile uint32_t *)cw + 1 >= smin) return;
      if ((int32_t)atomicAdd(cw, 1u) == smin - 2) {
        const int32_t p = atomicAdd(s_nsurv, 1);
        if (p < list_cap) list[p] = (int32_t)h;
      }
      return;
    }
    h = (h + 1) & mask;
  }
  *(volatile int32_t *)s_ovf = 1;
}

// A warp's queue of far ends to count (a few per hundred wedges).  They are
// gathered in shared memory and handled 32 at a time, so that the counting
// runs with whole warps; its code is there once per pass (the unrolled steps
// only append), which keeps the passes within the instruction cache.
struct SpQueue {
  int32_t *q;  // kSpQ entries of this warp
  int n;       // queued (warp-uniform), below 32 between steps
  __device__ __forceinline__ void push(bool c, int32_t f) {
    const unsigned bal = __ballot_sync(0xffffffffu, c);
    if (c) q[n + __popc(bal & ((1u << (threadIdx.x & 31)) - 1u))] = f;
    n += __popc(bal);
  }
  // fn(f) for whole warps of queued far ends; with `all`, for every one
  template <class Fn>
  __device__ __forceinline__ void drain(bool all, Fn &&fn) {
    if (n < (all ? 1 : 32)) return;
    __syncwarp();
    const int lane = threadIdx.x & 31;
    do {
      const int take = min(n, 32);
      n -= take;
      if (lane < take) fn(q[n + lane]);
    } while (n >= (all ? 1 : 32));
    __syncwarp();
  }
};

// First position in the ascending a[lo, hi) with a value >= x.
__device__ __forceinline__ int32_t lower_pos(const int32_t *__restrict__ a, int32_t lo, int32_t hi,
                                             int32_t x) {
  while (lo < hi) {
    const int32_t mid = lo + ((hi - lo) >> 1);
    if (__ldg(a + mid) < x) lo = mid + 1;
    else hi = mid;
  }
  return lo;
}

// part 0: the rows above kSparseBigWork wedges (the front of the list), 1: the
// others (its back), each on its own ticket.  buf: the CTA's share of the
// bin's scratch, for the pairs of rows of
// several ranges: buf_stride ints, at least the largest row's work.
template <class C>
__global__ __launch_bounds__(C::NT, C::MINB) void k_walk_sparse(
    Walk w, const int32_t *__restrict__ rows, EmitArgs a, int32_t *__restrict__ giant_rows,
    int32_t list_len, int32_t *__restrict__ buf, long long buf_stride, int32_t R, int part) {
  constexpr int NT = C::NT, NW = NT / 32, kSpT = 1 << C::LGT;
  Meta *meta = a.meta;
  if (meta->err) return;
  extern __shared__ __align__(16) unsigned char smem[];
  long long *s_base = reinterpret_cast<long long *>(smem);
  int32_t *s_ovf = reinterpret_cast<int32_t *>(smem + 8);
  int32_t *s_row = reinterpret_cast<int32_t *>(smem + 12);
  int32_t *s_any = reinterpret_cast<int32_t *>(smem + 16);
  int32_t *s_sum = reinterpret_cast<int32_t *>(smem + 20);
  int32_t *s_nsurv = reinterpret_cast<int32_t *>(smem + 24);
  // SM cycles of the CTA's first thread: row set-up, first pass, second
  // pass, order and write, clear; the last lap's time
  long long *s_cyc = reinterpret_cast<long long *>(smem + 32);
  uint32_t *once = reinterpret_cast<uint32_t *>(smem + 80);
  uint32_t *twice = once + kSpWords;
  unsigned long long *tab = reinterpret_cast<unsigned long long *>(twice + kSpWords);
  int2 *s_seg = reinterpret_cast<int2 *>(tab + kSpT + 32);  // (first far end, how many)
  int32_t *s_len = reinterpret_cast<int32_t *>(s_seg + sp_max_seg<C>());
  int32_t *ws = s_len + NT;
  const int32_t tid = (int32_t)threadIdx.x, lane = tid & 31, wq = tid >> 5;
  SpQueue q = {ws + NW + 1 + wq * kSpQ, 0};
  // the survivors' slots, in `once` (not read any more when they are listed),
  // and their keys, in `twice` (the same)
  int32_t *list = reinterpret_cast<int32_t *>(once);
  unsigned long long *keys = reinterpret_cast<unsigned long long *>(twice);
  auto zero = [&](uint32_t *p, int n) {  // words, rounded up to four
    uint4 *p4 = reinterpret_cast<uint4 *>(p);
    for (int i = tid; i < (n + 3) >> 2; i += NT) p4[i] = make_uint4(0, 0, 0, 0);
  };
  zero(once, 2 * kSpWords);
  clear_slots<NT>(tab, kSpT + 32);
  const unsigned nrows = part ? meta->sparse_rest : meta->sparse_huge;
  unsigned *ticket = part ? &meta->sparse_ticket_rest : &meta->sparse_ticket;
  const bool unweighted = a.unweighted != 0;
  const bool emit = a.mode != kCount;
  // pairs of a row of several ranges: at most work / 2 (s >= 2)
  int32_t *pj = buf + (long long)blockIdx.x * buf_stride, *pw = pj + buf_stride / 2;
  if (tid == 0) {
    for (int i = 0; i < 5; ++i) s_cyc[i] = 0;
    s_cyc[5] = clock64();
  }
  auto lap = [&](int i) {
    if (tid == 0) {
      const long long t1 = clock64();
      s_cyc[i] += t1 - s_cyc[5];
      s_cyc[5] = t1;
    }
  };
  for (;;) {
    __syncthreads();  // the previous row is done
    if (tid == 0) {
      const unsigned t = atomicAdd(ticket, 1u);
      *s_row = t >= nrows ? -1 : rows[part ? list_len - 1 - t : t];
      *s_ovf = 0;
      *s_any = 0;
      *s_sum = 0;
      *s_nsurv = 0;
    }
    __syncthreads();
    const int32_t e = *s_row;
    if (e < 0) break;
    const int32_t smin = s_of(a.row_s, a.smin, e);
    const int32_t work = a.row_work[e - a.row_begin];
    const int32_t k0 = w.r_off[e], k1 = w.r_off[e + 1];
    const bool single = k1 - k0 <= NT;  // one batch of tails: the longest are set aside
    const int32_t nset = smin <= 3 ? 1 : min(smin - 2, kSpDrop);
    // the ids of a range: the whole span for rows of up to `chunk` wedges
    const int32_t f_hi = a.row_fhi ? a.row_fhi[e] : R;
    const int32_t chunk = smin <= 3 ? kSpChunk : kSpChunkAside;
    int32_t step = (f_hi - (e + 1)) / ((work + chunk - 1) / chunk) + 1;
    bool multi = work > chunk;  // several ranges: the row's pairs are gathered in scratch
    // (both by the planning: cannot happen)
    bool hand_over = work > C::MAXW || work > buf_stride;
    bool full = false;  // the largest table, after an overflow
    int32_t out = 0;    // pairs of the earlier ranges
    int32_t next = 0, upto = 0;  // single: where the thread's tail goes on
    lap(0);
    for (int32_t Fa = e + 1; Fa < f_hi && !hand_over;) {
      const int32_t Fb = f_hi - Fa > step ? Fa + step : f_hi;
      int lgb = kSpLogB, lgt = C::LGT;
      // The range's tails of incidences [base, base + NT) as segments of at
      // most kSpSeg far ends: s_seg[0, nA) those to insert, s_seg[nA, nA + nD)
      // those of the tails set aside.
      int32_t nA = 0, nD = 0;
      auto load_batch = [&](int32_t base) {
        const int32_t k = base + tid;
        int32_t b = 0, len = 0;
        if (k < k1) {
          b = __ldg(w.tail_beg + k);
          int32_t end = __ldg(w.tail_end + k);
          if (multi) {
            // (one batch: the last range's end is kept)
            if (Fa > e + 1) b = single ? next : lower_pos(w.c_idx_s, b, end, Fa);
            if (Fb < f_hi) end = lower_pos(w.c_idx_s, b, end, Fb);
            upto = end;
          }
          len = end - b;
        }
        bool aside = false;
        if (single) {
          // a tail's rank by length (ties: the earlier one first)
          s_len[tid] = len;
          __syncthreads();
          if (len > 0) {
            int32_t r = 0;
            const int32_t n = k1 - k0;
            for (int32_t j = 0; j < n; ++j) {
              const int32_t x = s_len[j];
              r += x > len || (x == len && j < tid);
            }
            aside = r < nset;
          }
          const int32_t sum = __reduce_add_sync(0xffffffffu, aside ? 0 : len);
          if (lane == 0 && sum) atomicAdd(s_sum, sum);
        }
        const int32_t n = (len + kSpSeg - 1) / kSpSeg;
        const int32_t packed = aside ? n << 16 : n;
        int32_t total;
        const int32_t pos = block_inclusive_scan<NT>(packed, ws, &total) - packed;
        nA = total & 0xFFFF;
        nD = total >> 16;
        int2 *dst = s_seg + (aside ? nA + (pos >> 16) : pos & 0xFFFF);
        for (int32_t i = 0; i < n; ++i)
          dst[i] = make_int2(b + i * kSpSeg, min(kSpSeg, len - i * kSpSeg));
        __syncthreads();
      };
      // step(f, last) for every segment of s_seg[x0, x1): a warp each
      auto for_segments = [&](int32_t x0, int32_t x1, auto &&step) {
        for (int32_t x = x0 + wq; x < x1; x += NW) {
          const int2 sg = s_seg[x];
          int32_t f[kSpG];
#pragma unroll
          for (int g = 0; g < kSpG; ++g)
            f[g] = 32 * g + lane < sg.y ? __ldg(w.c_idx_s + sg.x + 32 * g + lane) : -1;
          step(f, x + NW >= x1);
        }
      };
      auto count = [&](int32_t x) {
        sp_insert(tab, x, smin, unweighted, lgt, s_ovf, list, kSpList, s_nsurv);
      };
      // 1. the inserted tails
      bool hit = false;
      for (int32_t base = k0; base < k1; base += NT) {
        if (base > k0) __syncthreads();  // the previous batch's segments are read
        load_batch(base);
        if (base == k0) {
          // a filter of >= 32 bits per inserted wedge (a single-wedge far end
          // finds its bit set by another with probability below 1/64), and a
          // table of half a slot per inserted wedge, within the maxima
          const int32_t ins = single ? *s_sum : min(work, 2 * chunk);
          lgb = min(max(ceil_log2(ins > 1 ? ins : 2) + 5, 12), kSpLogB);
          if (!full) lgt = min(max(ceil_log2(ins / 2 + 1), 8), C::LGT);
        }
        for_segments(0, nA, [&](const int32_t(&f)[kSpG], bool) {
          uint32_t old[kSpG], h[kSpG];
#pragma unroll
          for (int g = 0; g < kSpG; ++g) {
            h[g] = sp_bit(f[g], lgb);
            old[g] = f[g] >= 0 ? atomicOr(once + (h[g] >> 5), 1u << (h[g] & 31)) : 0u;
          }
#pragma unroll
          for (int g = 0; g < kSpG; ++g)
            if ((old[g] >> (h[g] & 31)) & 1u) {
              atomicOr(twice + (h[g] >> 5), 1u << (h[g] & 31));
              hit = true;
            }
        });
      }
      if (hit) *s_any = 1;
      __syncthreads();  // both filters as far as the inserted tails go
      // 2. one tail set aside (s <= 3)
      if (smin <= 3 && nA > 0 && nD > 0) {  // uniform
        bool in = false;
        for_segments(nA, nA + nD, [&](const int32_t(&f)[kSpG], bool last) {
#pragma unroll
          for (int g = 0; g < kSpG; ++g) {
            const uint32_t h = sp_bit(f[g], lgb);
            const bool c = f[g] >= 0 && ((once[h >> 5] >> (h & 31)) & 1u);
            if (c) {
              atomicOr(twice + (h >> 5), 1u << (h & 31));
              in = true;
            }
            q.push(c, f[g]);
          }
          q.drain(last, [&](int32_t x) {
            // (nothing is listed here: a first wedge, and s >= 2)
            sp_insert(tab, x, 0x7fffffff, unweighted, lgt, s_ovf, list, kSpList, s_nsurv);
          });
        });
        if (in) *s_any = 1;
        __syncthreads();  // `twice` is final, `once` is not read any more
      }
      lap(1);
      const int32_t T = 1 << lgt;
      int32_t n = 0, dirty_once = 1 << (lgb - 5), dirty_twice = dirty_once;
      bool redo = false;
      if (*s_any) {  // uniform: else no far end has two wedges
        // 3. counts
        for (int32_t base = k0; base < k1; base += NT) {
          if (!single) {
            if (base > k0) __syncthreads();
            load_batch(base);
          }
          for_segments(0, smin > 3 ? nA + nD : nA, [&](const int32_t(&f)[kSpG], bool last) {
            uint32_t word[kSpG], h[kSpG];
#pragma unroll
            for (int g = 0; g < kSpG; ++g) {  // loads in flight together
              h[g] = sp_bit(f[g], lgb);
              word[g] = f[g] >= 0 ? twice[h[g] >> 5] : 0u;
            }
#pragma unroll
            for (int g = 0; g < kSpG; ++g) q.push((word[g] >> (h[g] & 31)) & 1u, f[g]);
            q.drain(last, count);
          });
        }
        __syncthreads();  // counts and survivors final
        lap(2);
        n = *s_nsurv;
        dirty_once = max(dirty_once, min(n, kSpList));  // the list
        // 4. survivors in ascending f.  Those that fit are ranked in `twice`
        // while the table is cleared; more of them are ordered in the table.
        const bool small = n <= kSpSortMax;
        if (*s_ovf || (emit && !small && (n > NT * kSpRegQ || n > kSpList))) {
          redo = true;
        } else if (emit && n > 0) {
          long long base = -1;
          if (!multi && tid == 0) *s_base = reserve(a, e, n, kBinSparse);
          auto write = [&](int32_t i, unsigned long long x) {
            const int32_t f = (int32_t)(x >> 32), c = (int32_t)(uint32_t)x;
            if (multi) {
              pj[out + i] = f;
              if (!unweighted) pw[out + i] = c;
            } else if (base >= 0) {
              put(a, base, i, e, f, c);
            }
          };
          if (small) {
            dirty_twice = max(dirty_twice, 2 * ((n + 31) & ~31));
            for (int32_t i = tid; i < n; i += NT)
              keys[i] = tab[list[i]] + 1ull;  // the count word holds count - 1
            __syncthreads();  // keys and base in place, the table is read
            base = *s_base;
            clear_slots<NT>(tab, T);
            rank_keys<NT>(keys, n, write);
          } else {
            unsigned long long x[kSpRegQ];
#pragma unroll
            for (int i = 0; i < kSpRegQ; ++i)
              x[i] = tid + i * NT < n ? tab[list[tid + i * NT]] + 1ull : 0ull;
            __syncthreads();  // keys read, base in place
            base = *s_base;
            clear_slots<NT>(tab, T);
            __syncthreads();
#pragma unroll
            for (int i = 0; i < kSpRegQ; ++i)
              if (tid + i * NT < n) tab[tid + i * NT] = x[i];
            __syncthreads();
            int32_t used = 0;
            const int32_t at = sort_survivors<NT, true>(tab, n, &used);
            for (int32_t i = tid; i < n; i += NT) write(i, tab[at + i]);
            __syncthreads();  // the sorted keys are written
            clear_slots<NT>(tab, used);
          }
        } else {
          if (!multi && tid == 0) reserve(a, e, n, kBinSparse);
          clear_slots<NT>(tab, T);
        }
      } else {
        lap(2);
      }
      __syncthreads();  // every shared value of the range is read
      lap(3);
      if (redo) {
        const bool over = *s_ovf != 0;
        __syncthreads();  // s_ovf is read
        if (over && lgt < C::LGT) {
          full = true;
        } else {  // half the ids at a time
          multi = true;
          hand_over = step <= 64;
          step = (step + 1) / 2;
        }
        clear_slots<NT>(tab, T);
      } else {
        out += n;
        next = upto;
        Fa = Fb;
        full = false;
      }
      zero(once, dirty_once);
      zero(twice, dirty_twice);
      if (tid == 0) {
        *s_ovf = 0;
        *s_any = 0;
        *s_sum = 0;
        *s_nsurv = 0;
      }
      __syncthreads();
      lap(4);
    }
    if (hand_over) {
      // to the giant bin (launched after this kernel)
      if (tid == 0) {
        const unsigned pos = atomicAdd(&meta->giant_rest, 1u);
        giant_rows[list_len - 1 - pos] = e;
        atomicAdd(&meta->rows_bin[kBinGiant], 1ull);
      }
    } else if (multi) {
      if (tid == 0) *s_base = reserve(a, e, out, kBinSparse);
      __syncthreads();
      const long long base = *s_base;
      if (emit && base >= 0)
        for (int32_t i = tid; i < out; i += NT)
          put(a, base, i, e, pj[i], unweighted ? 0 : pw[i]);
    }
    lap(4);
  }
  if (tid == 0)
    for (int i = 0; i < 5; ++i) atomicAdd(&meta->sparse_cycles[i], (unsigned long long)s_cyc[i]);
}

// ------------------------------------------------------------ short tails --
//
// The flat bin: rows with s >= 2 of 1,025 to 16,384 wedges whose tails are short or
// alike (short_tails: web-shaped and uniform inputs).  A warp per tail, as in the
// sparse bin, leaves most of its lanes idle there (58 to 190 instead of 10 to 15 CTA
// cycles per wedge), and no tail is long enough to be worth setting aside.  The
// row's wedges are flattened: wedge i's tail is found by a search over
// the tails' prefix sums, each warp loads kSpSeg consecutive wedges per step and
// copies their far ends to the CTA's scratch, so that the second pass reads them
// in order.  Filters, table and survivors are the sparse bin's; a row that
// overflows the table or has more survivors than are ordered here goes to the
// giant bin.  (Its own kernel: with this path beside the other in k_walk_sparse the
// step of chung_lu_1m, which has few such rows, took 107.4 instead of 105.4 ms.)
//
// 100K rows of 250 of 1.9M vertices, L_2, whole counting pass: 6.8 -> 2.6 ms; 200K
// rows of 400 of 9M 19.7 -> 8.7; 4M x 10M lognormal hyperedges with the tile path,
// L_2, L_8, L_32, per build 23.3, 23.9, 22.5 -> 19.1, 18.0, 16.7.  Mean tails of
// up to 8, 16, 32: 5.0, 2.7, 2.7 ms and (100K rows of 100 of 300K) 2.9, 2.6, 1.7.

// The two instances of the kernel, for rows of up to kSparseBigWork wedges and more.
// (The smaller table alone: 92K rows of the 400K x 1,500 handed over, 87.7 -> 102.7
// ms a pass; the larger alone 9.5 instead of 9.1 on 200K x 400.)
struct FlSmall {
  static constexpr int NT = 256, LGT = 11, MINB = 5;
};
struct FlBig {  // (256 threads, four CTAs: 26.2 instead of 22.3 ms on 400K rows of 1,500)
  static constexpr int NT = 512, LGT = 12, MINB = 3;
};

// [s_base 8][s_ovf 4][s_row 4][s_any 4][s_nsurv 4][pad 8][s_cyc 6 x 8][once][twice][table x 8]
// [tail places NT][prefix sums NT][ws NT/32+1][queues]
template <class C>
constexpr size_t flat_smem() {
  return 80 + (size_t)kSpWords * 8 + (size_t)(1 << C::LGT) * 8 +
         (size_t)(2 * C::NT + C::NT / 32 + 1 + C::NT / 32 * kSpQ) * 4;
}

// part 0: the rows above kSparseBigWork wedges (the front of the list), 1: the
// others (its back).  buf: the CTA's share of the bin's scratch, at least the
// largest row's work.
template <class C>
__global__ __launch_bounds__(C::NT, C::MINB) void k_walk_flat(
    Walk w, const int32_t *__restrict__ rows, EmitArgs a, int32_t *__restrict__ giant_rows,
    int32_t list_len, int32_t *__restrict__ buf, long long buf_stride, int part) {
  constexpr int NT = C::NT, NW = NT / 32, T_MAX = 1 << C::LGT;
  Meta *meta = a.meta;
  if (meta->err) return;
  extern __shared__ __align__(16) unsigned char smem[];
  long long *s_base = reinterpret_cast<long long *>(smem);
  int32_t *s_ovf = reinterpret_cast<int32_t *>(smem + 8);
  int32_t *s_row = reinterpret_cast<int32_t *>(smem + 12);
  int32_t *s_any = reinterpret_cast<int32_t *>(smem + 16);
  int32_t *s_nsurv = reinterpret_cast<int32_t *>(smem + 20);
  long long *s_cyc = reinterpret_cast<long long *>(smem + 32);  // as in the sparse bin
  uint32_t *once = reinterpret_cast<uint32_t *>(smem + 80);
  uint32_t *twice = once + kSpWords;
  unsigned long long *tab = reinterpret_cast<unsigned long long *>(twice + kSpWords);
  int32_t *s_beg = reinterpret_cast<int32_t *>(tab + T_MAX);
  int32_t *s_pref = s_beg + NT;
  int32_t *ws = s_pref + NT;
  const int32_t tid = (int32_t)threadIdx.x, lane = tid & 31, wq = tid >> 5;
  SpQueue q = {ws + NW + 1 + wq * kSpQ, 0};
  int32_t *list = reinterpret_cast<int32_t *>(once);  // survivors' slots, then their keys
  unsigned long long *keys = reinterpret_cast<unsigned long long *>(twice);
  auto zero = [&](uint32_t *p, int n) {  // words, rounded up to four
    uint4 *p4 = reinterpret_cast<uint4 *>(p);
    for (int i = tid; i < (n + 3) >> 2; i += NT) p4[i] = make_uint4(0, 0, 0, 0);
  };
  zero(once, 2 * kSpWords);
  clear_slots<NT>(tab, T_MAX);
  const unsigned nrows = part ? meta->flat_rest : meta->flat_huge;
  unsigned *ticket = part ? &meta->flat_ticket_rest : &meta->flat_ticket;
  const bool unweighted = a.unweighted != 0;
  const bool emit = a.mode != kCount;
  int32_t *copy = buf + (long long)blockIdx.x * buf_stride;
  if (tid == 0) {
    for (int i = 0; i < 5; ++i) s_cyc[i] = 0;
    s_cyc[5] = clock64();
  }
  auto lap = [&](int i) {
    if (tid == 0) {
      const long long t1 = clock64();
      s_cyc[i] += t1 - s_cyc[5];
      s_cyc[5] = t1;
    }
  };
  for (;;) {
    __syncthreads();  // the previous row is done
    if (tid == 0) {
      const unsigned t = atomicAdd(ticket, 1u);
      *s_row = t >= nrows ? -1 : rows[part ? list_len - 1 - t : t];
      *s_ovf = 0;
      *s_any = 0;
      *s_nsurv = 0;
    }
    __syncthreads();
    const int32_t e = *s_row;
    if (e < 0) break;
    const int32_t smin = s_of(a.row_s, a.smin, e);
    const int32_t work = a.row_work[e - a.row_begin];
    const int32_t k0 = w.r_off[e], k1 = w.r_off[e + 1];
    // (by the planning: cannot happen)
    bool hand_over = work > kFlatMaxWork || work > buf_stride;
    const int lgb = min(max(ceil_log2(work) + 5, 12), kSpLogB);  // as in the sparse bin
    const int lgt = min(max(ceil_log2(work / 2 + 1), 8), C::LGT);
    lap(0);
    // 1. both filters, and the copy
    bool hit = false;
    int32_t done = 0;
    for (int32_t base = k0; base < k1 && !hand_over; base += NT) {
      if (base > k0) __syncthreads();  // the previous batch is read
      const int32_t k = base + tid;
      int32_t b = 0, len = 0, total;
      if (k < k1) {
        b = __ldg(w.tail_beg + k);
        len = __ldg(w.tail_end + k) - b;
      }
      const int32_t inc = block_inclusive_scan<NT>(len, ws, &total);
      s_beg[tid] = b - (inc - len);  // + i: wedge i's place
      s_pref[tid] = inc;             // wedges up to this tail
      __syncthreads();
      for (int32_t c0 = wq * kSpSeg; c0 < total; c0 += NW * kSpSeg) {
        int32_t j = 0, hi = NT - 1;  // the first tail with s_pref > c0
        while (j < hi) {
          const int32_t mid = (j + hi) >> 1;
          if (s_pref[mid] > c0) hi = mid;
          else j = mid + 1;
        }
        int32_t f[kSpG];
        uint32_t old[kSpG], h[kSpG];
#pragma unroll
        for (int g = 0; g < kSpG; ++g) {
          const int32_t i = c0 + 32 * g + lane;
          f[g] = -1;
          if (i < total) {
            while (s_pref[j] <= i) ++j;
            f[g] = s_beg[j] + i;
          }
        }
#pragma unroll
        for (int g = 0; g < kSpG; ++g) f[g] = f[g] >= 0 ? __ldg(w.c_idx_s + f[g]) : -1;
#pragma unroll
        for (int g = 0; g < kSpG; ++g) {
          h[g] = sp_bit(f[g], lgb);
          old[g] = 0;
          if (f[g] >= 0) {
            copy[done + c0 + 32 * g + lane] = f[g];
            old[g] = atomicOr(once + (h[g] >> 5), 1u << (h[g] & 31));
          }
        }
#pragma unroll
        for (int g = 0; g < kSpG; ++g)
          if ((old[g] >> (h[g] & 31)) & 1u) {
            atomicOr(twice + (h[g] >> 5), 1u << (h[g] & 31));
            hit = true;
          }
      }
      done += total;
    }
    if (hit) *s_any = 1;
    __syncthreads();  // filters and copy complete
    lap(1);
    const int32_t T = 1 << lgt;
    int32_t dirty_once = 1 << (lgb - 5), dirty_twice = dirty_once;
    if (*s_any) {  // uniform: else no far end has two wedges
      // 2. counts
      for (int32_t c0 = wq * kSpSeg; c0 < work; c0 += NW * kSpSeg) {
        int32_t f[kSpG];
        uint32_t word[kSpG], h[kSpG];
#pragma unroll
        for (int g = 0; g < kSpG; ++g)
          f[g] = c0 + 32 * g + lane < work ? copy[c0 + 32 * g + lane] : -1;
#pragma unroll
        for (int g = 0; g < kSpG; ++g) {
          h[g] = sp_bit(f[g], lgb);
          word[g] = f[g] >= 0 ? twice[h[g] >> 5] : 0u;
        }
#pragma unroll
        for (int g = 0; g < kSpG; ++g) q.push((word[g] >> (h[g] & 31)) & 1u, f[g]);
        q.drain(c0 + NW * kSpSeg >= work, [&](int32_t x) {
          sp_insert(tab, x, smin, unweighted, lgt, s_ovf, list, kSpList, s_nsurv);
        });
      }
      __syncthreads();  // counts and survivors final
      lap(2);
      // 3. survivors in ascending f, ranked in `twice` while the table is cleared
      const int32_t n = *s_nsurv;
      dirty_once = max(dirty_once, min(n, kSpList));  // the list
      if (*s_ovf || (emit && n > kSpSortMax)) {
        hand_over = true;
        clear_slots<NT>(tab, T);
      } else if (emit && n > 0) {
        if (tid == 0) *s_base = reserve(a, e, n, kBinFlat);
        dirty_twice = max(dirty_twice, 2 * ((n + 31) & ~31));
        for (int32_t i = tid; i < n; i += NT)
          keys[i] = tab[list[i]] + 1ull;  // the count word holds count - 1
        __syncthreads();  // keys and base in place, the table is read
        const long long base = *s_base;
        clear_slots<NT>(tab, T);
        rank_keys<NT>(keys, n, [&](int32_t i, unsigned long long x) {
          if (base >= 0) put(a, base, i, e, (int32_t)(x >> 32), (int32_t)(uint32_t)x);
        });
      } else {
        if (tid == 0) reserve(a, e, n, kBinFlat);
        clear_slots<NT>(tab, T);
      }
    }
    lap(3);
    __syncthreads();  // keys and list are read
    zero(once, dirty_once);
    zero(twice, dirty_twice);
    if (hand_over && tid == 0) {  // to the giant bin (launched after this kernel)
      const unsigned pos = atomicAdd(&meta->giant_rest, 1u);
      giant_rows[list_len - 1 - pos] = e;
      atomicAdd(&meta->rows_bin[kBinGiant], 1ull);
    }
    lap(4);
  }
  if (tid == 0)
    for (int i = 0; i < 5; ++i) atomicAdd(&meta->sparse_cycles[i], (unsigned long long)s_cyc[i]);
}

// ------------------------------------------------------------- short rows --
//
// Rows of at most kCtaSMaxWork wedges with s >= 2, a warp each: 4 KB of shared
// memory per warp (two filters of 2^13 bits, a table of 256 slots), up to 32
// tails at a time with the longest set aside, wedges found by a search over
// the tails' prefix sums in registers.  A row that overflows the table goes to
// the giant bin.  Rows of up to 1,536 or 2,048 wedges here: chung_lu_1m step
// 105.7 -> 104.0, 106.2 ms, but host builds of 200K x 400K 4.13 -> 4.34, 4.71.
// (The sort of a warp's wedge ends and the CTA-wide hash table
// that these rows took before cost 11 and 4 to 5 SM cycles per wedge:
// L_3 of 500K x 1M, these rows 1,755 -> 566 us.)

constexpr int kRwNT = 256;
constexpr int kRwNW = kRwNT / 32;
constexpr int kRwLogB = 13;
constexpr int kRwWords = 1 << (kRwLogB - 5);
constexpr int kRwLgT = 8;
constexpr int kRwT = 1 << kRwLgT;
#ifndef SLG_RW_MINB
#define SLG_RW_MINB 6
#endif

struct RwShared {
  uint32_t once[kRwWords];      // then the survivors' slots
  uint32_t twice[kRwWords];
  unsigned long long tab[kRwT];
};

__global__ __launch_bounds__(kRwNT, SLG_RW_MINB) void k_walk_rows(
    Walk w, const int32_t *__restrict__ rows, EmitArgs a, int32_t *__restrict__ giant_rows,
    int32_t list_len) {
  Meta *meta = a.meta;
  if (meta->err) return;
  extern __shared__ __align__(16) unsigned char smem[];
  const int lane = threadIdx.x & 31, wq = threadIdx.x >> 5;
  RwShared &sh = reinterpret_cast<RwShared *>(smem)[wq];
  int32_t *s_flag = reinterpret_cast<int32_t *>(smem + kRwNW * sizeof(RwShared)) + 2 * wq;
  int32_t *s_ovf = s_flag, *s_nsurv = s_flag + 1;
  int32_t *list = reinterpret_cast<int32_t *>(sh.once);
  auto clear = [&](bool table) {
    uint4 *f4 = reinterpret_cast<uint4 *>(sh.once);
    for (int i = lane; i < kRwWords / 2; i += 32) f4[i] = make_uint4(0, 0, 0, 0);  // both filters
    if (table) {
      ulonglong2 *t2 = reinterpret_cast<ulonglong2 *>(sh.tab);
      for (int i = lane; i < kRwT / 2; i += 32) t2[i] = make_ulonglong2(kEmpty64, kEmpty64);
    }
    if (lane < 2) s_flag[lane] = 0;
    __syncwarp();
  };
  clear(true);
  const bool unweighted = a.unweighted != 0;
  const bool emit = a.mode != kCount;
  const int64_t nrows = (int64_t)meta->rows_bin[kBinRows];
  const int64_t nw = (int64_t)gridDim.x * kRwNW;
  for (int64_t r = (int64_t)blockIdx.x * kRwNW + wq; r < nrows; r += nw) {
    const int32_t e = rows[r];
    const int32_t smin = s_of(a.row_s, a.smin, e);
    const int32_t k0 = w.r_off[e], k1 = w.r_off[e + 1];
    const bool single = k1 - k0 <= 32;
    const int nset = smin <= 3 ? 1 : min(smin - 2, kSpDrop);
    int32_t b = 0, len = 0, inc = 0, total = 0;
    unsigned aside = 0;  // lanes whose tail is set aside
    auto load = [&](int32_t base) {
      const int32_t k = base + lane;
      b = len = 0;
      if (k < k1) {
        b = __ldg(w.tail_beg + k);
        len = __ldg(w.tail_end + k) - b;
      }
      bool mine = false;
      if (single) {
        uint32_t key = len > 0 ? ((uint32_t)len << 5) | (31 - lane) : 0u;
        for (int t = 0; t < nset; ++t) {
          const uint32_t m = __reduce_max_sync(0xffffffffu, key);
          if (m == 0) break;
          if (key == m) {
            mine = true;
            key = 0;
          }
        }
        aside = __ballot_sync(0xffffffffu, mine);
      }
      inc = warp_inclusive_scan(mine ? 0 : len);
      total = __shfl_sync(0xffffffffu, inc, 31);
    };
    // fn(f) for the batch's wedges outside the tails set aside (f < 0: none);
    // two steps of 32 wedges in flight
    auto for_wedges = [&](auto &&fn) {
      const int32_t before = b - (inc - (((aside >> lane) & 1u) ? 0 : len));  // + i: wedge i's place
      for (int32_t i0 = 0; i0 < total; i0 += 64) {
        int32_t f[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const int32_t i = i0 + 32 * u + lane;
          int j = 0;
#pragma unroll
          for (int step = 16; step > 0; step >>= 1)
            if (__shfl_sync(0xffffffffu, inc, j + step - 1) <= i) j += step;
          const int32_t at = __shfl_sync(0xffffffffu, before, j) + i;
          f[u] = i < total ? __ldg(w.c_idx_s + at) : -1;
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) fn(f[u]);
      }
    };
    auto for_aside = [&](auto &&fn) {
      for (unsigned m = aside; m; m &= m - 1) {
        const int src = __ffs(m) - 1;
        const int32_t b0 = __shfl_sync(0xffffffffu, b, src), n = __shfl_sync(0xffffffffu, len, src);
        for (int32_t i0 = 0; i0 < n; i0 += 64) {
          int32_t f[2];
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            const int32_t i = i0 + 32 * u + lane;
            f[u] = i < n ? __ldg(w.c_idx_s + b0 + i) : -1;
          }
#pragma unroll
          for (int u = 0; u < 2; ++u) fn(f[u]);
        }
      }
    };
    auto insert = [&](int32_t f, int32_t s) {
      sp_insert(sh.tab, f, s, unweighted, kRwLgT, s_ovf, list, kRwWords, s_nsurv);
    };
    // 1. the inserted tails
    bool hit = false;
    for (int32_t base = k0; base < k1; base += 32) {
      load(base);
      for_wedges([&](int32_t f) {
        if (f < 0) return;
        const uint32_t h = sp_bit(f, kRwLogB), m = 1u << (h & 31);
        if (atomicOr(sh.once + (h >> 5), m) & m) {
          atomicOr(sh.twice + (h >> 5), m);
          hit = true;
        }
      });
    }
    __syncwarp();
    // 2. one tail set aside (s <= 3)
    if (smin <= 3 && total > 0)
      for_aside([&](int32_t f) {
        if (f < 0) return;
        const uint32_t h = sp_bit(f, kRwLogB), m = 1u << (h & 31);
        if (sh.once[h >> 5] & m) {
          atomicOr(sh.twice + (h >> 5), m);
          hit = true;
          insert(f, 0x7fffffff);
        }
      });
    __syncwarp();
    if (!__any_sync(0xffffffffu, hit)) {  // no far end with two wedges
      clear(false);
      continue;
    }
    // 3. counts
    auto count = [&](int32_t f) {
      if (f < 0) return;
      const uint32_t h = sp_bit(f, kRwLogB);
      if ((sh.twice[h >> 5] >> (h & 31)) & 1u) insert(f, smin);
    };
    for (int32_t base = k0; base < k1; base += 32) {
      if (!single) load(base);
      for_wedges(count);
    }
    if (smin > 3) for_aside(count);
    __syncwarp();
    // 4. survivors in ascending f
    const int32_t n = *s_nsurv;
    if (*s_ovf || (emit && n > kRwWords)) {
      if (lane == 0) {  // to the giant bin (launched after this kernel)
        const unsigned pos = atomicAdd(&meta->giant_rest, 1u);
        giant_rows[list_len - 1 - pos] = e;
        atomicAdd(&meta->rows_bin[kBinGiant], 1ull);
      }
    } else if (n > 0) {
      long long base = -1;
      if (lane == 0) base = reserve(a, e, n, kBinRows);
      base = __shfl_sync(0xffffffffu, base, 0);
      if (emit && base >= 0) {
        if (n <= 32) {
          const unsigned long long x = lane < n ? sh.tab[list[lane]] + 1ull : ~0ull;
          int32_t rank = 0;
          for (int j = 0; j < n; ++j) rank += __shfl_sync(0xffffffffu, x, j) < x;
          if (lane < n) put(a, base, rank, e, (int32_t)(x >> 32), (int32_t)(uint32_t)x);
        } else {
          for (int32_t i = lane; i < n; i += 32) {
            const unsigned long long x = sh.tab[list[i]] + 1ull;
            int32_t rank = 0;
            for (int32_t j = 0; j < n; ++j) rank += sh.tab[list[j]] + 1ull < x;
            put(a, base, rank, e, (int32_t)(x >> 32), (int32_t)(uint32_t)x);
          }
        }
      }
    }
    __syncwarp();
    clear(true);
  }
}

// The flat bin's rows behind the sparse bin's, at both ends of its list.
__global__ __launch_bounds__(256) void k_join_flat(const int32_t *__restrict__ flat,
                                                   int32_t *__restrict__ sparse,
                                                   int32_t list_len, unsigned flat_huge,
                                                   unsigned flat_rest, unsigned huge,
                                                   unsigned rest, Meta *meta) {
  const unsigned t = blockIdx.x * 256 + threadIdx.x;
  if (t < flat_huge) sparse[huge + t] = flat[t];
  if (t < flat_rest) sparse[list_len - 1 - (rest + t)] = flat[list_len - 1 - t];
  if (t == 0) {
    meta->sparse_huge = huge + flat_huge;
    meta->sparse_rest = rest + flat_rest;
  }
}

constexpr size_t rows_smem() { return kRwNW * (sizeof(RwShared) + 8); }

struct SpOcc {
  int small = 0, big = 0;  // CTAs
  int rows = 0;            // CTAs of k_walk_rows
  int flat_small = 0, flat_big = 0;
  int dev = -1;
};

template <class C>
int sp_ctas(int sms) {
  int nb = 0;
  cudaFuncSetAttribute(k_walk_sparse<C>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       (int)sparse_smem<C>());
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_walk_sparse<C>, C::NT, sparse_smem<C>());
  return sms * std::max(nb, 1);
}

template <class C>
int fl_ctas(int sms) {
  int nb = 0;
  cudaFuncSetAttribute(k_walk_flat<C>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       (int)flat_smem<C>());
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_walk_flat<C>, C::NT, flat_smem<C>());
  return sms * std::max(nb, 1);
}

SpOcc &sp_occ() {
  static SpOcc occ[64];
  static std::mutex mu;
  int dev = 0;
  cudaGetDevice(&dev);
  SpOcc &o = occ[dev & 63];
  std::lock_guard<std::mutex> lock(mu);
  if (o.dev != dev) {
    int sms = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    o.small = sp_ctas<SpSmall>(sms);
    o.big = sp_ctas<SpBig>(sms);
    int nb = 0;
    cudaFuncSetAttribute(k_walk_rows, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)rows_smem());
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_walk_rows, kRwNT, rows_smem());
    o.rows = sms * std::max(nb, 1);
    o.flat_small = fl_ctas<FlSmall>(sms);
    o.flat_big = fl_ctas<FlBig>(sms);
    o.dev = dev;
  }
  return o;
}

template <class C>
void fl_launch(const WalkLaunch &L, int ctas, int part, cudaStream_t st) {
  const int64_t stride = L.rows;
  k_walk_flat<C><<<ctas, C::NT, flat_smem<C>(), st>>>(
      L.w, L.bin_rows + (int64_t)kBinFlat * stride, L.a,
      const_cast<int32_t *>(L.bin_rows) + (int64_t)kBinGiant * stride, (int32_t)stride,
      L.sparse_scratch, (L.sparse_ints / (long long)ctas) & ~31ll, part);
}

template <class C>
void sp_launch(const WalkLaunch &L, int ctas, int part, cudaStream_t st) {
  const int64_t stride = L.rows;
  k_walk_sparse<C><<<ctas, C::NT, sparse_smem<C>(), st>>>(
      L.w, L.bin_rows + (int64_t)kBinSparse * stride, L.a,
      const_cast<int32_t *>(L.bin_rows) + (int64_t)kBinGiant * stride, (int32_t)stride,
      L.sparse_scratch, (L.sparse_ints / (long long)ctas) & ~31ll, L.R, part);
}

}  // namespace

// Scratch ints for rows of up to `max_work` wedges.
long long sparse_ints(int32_t max_work) {
  SpOcc &o = sp_occ();
  return std::max({(long long)std::max(o.small, o.flat_small) *
                       (std::min(max_work, kSparseBigWork) + 128ll),
                   (long long)o.flat_big * (std::min(max_work, kFlatMaxWork) + 128ll),
                   (long long)o.big * (max_work + 128ll)});
}

// Gives the flat bin's rows to the sparse bin (m: the planning's totals).
cudaError_t launch_join_flat(int32_t *bin_rows, int32_t rows, const Meta &m, Meta *meta,
                             cudaStream_t st) {
  const unsigned n = std::max(m.flat_huge, m.flat_rest);
  if (n == 0) return cudaSuccess;
  k_join_flat<<<(n + 255) / 256, 256, 0, st>>>(
      bin_rows + (int64_t)kBinFlat * rows, bin_rows + (int64_t)kBinSparse * rows, rows, m.flat_huge,
      m.flat_rest, m.sparse_huge, m.sparse_rest, meta);
  return cudaGetLastError();
}

cudaError_t launch_walk_rows(const WalkLaunch &L, cudaStream_t st) {
  const int64_t stride = L.rows;
  k_walk_rows<<<sp_occ().rows, kRwNT, rows_smem(), st>>>(
      L.w, L.bin_rows + (int64_t)kBinRows * stride, L.a,
      const_cast<int32_t *>(L.bin_rows) + (int64_t)kBinGiant * stride, (int32_t)stride);
  return cudaGetLastError();
}

cudaError_t launch_walk_sparse(const WalkLaunch &L, cudaStream_t st, int32_t *launches) {
  if (!L.sparse_scratch) return cudaSuccess;  // no row in the bin
  SpOcc &o = sp_occ();
  if (!(L.skip & kSkipSparseBig)) {
    sp_launch<SpBig>(L, o.big, 0, st);
    ++*launches;
  }
  if (!(L.skip & kSkipSparseSmall)) {
    sp_launch<SpSmall>(L, o.small, 1, st);
    ++*launches;
  }
  if (!(L.skip & kSkipFlatBig)) {
    fl_launch<FlBig>(L, o.flat_big, 0, st);
    ++*launches;
  }
  if (!(L.skip & kSkipFlatSmall)) {
    fl_launch<FlSmall>(L, o.flat_small, 1, st);
    ++*launches;
  }
  return cudaGetLastError();
}

}  // namespace slg
