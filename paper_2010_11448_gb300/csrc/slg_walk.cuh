// Device helpers shared by the walk kernels (slg_walk.cu, slg_dense.cu,
// slg_sparse.cu, slg_small.cu).
#pragma once

#include "slg_internal.cuh"

namespace slg {

// Reserve the output slots of one row; returns the base (or -1: no room).
__device__ __forceinline__ long long reserve(const EmitArgs &a, int32_t e, int32_t n, int bin) {
  const int32_t r = e - a.row_begin;
  a.n_e[r] = n;
  if (n) atomicAdd(&a.meta->pairs_bin[bin], (unsigned long long)n);
  if (a.mode == kCount) return -1;
  if (a.mode == kDirect) return a.row_ptr[r];
  if (n == 0) return -1;
  long long base = (long long)atomicAdd(&a.meta->stage_cursor, (unsigned long long)n);
  if (base + n > a.stage_cap) {
    atomicAdd(&a.meta->stage_overflow, 1ull);
    base = -1;
  }
  a.stage_pos[r] = base;
  return base;
}

__device__ __forceinline__ void put(const EmitArgs &a, long long base, int32_t t, int32_t e,
                                    int32_t f, int32_t c) {
  if (a.mode == kDirect) {
    if (a.out_i) a.out_i[base + t] = e;  // null: compressed row form, i implied
    a.out_j[base + t] = f;
    if (!a.unweighted) a.out_w[base + t] = c;
  } else {
    a.stage_j[base + t] = f;
    if (!a.unweighted) a.stage_w[base + t] = c;
  }
}

__device__ __forceinline__ int ceil_log2(int32_t x) {
  return x <= 1 ? 0 : 32 - __clz(x - 1);
}

// Drops from L2, without writing them back to DRAM, the 128-byte lines that
// lie wholly inside [p, p + n) (PTX discard.global.L2): for per-CTA scratch
// whose contents are dead.  Every reader of the range must have passed a
// block barrier since its last read; lines that the range shares with
// neighbouring data at its two ends are left alone.
__device__ __forceinline__ void l2_discard(const int32_t *p, long long n) {
  if (n <= 0) return;
  const unsigned long long g = (unsigned long long)__cvta_generic_to_global(p);
  const unsigned long long b = (g + 127ull) & ~127ull;
  const unsigned long long e = (g + 4ull * (unsigned long long)n) & ~127ull;
  for (unsigned long long x = b + 128ull * threadIdx.x; x < e; x += 128ull * blockDim.x)
    asm volatile("discard.global.L2 [%0], 128;" ::"l"(x) : "memory");
}

// Survivors per word of the bits from which for_survivors works by words.
constexpr int32_t kSurvDense = 4;

// fn(t, o) for every set bit o of map[m0, m1) in ascending o, t counting from
// `start`, where each thread owns consecutive words and `start` is its first
// place; clears the words.  `dense` (uniform): the bits are many, so a warp
// takes its threads' words one by one, a lane per bit (consecutive places are
// then written by consecutive lanes); else each thread takes its own.
template <class Fn>
__device__ __forceinline__ void for_survivors(uint32_t *map, int32_t m0, int32_t m1, int32_t start,
                                              bool dense, Fn &&fn) {
  if (!dense) {
    for (int32_t x = m0; x < m1; ++x) {
      uint32_t m = map[x];
      if (!m) continue;
      map[x] = 0;
      do {
        const int32_t b = __ffs(m) - 1;
        m &= m - 1;
        fn(start++, (x << 5) + b);
      } while (m);
    }
    return;
  }
  const int lane = threadIdx.x & 31;
  for (int src = 0; src < 32; ++src) {
    const int32_t a = __shfl_sync(0xffffffffu, m0, src), b = __shfl_sync(0xffffffffu, m1, src);
    int32_t t = __shfl_sync(0xffffffffu, start, src);
    for (int32_t x = a; x < b; ++x) {
      const uint32_t m = map[x];
      if ((m >> lane) & 1u) fn(t + __popc(m & ((1u << lane) - 1u)), (x << 5) + lane);
      t += __popc(m);
    }
  }
  __syncwarp();  // the warp's words are read
  for (int32_t x = m0; x < m1; ++x) map[x] = 0;
}

// fn(a[i]) for i = lo + threadIdx.x, lo + threadIdx.x + NT, ... < hi, with Q
// loads issued together before their first use (the scratch reads are
// latency-bound).
template <int NT, int Q, class Fn>
__device__ __forceinline__ void for_each_batched(const int32_t *a, int32_t lo, int32_t hi,
                                                 Fn &&fn) {
  for (int32_t i0 = lo + (int32_t)threadIdx.x; i0 < hi; i0 += Q * NT) {
    int32_t v[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      const int32_t i = i0 + q * NT;
      v[q] = i < hi ? a[i] : 0;
    }
#pragma unroll
    for (int q = 0; q < Q; ++q)
      if (i0 + q * NT < hi) fn(v[q]);
  }
}

// First position p in core_list[0, n) with core_list[p] >= x.
__device__ __forceinline__ int32_t core_lower(const int32_t *core_list, int32_t n, int32_t x) {
  int32_t a = 0, b = n;
  while (a < b) {
    const int32_t mid = (a + b) >> 1;
    if (__ldg(core_list + mid) < x) a = mid + 1;
    else b = mid;
  }
  return a;
}

// ------------------------------------------------- shared-memory tables --
//
// An open-addressing table of T = 2^lgT 64-bit slots in shared memory, each
// slot (f << 32 | count) for a far end f; kEmpty64 marks a free slot.  The
// table holds at least twice the distinct keys it will receive, so it never
// fills.  A new key costs one CAS, a repeated one a 32-bit add to the slot's
// count word (see table_insert).  After the walk the slots with count >= s (found
// from the survivor list for s >= 2, by a pass over the table for s = 1) are
// moved to the front of the table, already packed as sort keys, and sorted
// by f.

constexpr unsigned long long kEmpty64 = 0xFFFFFFFF00000000ull;

// Survivor list (s >= 2): a key whose count reaches s during the inserts
// appends its slot to `slot` (one extra shared atomic per surviving pair),
// so collecting the survivors needs no pass over the table.  Counts only
// grow, so each key crosses s exactly once.  `cap` bounds the list (a
// survivor takes at least two wedges, or is one of at most T/2 keys).
struct SurvList {
  int32_t *slot;
  int32_t *n;
  int32_t cap;
};

__device__ __forceinline__ void note_survivor(const SurvList &sl, uint32_t h, int32_t old,
                                              int32_t add, int32_t smin, Meta *meta) {
  if (old < smin && old + add >= smin) {
    const int32_t p = atomicAdd(sl.n, 1);
    if (p < sl.cap) sl.slot[p] = (int32_t)h;
    else raise_error(meta, SLG_ERR_INVALID, kWhereHash);  // unreachable by the bound
  }
}

// The count word of slot h: its low 32 bits (the key word is the high half).
// Counts grow by 32-bit atomic adds, several times faster than 64-bit ones
// in shared memory on this GPU.
__device__ __forceinline__ uint32_t *count_word(unsigned long long *tab, uint32_t h) {
  return reinterpret_cast<uint32_t *>(tab + h);
}

// Inserts `add` wedges to far end f.  Unweighted: a count that reached s is
// not raised further.
//  - With the survivor list (s >= 2; mostly new keys in sparse rows) the key
//    word alone is claimed with a 32-bit CAS and the claim itself stands for
//    one wedge: the count word holds count - 1 (table_collect_list adds the
//    1 back).  A repeated key adds to the count word.
//  - Otherwise a probe reads the slot first (sparing repeated keys the CAS)
//    and a new key is claimed with one 64-bit CAS that also sets its count.
template <bool LIST>
__device__ __forceinline__ void table_insert(unsigned long long *tab, int lgT, int32_t f,
                                             int32_t add, int32_t smin, bool unweighted,
                                             Meta *meta, const SurvList &sl) {
  const uint32_t mask = (1u << lgT) - 1u;
  const unsigned long long key = (unsigned long long)(uint32_t)f << 32;
  uint32_t h = ((uint32_t)f * 0x9E3779B1u) >> (32 - lgT);
  for (uint32_t probe = 0; probe <= mask; ++probe) {
    if (LIST) {
      uint32_t *cw = count_word(tab, h);
      const uint32_t k = atomicCAS(cw + 1, 0xFFFFFFFFu, (uint32_t)f);  // key word
      if (k == 0xFFFFFFFFu) {  // claimed: count 1 so far
        if (add > 1) {
          const int32_t old = (int32_t)atomicAdd(cw, (uint32_t)(add - 1));
          note_survivor(sl, h, old + 1, add - 1, smin, meta);
        }
        return;
      }
      if (k == (uint32_t)f) {
        if (unweighted && (int32_t)*(volatile uint32_t *)cw + 1 >= smin) return;
        const int32_t old = (int32_t)atomicAdd(cw, (uint32_t)add);
        note_survivor(sl, h, old + 1, add, smin, meta);
        return;
      }
      h = (h + 1) & mask;
      continue;
    }
    unsigned long long cur = *(volatile unsigned long long *)(tab + h);
    if (cur == kEmpty64) {
      cur = atomicCAS(tab + h, kEmpty64, key | (uint32_t)add);
      if (cur == kEmpty64) return;
    }
    if ((cur & kEmpty64) == key) {
      if (!unweighted || (int32_t)(uint32_t)cur < smin) atomicAdd(count_word(tab, h), (uint32_t)add);
      return;
    }
    h = (h + 1) & mask;
  }
  raise_error(meta, SLG_ERR_INVALID, kWhereHash);  // unreachable: T >= 2 x distinct
}

// Table size for a multiset with at most `distinct` keys: 2^lgT >= 2 x distinct.
__device__ __forceinline__ int table_lg(int32_t distinct, int lg_max) {
  int lg = ceil_log2(2 * (distinct > 16 ? distinct : 16));
  return lg < lg_max ? lg : lg_max;
}

// Ascending order of one key per lane across a warp: a bitonic network on
// shuffles (for k = 32 every lane is in an ascending half).
__device__ __forceinline__ unsigned long long warp_sort32(unsigned long long x) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int k = 2; k <= 32; k <<= 1)
#pragma unroll
    for (int j = k >> 1; j > 0; j >>= 1) {
      const unsigned long long y = __shfl_xor_sync(0xffffffffu, x, j);
      const bool keep_min = ((lane & j) == 0) == ((lane & k) == 0);
      x = keep_min ? (x < y ? x : y) : (x < y ? y : x);
    }
  return x;
}

// Number of keys below x in a sorted run a[0, 32): branch-free binary search.
__device__ __forceinline__ int32_t run_below(const unsigned long long *a, unsigned long long x) {
  int32_t c = 0;
#pragma unroll
  for (int st = 16; st > 0; st >>= 1)
    if (a[c + st - 1] < x) c += st;
  return c + (a[c] < x);  // adds one only when c = 31 and all 32 are below
}

// Sorts the distinct keys tab[0, n) by f and returns where they are.
//  - small n (<= 64 with 512 threads, <= 512 with fewer): each key's rank is
//    the number of keys below it (one broadcast pass), written to [n, 2 n);
//  - 512 threads, n <= 1024: each warp sorts runs of 32 keys in registers
//    (padding ~0, above every key) and stores them back; a key's place is
//    then the sum over all runs of the keys below it (its own run contributes
//    its index), written to [32 nr, 32 nr + n) for nr = ceil(n / 32) runs.
//    (Smaller blocks keep the rank pass: the run code's registers would cost
//    them a resident block per SM.)
//  - larger n: a bitonic sort in place over [0, n2), n2 = 2^ceil(log2 n).
// `*used` receives the end of the region touched; it stays within
// max(T, 2 n + 32) <= the table's capacity for T >= 2 n.
template <int NT, bool RUNS = (NT >= 512)>
__device__ __forceinline__ int32_t sort_survivors(unsigned long long *tab, int32_t n,
                                                  int32_t *used) {
  constexpr bool kRuns = RUNS;
  if (n <= (kRuns ? 64 : 512)) {
    for (int32_t i = threadIdx.x; i < n; i += NT) {
      const unsigned long long x = tab[i];
      int32_t r = 0;
      for (int32_t j = 0; j < n; ++j) r += tab[j] < x;
      tab[n + r] = x;
    }
    __syncthreads();
    *used = 2 * n;
    return n;
  }
  if constexpr (kRuns) {
    if (n <= 8 * NT) {
      const int32_t nr = (n + 31) >> 5;
      for (int32_t r = (int32_t)threadIdx.x >> 5; r < nr; r += NT / 32) {
        const int32_t i = (r << 5) + (int32_t)(threadIdx.x & 31);
        const unsigned long long x = warp_sort32(i < n ? tab[i] : ~0ull);
        tab[i] = x;  // the run's loads precede the shuffles
      }
      __syncthreads();
      const int32_t out = nr << 5;
      for (int32_t i = threadIdx.x; i < n; i += NT) {
        const unsigned long long x = tab[i];
        int32_t r = 0;
        int32_t q = 0;
        for (; q + 4 <= nr; q += 4) {
          const int32_t c0 = run_below(tab + (q << 5), x);
          const int32_t c1 = run_below(tab + ((q + 1) << 5), x);
          const int32_t c2 = run_below(tab + ((q + 2) << 5), x);
          const int32_t c3 = run_below(tab + ((q + 3) << 5), x);
          r += c0 + c1 + c2 + c3;
        }
        for (; q < nr; ++q) r += run_below(tab + (q << 5), x);
        tab[out + r] = x;
      }
      __syncthreads();
      *used = out + n;
      return out;
    }
  }
  int32_t n2 = 1;
  while (n2 < n) n2 <<= 1;
  for (int32_t i = n + threadIdx.x; i < n2; i += NT) tab[i] = ~0ull;
  __syncthreads();
  for (int32_t k = 2; k <= n2; k <<= 1) {
    for (int32_t jj = k >> 1; jj > 0; jj >>= 1) {
      for (int32_t i = threadIdx.x; i < n2; i += NT) {
        const int32_t ixj = i ^ jj;
        if (ixj > i) {
          const unsigned long long x = tab[i], y = tab[ixj];
          if ((x > y) == ((i & k) == 0)) {
            tab[i] = y;
            tab[ixj] = x;
          }
        }
      }
      __syncthreads();
    }
  }
  *used = n2;
  return 0;
}

// fn(r, x) for every key x of k[0, n) with r = the number of keys below x
// (distinct keys): for n <= 64 (or always, without RUNS) by one broadcast
// pass, else from runs of 32
// sorted in place (k[0, 32 ceil(n / 32)) is overwritten, padded with ~0)
// and binary searches over them.  No barrier after the calls.
template <int NT, bool RUNS = true, class Fn>
__device__ __forceinline__ void rank_keys(unsigned long long *k, int32_t n, Fn &&fn) {
  if (!RUNS || n <= 64) {
    for (int32_t i = threadIdx.x; i < n; i += NT) {
      const unsigned long long x = k[i];
      int32_t r = 0;
      for (int32_t j = 0; j < n; ++j) r += k[j] < x;
      fn(r, x);
    }
    return;
  }
  if constexpr (!RUNS) return;
  const int32_t nr = (n + 31) >> 5;
  for (int32_t q = (int32_t)threadIdx.x >> 5; q < nr; q += NT / 32) {
    const int32_t i = (q << 5) + (int32_t)(threadIdx.x & 31);
    const unsigned long long x = warp_sort32(i < n ? k[i] : ~0ull);
    k[i] = x;  // the run's loads precede the shuffles
  }
  __syncthreads();
  // runs 0 .. nr-2 are full and the last one holds its keys first, so
  // k[0, n) holds every key once
  for (int32_t i = threadIdx.x; i < n; i += NT) {
    const unsigned long long x = k[i];
    int32_t r = 0;
    for (int32_t q = 0; q < nr; ++q) r += run_below(k + (q << 5), x);
    fn(r, x);
  }
}

// Survivors by a pass over the table (used for s = 1, where every key
// survives).
// Rounds of RND slots per thread (slot = (round * RND + i) * NT + thread):
// a round reads its slots into registers, a block scan places the ones that
// qualify, and they are written to the front of the table.  A write of round
// r lands below the number of qualifying slots seen so far, hence on a slot
// of round r or earlier, all of which were read before the round's scan.
// Returns the number of survivors; with `sort` they are in ascending f at
// tab[*sorted_at, *sorted_at + count), and tab[0, *used) must be cleared
// after use (table_reset_front).
template <int NT, int SPT, bool RUNS = (NT >= 512)>
__device__ __forceinline__ int32_t table_collect(unsigned long long *tab, int32_t T, int32_t smin,
                                                 bool sort, int32_t *ws, int32_t *sorted_at,
                                                 int32_t *used) {
  constexpr int RND = SPT < 8 ? SPT : 8;
  int32_t run = 0;
  for (int32_t r0 = 0; r0 * NT < T; r0 += RND) {
    unsigned long long kv[RND];
    int32_t c = 0;
#pragma unroll
    for (int i = 0; i < RND; ++i) {
      const int32_t slot = (r0 + i) * NT + (int32_t)threadIdx.x;
      kv[i] = slot < T ? tab[slot] : kEmpty64;
      c += (kv[i] != kEmpty64) & ((int32_t)(uint32_t)kv[i] >= smin);
    }
    int32_t total;
    const int32_t inc = block_inclusive_scan<NT>(c, ws, &total);  // the round's reads done
    if (sort) {
      int32_t pos = run + inc - c;
#pragma unroll
      for (int i = 0; i < RND; ++i)
        if (kv[i] != kEmpty64 && (int32_t)(uint32_t)kv[i] >= smin) tab[pos++] = kv[i];
    }
    run += total;
  }
  *used = T;
  if (sort && run > 0) {
    __syncthreads();  // compaction writes done
    int32_t u;
    *sorted_at = sort_survivors<NT, RUNS>(tab, run, &u);
    *used = max(T, u);
  }
  return run;
}

// Marks tab[0, n) free with 16-byte stores (tab is 16-byte aligned; an odd n
// also clears slot n, which is free already or inside the region in use).
template <int NT>
__device__ __forceinline__ void clear_slots(unsigned long long *tab, int32_t n) {
  ulonglong2 *t2 = reinterpret_cast<ulonglong2 *>(tab);
  const ulonglong2 e = make_ulonglong2(kEmpty64, kEmpty64);
  for (int32_t i = threadIdx.x; i < (n + 1) >> 1; i += NT) t2[i] = e;
}

// Survivors from the list: read their (f, count) slots, clear the whole
// table (plain stores), and with `sort` place them compactly at the front
// and sort them.  Returns the number of survivors; with `sort` they are in
// ascending f at tab[*sorted_at, + count) and tab[0, *used) must be cleared
// after use (table_reset_front).  QMAX x NT >= the list's capacity.
template <int NT, int QMAX>
__device__ __forceinline__ int32_t table_collect_list(unsigned long long *tab, int32_t T,
                                                      const SurvList &sl, bool sort,
                                                      int32_t *sorted_at, int32_t *used) {
  __syncthreads();  // every insert done: the list is final
  const int32_t n = min(*sl.n, sl.cap);
  unsigned long long x[QMAX];
#pragma unroll
  for (int q = 0; q < QMAX; ++q) {
    const int32_t i = (int32_t)threadIdx.x + q * NT;
    x[q] = (sort && i < n) ? tab[sl.slot[i]] + 1ull : 0ull;  // count word holds count - 1
  }
  __syncthreads();  // reads done before the table is cleared
  clear_slots<NT>(tab, T);
  if (threadIdx.x == 0) *sl.n = 0;
  __syncthreads();
  *used = 0;
  *sorted_at = 0;
  if (!sort || n == 0) return n;
#pragma unroll
  for (int q = 0; q < QMAX; ++q) {
    const int32_t i = (int32_t)threadIdx.x + q * NT;
    if (i < n) tab[i] = x[q];
  }
  __syncthreads();
  *sorted_at = sort_survivors<NT>(tab, n, used);
  return n;
}

// Clears tab[0, used) after the survivors were emitted.
template <int NT>
__device__ __forceinline__ void table_reset_front(unsigned long long *tab, int32_t used) {
  __syncthreads();  // sorted entries may still be read
  clear_slots<NT>(tab, used);
  __syncthreads();
}

}  // namespace slg
