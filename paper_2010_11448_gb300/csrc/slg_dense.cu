// The dense bin of the s-overlap walk: rows whose far ends are dense enough
// in their id span to be counted in an array of counters, one per id, a
// window of ids at a time.
//
// A row's tails are ascending lists.  The kernel keeps a cursor per tail and
// sweeps the row's id span [f_lo, f_hi) in windows; in a window every tail
// gives its entries below the window's end, read in order from its cursor,
// straight to the shared counters (one shared atomic per wedge).  There is
// no flattened copy, no partition and no hashing: the row's wedges are read
// once, as they lie in the filtered CSC, and the survivors come out in
// ascending id.
//
// Counters are as narrow as the row allows: a count |e ∩ f| never exceeds
// |e|, so rows of at most 15, 255 and 65,535 vertices use 4-, 8- and 16-bit
// counters packed in 32-bit words (additions never carry into a neighbour).
// A window of the small instance's 10,240 words holds 81,920 ids with 4-bit and
// 40,960 with 8-bit counters; one of the large instance's 48,128 words 96,256 with
// 16 bits and 48,128 with 32.
//
// A counter that reaches s sets its id's bit in a map of survivors (one more
// shared atomic per surviving pair), so that the window's end reads one bit
// per id, not the counters.  A sweep step's cost is the latency of its cursor
// and far-end loads, so several list entries are in flight per warp, and the
// fewer windows a row has the better: rows of more than kDenseBigSize
// vertices (short pieces of many tails: 3 to 8 entries of a tail in a window
// of 26K ids) take the large instance, one CTA of 1,024 threads per SM; the
// others the small one, four CTAs of 256 threads.
//
// Measured on chung_lu_1m (1M x 2M) against the partitioned hash buckets and
// dense windows of the giant bin that these rows took before: L_8 of H, giant
// bin 8.8 ms -> big 4.1, small 1.1, giant 1.5 ms; L_2 of H*, 47.7 ms -> big
// 8.7, small 10.7, giant 17.3 ms.  A scan of the counters in place of the
// survivor bits cost 26 instead of 13 x 10^9 CTA cycles on L_2(H*) (rows down
// to one wedge per 32 ids); windows of 26K ids for every row took 13.9
// instead of 9.2 ms on L_2(H).  The small instance with three CTAs of 512
// threads and windows of 104K / 52K ids, as it first was: half of its warps'
// time went on barriers (few tails per window and warp); L_8 of a 300K x 600K
// dual 10.98 -> 9.53 ms, step of chung_lu_1m 118.4 -> 115.1 ms with four
// of 256 threads (five with 8,192 words: 9.83, 117.6; eight of 128 threads
// with 4,608 words: 8.86, 118.8).
//
// The longest tails are split over the warps in blocks of 32 entries, a
// cursor per warp.  They had been cut into runs of 256 entries per window, of
// which a window meets only some, so that its warps waited for one another
// (barriers were half of a warp's time): L_2 sweep of a 150K x 300K dual
// 10,134 -> 9,351 us (11,383 with the tails left whole), L_3 of a 30K x 60K
// dual 1,346 -> 1,322 (1,702).  From 128, 256, 512 entries per window: sweep
// 9,651, 9,661, 9,866 us, step of chung_lu_1m 106.3, 105.7, 105.7 ms.  4-bit
// counters tried first for rows of 16 to 64 vertices, the row counted anew on
// an overflow, gave 3 % on the sweep, nothing elsewhere, and lose where rows
// are alike: not kept.
#include <algorithm>
#include <mutex>

#include "slg_walk.cuh"

namespace slg {

namespace {

#ifndef SLG_DN_NT
#define SLG_DN_NT 256
#endif
#ifndef SLG_DN_MINB
#define SLG_DN_MINB 4
#endif
#ifndef SLG_DN_LONG
#define SLG_DN_LONG 16
#endif
#ifndef SLG_DN_SPLIT
#define SLG_DN_SPLIT 256
#endif
#ifndef SLG_DN_BIG_SPLIT
#define SLG_DN_BIG_SPLIT 1024
#endif
#ifndef SLG_DN_US
#define SLG_DN_US 2
#endif
#ifndef SLG_DN_UL
#define SLG_DN_UL 2
#endif

// The two instances of the kernel: NT threads, WORDS counter words per
// window, MAP words of survivor bits (counters of at least 32 WORDS / (32
// MAP) bits), MINB CTAs per SM, ENT list entries in shared memory, NSPLIT
// split tails at most, from SPLIT entries per window.
struct DnSmall {
  static constexpr int NT = SLG_DN_NT, MINB = SLG_DN_MINB, WORDS = SLG_DN_WORDS, MAP = WORDS / 4;
  static constexpr int NSPLIT = 16, SPLIT = SLG_DN_SPLIT, UL = SLG_DN_UL, US = SLG_DN_US;
  static constexpr int ENT = kDenseBigSize + 1;
};
struct DnBig {
  static constexpr int NT = 1024, MINB = 1, WORDS = SLG_DN_BIG_WORDS, MAP = WORDS / 16;
  static constexpr int NSPLIT = 16, SPLIT = SLG_DN_BIG_SPLIT, UL = 2, US = 4;
  static constexpr int ENT = 512;
};

// [counters][survivor bits][entries C::ENT x 8][split cursors NSPLIT x NW x 8]
// [totals 2 x 32 x 4][n_long, n_short, row, n_split][base 8]
template <class C>
constexpr size_t dense_smem() {
  static_assert(C::WORDS % 64 == 0, "16-byte alignment of the parts");
  return (size_t)C::WORDS * 4 + (size_t)C::MAP * 4 + (size_t)C::ENT * 8 +
         (size_t)C::NSPLIT * (C::NT / 32) * 8 + 2 * 32 * 4 + 16 + 16;
}

// Adds n to counter o (2^LB bits wide, packed in 32-bit words); when this
// takes it to s or above, marks o in the survivor bits and returns 1.
template <int LB>
__device__ __forceinline__ int32_t dn_add(uint32_t *cnt, uint32_t *map, int32_t o, uint32_t n,
                                          uint32_t smin, bool mark) {
  constexpr int LW = 5 - LB;                     // log2 counters per word
  constexpr uint32_t kField = LB == 5 ? ~0u : (1u << ((1 << LB) & 31)) - 1u;
  const int sh = (o & ((1 << LW) - 1)) << LB;
  const uint32_t old = (atomicAdd(cnt + (o >> LW), n << sh) >> sh) & kField;
  if (!(old < smin && old + n >= smin)) return 0;
  if (mark) atomicOr(map + (o >> 5), 1u << (o & 31));
  return 1;
}

// One window's sweep over the row's list entries; the counters of ids
// [F0, F1).  Returns the thread's number of survivors; *any: something was
// counted.  Bound by the latency of the cursor and far-end loads, so several
// entries' loads are in flight per warp.
template <int LB, class C>
__device__ __forceinline__ int32_t dn_sweep(const int32_t *__restrict__ c_idx, int2 *ent,
                                            int32_t nl, int2 *ent_s, int32_t ns, int2 *split,
                                            int32_t nh, int32_t F0, int32_t F1, uint32_t *cnt,
                                            uint32_t *map, uint32_t smin, bool mark, bool *any) {
  constexpr int NW = C::NT / 32, UL = C::UL, US = C::US;
  const int32_t lane = (int32_t)(threadIdx.x & 31), wq = (int32_t)(threadIdx.x >> 5);
  int32_t c = 0;
  // split tails: every warp takes each NW-th block of 32 entries, two blocks
  // per step; the block in which the window ends is read again by the next
  const uint32_t span = (uint32_t)(F1 - F0);
  for (int32_t x = 0; x < nh; ++x) {
    const int2 en = split[x * NW + wq];
    // unsigned: a cursor may lie 64 NW beyond the last incidence
    const uint32_t end = (uint32_t)en.y;
    uint32_t cur = (uint32_t)en.x;
    for (;;) {  // warp-uniform
      const uint32_t i = cur + lane;
      const int32_t a = i < end ? __ldg(c_idx + i) : 0x7fffffff;
      const int32_t b = i + 32 * NW < end ? __ldg(c_idx + i + 32 * NW) : 0x7fffffff;
      const bool v0 = (uint32_t)(a - F0) < span, v1 = (uint32_t)(b - F0) < span;
      if (v0) c += dn_add<LB>(cnt, map, a - F0, 1u, smin, mark);
      if (v1) c += dn_add<LB>(cnt, map, b - F0, 1u, smin, mark);
      *any |= v0 | v1;
      if (!__all_sync(0xffffffffu, a < F1)) break;
      cur += 32 * NW;
      if (!__all_sync(0xffffffffu, b < F1)) break;
      cur += 32 * NW;
    }
    if (cur != (uint32_t)en.x && lane == 0) split[x * NW + wq].x = (int32_t)cur;
  }
  // long tails, a warp each, 64 entries per step
  for (int32_t x0 = wq; x0 < nl; x0 += UL * NW) {
    int2 en[UL];
    int32_t f[UL][2];
#pragma unroll
    for (int u = 0; u < UL; ++u) {
      const int32_t x = x0 + u * NW;
      en[u] = x < nl ? ent[x] : make_int2(0, 0);
    }
#pragma unroll
    for (int u = 0; u < UL; ++u) {
      const uint32_t i = (uint32_t)en[u].x + lane, end = (uint32_t)en[u].y;  // (as above)
      f[u][0] = i < end ? __ldg(c_idx + i) : 0x7fffffff;
      f[u][1] = i + 32 < end ? __ldg(c_idx + i + 32) : 0x7fffffff;
    }
#pragma unroll
    for (int u = 0; u < UL; ++u) {
      int32_t cur = en[u].x, a = f[u][0], b = f[u][1];
      for (;;) {  // warp-uniform
        const bool v0 = a < F1, v1 = b < F1;
        if (v0) c += dn_add<LB>(cnt, map, a - F0, 1u, smin, mark);
        if (v1) c += dn_add<LB>(cnt, map, b - F0, 1u, smin, mark);
        const int32_t n = __popc(__ballot_sync(0xffffffffu, v0)) +
                          __popc(__ballot_sync(0xffffffffu, v1));
        cur += n;
        if (n < 64) break;
        const uint32_t i = (uint32_t)cur + lane, end = (uint32_t)en[u].y;
        a = i < end ? __ldg(c_idx + i) : 0x7fffffff;
        b = i + 32 < end ? __ldg(c_idx + i + 32) : 0x7fffffff;
      }
      if (cur != en[u].x) {
        *any = true;
        if (lane == 0) ent[x0 + u * NW].x = cur;
      }
    }
  }
  // short tails, 8 lanes each
  const int sub = lane >> 3, l8 = lane & 7;
  for (int32_t x0 = wq * 4; x0 < ns; x0 += US * NW * 4) {
    int2 en[US];
    int32_t f[US];
#pragma unroll
    for (int u = 0; u < US; ++u) {
      const int32_t x = x0 + u * NW * 4 + sub;
      en[u] = x < ns ? ent_s[x] : make_int2(0, 0);
    }
#pragma unroll
    for (int u = 0; u < US; ++u) {
      const uint32_t i = (uint32_t)en[u].x + l8;
      f[u] = i < (uint32_t)en[u].y ? __ldg(c_idx + i) : 0x7fffffff;
    }
#pragma unroll
    for (int u = 0; u < US; ++u) {
      int32_t cur = en[u].x, a = f[u];
      for (;;) {
        const bool v = a < F1;
        if (v) c += dn_add<LB>(cnt, map, a - F0, 1u, smin, mark);
        const int32_t n = __popc((__ballot_sync(0xffffffffu, v) >> (sub << 3)) & 0xFFu);
        cur += n;
        if (!__any_sync(0xffffffffu, n == 8)) break;
        const uint32_t i = (uint32_t)cur + l8;
        a = n == 8 && i < (uint32_t)en[u].y ? __ldg(c_idx + i) : 0x7fffffff;
      }
      if (cur != en[u].x) {
        *any = true;
        if (l8 == 0) ent_s[x0 + u * NW * 4 + sub].x = cur;
      }
    }
  }
  return c;
}

// part 0: the rows handed out first (the front of the list), 1: the others
// (its back), each on its own ticket.
template <class C>
__global__ __launch_bounds__(C::NT, C::MINB) void k_walk_dense(
    Walk w, const int32_t *__restrict__ rows, EmitArgs a, int32_t *__restrict__ scratch,
    long long stride, long long pair_cap, int32_t ent_cap, int32_t R, int32_t list_len, int part) {
  constexpr int NT = C::NT, NW = NT / 32;
  Meta *meta = a.meta;
  if (meta->err) return;
  extern __shared__ __align__(16) unsigned char smem[];
  uint32_t *cnt = reinterpret_cast<uint32_t *>(smem);
  uint4 *cnt4 = reinterpret_cast<uint4 *>(smem);
  uint32_t *map = cnt + C::WORDS;
  int2 *s_ent = reinterpret_cast<int2 *>(map + C::MAP);
  int2 *split = s_ent + C::ENT;
  int32_t *s_tot = reinterpret_cast<int32_t *>(split + C::NSPLIT * NW);
  int32_t *s_n = s_tot + 64;  // [0] long entries, [1] short entries, [2] row, [3] split tails
  long long *s_base = reinterpret_cast<long long *>(s_n + 4);
  // per-CTA global scratch: staged pairs (j, w), then the list entries of
  // rows with more tails than shared memory holds
  int32_t *tj = scratch + (long long)blockIdx.x * stride;
  int32_t *tw = tj + pair_cap;
  int2 *g_ent = reinterpret_cast<int2 *>(tw + pair_cap);
  const int32_t tid = (int32_t)threadIdx.x, lane = tid & 31, wq = tid >> 5;
  for (int32_t i = tid; i < (C::WORDS + C::MAP) / 4; i += NT)
    cnt4[i] = make_uint4(0, 0, 0, 0);
  // part 0: rows[0, dense_huge); part 1: the others, which end at rows[list_len)
  const unsigned nrows = part ? meta->dense_rest : meta->dense_huge;
  unsigned *ticket = part ? &meta->dense_ticket_rest : &meta->dense_ticket;
  const bool unweighted = a.unweighted != 0;
  const bool emit = a.mode != kCount;
  long long cycles = 0;
  for (;;) {
    __syncthreads();
    if (tid == 0) {
      const unsigned t = atomicAdd(ticket, 1u);
      s_n[0] = 0;
      s_n[1] = 0;
      s_n[3] = 0;
      s_n[2] = t >= nrows ? -1 : rows[part ? list_len - 1 - t : t];
    }
    __syncthreads();
    const int32_t e = s_n[2];
    if (e < 0) break;
    const long long t0 = clock64();
    const int32_t smin = s_of(a.row_s, a.smin, e);
    const int32_t f_lo = a.full_rows ? 0 : e + 1;
    const int32_t f_hi = a.row_fhi ? a.row_fhi[e] : R;
    const int32_t k0 = w.r_off[e], k1 = w.r_off[e + 1];
    const CoreInfo &ci = a.core;
    const bool core_row = ci.T && ci.row_rank[e + 1] != ci.row_rank[e];
    const int32_t ri = core_row ? ci.row_rank[e] : 0;
    const int32_t *Trow = core_row ? ci.T + (long long)ri * ci.Mp : nullptr;
    const long long dbase = a.mode == kDirect ? a.row_ptr[e - a.row_begin] : -1;
    int32_t out = 0;  // pairs of the row so far
    int32_t mine = 0;  // count mode: the thread's survivors
    bool fail = false;
    const int lb = dense_lg_bits(k1 - k0);
    const int lw = 5 - lb;
    const int32_t win = C::WORDS << lw;  // ids per window
    const int32_t nwin = (f_hi - f_lo + win - 1) / win;
    // 1. the row's non-empty tails as list entries (cursor, end): the ones
    // with many entries per window from the front (a warp sweeps one), the
    // others from the back (8 lanes sweep one).  The longest, of which there
    // can be fewer than NSPLIT, are split over all warps, with a cursor each,
    // so that no warp sweeps far more of a window than the others.
    const bool in_smem = k1 - k0 <= C::ENT;
    int2 *ent = in_smem ? s_ent : g_ent;
    const int32_t ecap = in_smem ? C::ENT : ent_cap;
    if (!in_smem && k1 - k0 > ent_cap) {  // sized by the planning: cannot happen
      if (tid == 0) raise_error(meta, SLG_ERR_INVALID, kWhereGiant);
      break;
    }
    const int32_t work = a.row_work[e - a.row_begin];
    const int32_t split_min = max(C::SPLIT * min(nwin, 1 << 20), work / C::NSPLIT + 1);
    const int32_t long_min = SLG_DN_LONG * min(nwin, 1 << 24);
    for (int32_t k = k0 + tid; k < k1; k += NT) {
      const int32_t b = __ldg(w.tail_beg + k), end = __ldg(w.tail_end + k), n = end - b;
      if (n <= 0) continue;
      const int32_t h = n >= split_min ? atomicAdd(s_n + 3, 1) : C::NSPLIT;
      if (h < C::NSPLIT) {
        for (int32_t q = 0; q < NW; ++q)
          split[h * NW + q] = make_int2((int32_t)((uint32_t)b + 32u * q), end);
      } else {
        const int32_t pos =
            n >= long_min ? atomicAdd(s_n + 0, 1) : ecap - 1 - atomicAdd(s_n + 1, 1);
        ent[pos] = make_int2(b, end);
      }
    }
    __syncthreads();
    const int32_t nl = s_n[0], ns = s_n[1], nh = min(s_n[3], C::NSPLIT);
    int2 *ent_s = ent + (ecap - ns);
    int par = 0;
    for (int32_t F0 = f_lo; F0 < f_hi; F0 += win) {
      const int32_t F1 = f_hi - F0 > win ? F0 + win : f_hi;
      bool any = false;
      // 2. sweep
      if (lb == 2) mine += dn_sweep<2, C>(w.c_idx_s, ent, nl, ent_s, ns, split, nh, F0, F1, cnt, map, smin, emit, &any);
      else if (lb == 3) mine += dn_sweep<3, C>(w.c_idx_s, ent, nl, ent_s, ns, split, nh, F0, F1, cnt, map, smin, emit, &any);
      else if (lb == 4) mine += dn_sweep<4, C>(w.c_idx_s, ent, nl, ent_s, ns, split, nh, F0, F1, cnt, map, smin, emit, &any);
      else mine += dn_sweep<5, C>(w.c_idx_s, ent, nl, ent_s, ns, split, nh, F0, F1, cnt, map, smin, emit, &any);
      if (core_row) {
        // tile counts of the core rows in the window, after row e itself
        const int32_t p0 = max(core_lower(ci.core_list, ci.n_core, F0), ri + 1);
        const int32_t p1 = core_lower(ci.core_list, ci.n_core, F1);
        for (int32_t p = p0 + tid; p < p1; p += NT) {
          const int32_t f = ci.core_list[p];
          const int32_t wt = Trow[p];
          if (wt > 0 && w.r_off[f + 1] - w.r_off[f] >= smin) {
            any = true;
            const int32_t o = f - F0;
            if (lb == 2) mine += dn_add<2>(cnt, map, o, wt, smin, emit);
            else if (lb == 3) mine += dn_add<3>(cnt, map, o, wt, smin, emit);
            else if (lb == 4) mine += dn_add<4>(cnt, map, o, wt, smin, emit);
            else mine += dn_add<5>(cnt, map, o, wt, smin, emit);
          }
        }
      }
      if (!__syncthreads_or(any)) continue;  // nothing counted: the counters are clear
      const int32_t nword = ((F1 - F0) + (1 << lw) - 1) >> lw;  // counter words in use
      if (emit) {
        // 3. survivors in ascending id: each thread owns consecutive words
        // of the survivor bits
        const int32_t nm = ((F1 - F0) + 31) >> 5;
        const int32_t wpt = (nm + NT - 1) / NT;
        const int32_t m0 = min(tid * wpt, nm), m1 = min(m0 + wpt, nm);
        int32_t c = 0;
        for (int32_t x = m0; x < m1; ++x) c += __popc(map[x]);
        const int32_t inc = warp_inclusive_scan(c);
        if (lane == 31) s_tot[par * 32 + wq] = inc;
        __syncthreads();
        const int32_t wt = lane < NW ? s_tot[par * 32 + lane] : 0;
        const int32_t wi = warp_inclusive_scan(wt);
        const int32_t total = __shfl_sync(0xffffffffu, wi, 31);
        const int32_t before = __shfl_sync(0xffffffffu, wi - wt, wq);
        par ^= 1;
        if (a.mode == kStage && (long long)out + total > pair_cap) {  // uniform: cannot happen
          if (tid == 0) raise_error(meta, SLG_ERR_INVALID, kWhereGiant);
          fail = true;
          break;
        }
        const uint32_t field = lb == 5 ? ~0u : (1u << (1 << lb)) - 1u;
        auto emit_one = [&](int32_t t, int32_t o) {
          const int32_t n =
              (int32_t)((cnt[o >> lw] >> ((o & ((1 << lw) - 1)) << lb)) & field);
          if (a.mode == kDirect) {
            put(a, dbase, t, e, F0 + o, n);
          } else {
            tj[t] = F0 + o;
            if (!unweighted) tw[t] = n;
          }
        };
        for_survivors(map, m0, m1, out + before + inc - c, total > kSurvDense * nm, emit_one);
        out += total;
        __syncthreads();  // the counters are read
      }
      for (int32_t i = tid; i < (nword + 3) >> 2; i += NT) cnt4[i] = make_uint4(0, 0, 0, 0);
      __syncthreads();
    }
    if (fail) break;
    if (!emit) {  // uniform: the survivors were counted as they appeared
#pragma unroll
      for (int d = 16; d > 0; d >>= 1) mine += __shfl_xor_sync(0xffffffffu, mine, d);
      if (lane == 0) s_tot[wq] = mine;
      __syncthreads();
      if (tid == 0) {
        out = 0;
        for (int i = 0; i < NW; ++i) out += s_tot[i];
      }
    }
    if (tid == 0) *s_base = reserve(a, e, out, kBinDense);
    __syncthreads();
    if (a.mode == kStage) {
      const long long b = *s_base;
      if (b >= 0) {
        for (int32_t i0 = tid; i0 < out; i0 += 4 * NT) {
          int32_t vj[4], vw[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int32_t i = i0 + u * NT;
            vj[u] = i < out ? tj[i] : 0;
            vw[u] = i < out && !unweighted ? tw[i] : 0;
          }
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int32_t i = i0 + u * NT;
            if (i < out) {
              a.stage_j[b + i] = vj[u];
              if (!unweighted) a.stage_w[b + i] = vw[u];
            }
          }
        }
      }
      __syncthreads();
      l2_discard(tj, out);  // the row's pairs are in the staging area
      if (!unweighted) l2_discard(tw, out);
    }
    cycles += clock64() - t0;
  }
  if (tid == 0) atomicAdd(&meta->giant_cycles[3], (unsigned long long)cycles);
}

struct DnOcc {
  int big = 0, small = 0;  // CTAs
  int dev = -1;
};

DnOcc &dn_occ() {
  static DnOcc occ[64];
  static std::mutex mu;
  int dev = 0;
  cudaGetDevice(&dev);
  DnOcc &o = occ[dev & 63];
  std::lock_guard<std::mutex> lock(mu);
  if (o.dev != dev) {
    int sms = 0, nb = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaFuncSetAttribute(k_walk_dense<DnBig>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)dense_smem<DnBig>());
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_walk_dense<DnBig>, DnBig::NT,
                                                  dense_smem<DnBig>());
    o.big = sms * std::max(nb, 1);
    cudaFuncSetAttribute(k_walk_dense<DnSmall>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)dense_smem<DnSmall>());
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_walk_dense<DnSmall>, DnSmall::NT,
                                                  dense_smem<DnSmall>());
    o.small = sms * std::max(nb, 1);
    o.dev = dev;
  }
  return o;
}

// Ints per CTA: pairs of the largest row (two arrays) and the entries of the
// row with the most tails.
template <class C>
long long dense_stride(long long max_pairs, int32_t max_size, long long *pair_cap,
                       int32_t *ent_cap) {
  *pair_cap = (max_pairs + 31) & ~31ll;
  *ent_cap = max_size > C::ENT ? (max_size + 15) & ~15 : 0;
  return 2 * *pair_cap + 2ll * *ent_cap;
}

}  // namespace

// Scratch ints of an instance (small: 0 the big one, 1 the other).
long long dense_ints(int small, long long pairs, int32_t size_big) {
  if (pairs <= 0) return 0;
  DnOcc &o = dn_occ();
  long long pc = 0;
  int32_t ec = 0;
  return small ? o.small * dense_stride<DnSmall>(pairs, kDenseBigSize, &pc, &ec)
               : o.big * dense_stride<DnBig>(pairs, size_big, &pc, &ec);
}

cudaError_t launch_walk_dense(const WalkLaunch &L, int small, cudaStream_t st) {
  DnOcc &o = dn_occ();
  const int32_t *rows = L.bin_rows + (int64_t)kBinDense * L.rows;
  long long pc = 0;
  int32_t ec = 0;
  if (!small) {
    const long long stride = dense_stride<DnBig>(L.dense_pairs[0], L.dense_size, &pc, &ec);
    k_walk_dense<DnBig><<<o.big, DnBig::NT, dense_smem<DnBig>(), st>>>(
        L.w, rows, L.a, L.dense_scratch[0], stride, pc, ec, L.R, L.rows, 0);
  } else {
    const long long stride = dense_stride<DnSmall>(L.dense_pairs[1], kDenseBigSize, &pc, &ec);
    k_walk_dense<DnSmall><<<o.small, DnSmall::NT, dense_smem<DnSmall>(), st>>>(
        L.w, rows, L.a, L.dense_scratch[1], stride, pc, ec, L.R, L.rows, 1);
  }
  return cudaGetLastError();
}

}  // namespace slg
