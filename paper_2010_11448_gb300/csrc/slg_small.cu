// Sides of at most kSmallRows rows: the whole call in three kernels and one
// host round trip.
//
// A small build is bound by the latency of its kernels (about 2 us each at
// the least) and host round trips (about 10 us), not by its wedges: the
// general path's planning, binning, five bin kernels, row scan, gather and
// three round trips took about 190 us on 2,000 hyperedges over 4,000
// vertices.  With the far ends of a row below kSmallRows there is nothing to
// plan: every row is counted in one window of counters over all ids.
//   k_small_check  validates both sides, finds each incidence's position in
//                  its column, marks the rows of size >= s;
//   k_small_walk   a CTA takes a row at a time: its tails (the entries after
//                  it in its columns) are counted in shared memory, far ends
//                  of size < s left out; the survivors, in ascending id from
//                  a bit map, go to the staging area;
//   k_small_emit   places the rows and copies them to the output; its last
//                  CTA hands the call's totals to the host.
#include <algorithm>
#include <mutex>

#include "slg_walk.cuh"

namespace slg {

namespace {

constexpr int kCkNT = 256;
constexpr int kCkK = 4;          // incidences per lane and warp of the map
constexpr int kSwNT = 256;      // (128, 512: L_2 of 16K x 30K 473, 310 us against 328, of a 16,000-row
                                // dual 616, 721 against 547)
constexpr int kSwNW = kSwNT / 32;
constexpr int kSwLongMin = 64;   // entries of a long tail (8 lanes read a short one)
constexpr int kEmNT = 256;
constexpr int kEmRows = 32;     // rows per CTA of the emission
constexpr int kEmQ = 4;         // places per thread whose loads are in flight together

// Warps take four rows (CSR) or columns (CSC) at a time, eight lanes each (a
// long one by the whole warp), and, after them, kCkK x 32 consecutive
// incidences, whose rows are found by search.  `map` null: validated before,
// only the rows of size >= smin are marked.
__global__ __launch_bounds__(kCkNT) void k_small_check(Side s, int32_t smin,
                                                       int32_t *__restrict__ map,
                                                       uint32_t *__restrict__ active, Meta *meta) {
  const int lane = threadIdx.x & 31, sub = lane >> 3, l8 = lane & 7;
  const int64_t warp = ((int64_t)blockIdx.x * kCkNT + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * kCkNT) >> 5;
  if (warp == 0 && lane == 0) {
    if (s.r_off[0] != 0 || (int64_t)s.r_off[s.R] != s.nnz)
      raise_error(meta, SLG_ERR_INVALID, kWhereRowOffsets);
    if (s.c_off[0] != 0 || (int64_t)s.c_off[s.C] != s.nnz)
      raise_error(meta, SLG_ERR_INVALID, kWhereColOffsets);
  }
  const int64_t gr = ((int64_t)s.R + 3) / 4, gc = map ? ((int64_t)s.C + 3) / 4 : 0;
  const int64_t gk = map ? (s.nnz + 32 * kCkK - 1) / (32 * kCkK) : 0;
  for (int64_t x = warp; x < gr + gc + gk; x += nwarps) {
    bool bad = false;
    if (x < gr + gc) {
      const bool row = x < gr;
      const int32_t n = row ? s.R : s.C, ids = row ? s.C : s.R;
      const int64_t r = 4 * (row ? x : x - gr) + sub;
      const int32_t *off = row ? s.r_off : s.c_off, *idx = row ? s.r_idx : s.c_idx;
      int32_t lo = 0, hi = 0;
      if (r < n) {
        lo = __ldg(off + r);
        hi = __ldg(off + r + 1);
        if (lo < 0 || hi < lo || (int64_t)hi > s.nnz) {
          if (l8 == 0)
            raise_error(meta, SLG_ERR_INVALID, row ? kWhereRowOffsets : kWhereColOffsets);
          lo = hi = 0;
        } else if (row && l8 == 0 && hi - lo >= smin) {
          atomicOr(active + (r >> 5), 1u << (r & 31));
        }
      }
      if (!map) continue;
      auto check = [&](uint32_t a, uint32_t b, uint32_t k0, uint32_t step) {
        for (; k0 < b; k0 += 4 * step) {
          int32_t v[4], p[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const uint32_t k = k0 + u * step;
            v[u] = k < b ? __ldg(idx + k) : 0;
            p[u] = k < b && k > a ? __ldg(idx + k - 1) : -1;
          }
#pragma unroll
          for (int u = 0; u < 4; ++u)
            if (k0 + u * step < b) bad |= v[u] < 0 || v[u] >= ids || p[u] >= v[u];
        }
      };
      const bool big = hi - lo > 128;
      if (!big) check(lo, hi, lo + l8, 8);
      unsigned bigs = __ballot_sync(0xffffffffu, big && l8 == 0);
      while (bigs) {
        const int src = __ffs(bigs) - 1;
        bigs &= bigs - 1;
        const int32_t a = __shfl_sync(0xffffffffu, lo, src), b = __shfl_sync(0xffffffffu, hi, src);
        check(a, b, a + lane, 32);
      }
      if (bad) raise_error(meta, SLG_ERR_INVALID, row ? kWhereRowIds : kWhereColIds);
      continue;
    }
    // (the rows may be invalid still: every position is checked before use)
    const int64_t base = (x - gr - gc) * (32 * kCkK);
#pragma unroll
    for (int u = 0; u < kCkK; ++u) {
      const int64_t k = base + 32 * u + lane;
      if (k >= s.nnz) break;
      int32_t f = 0, hi = s.R;
      while (hi - f > 1) {
        const int32_t mid = f + ((hi - f) >> 1);
        if (__ldg(s.r_off + mid) <= (int32_t)k) f = mid;
        else hi = mid;
      }
      const int32_t v = __ldg(s.r_idx + k);
      int32_t q = -1;
      if (v >= 0 && v < s.C && __ldg(s.r_off + f) <= k && __ldg(s.r_off + f + 1) > k) {
        const int32_t c0 = __ldg(s.c_off + v), c1 = __ldg(s.c_off + v + 1);
        if (c0 >= 0 && c1 >= c0 && (int64_t)c1 <= s.nnz) q = find_sorted(s.c_idx, c0, c1, f);
      }
      if (q < 0) bad = true;
      else map[k] = q;
    }
    if (bad) raise_error(meta, SLG_ERR_INVALID, kWhereMismatch);
  }
}

struct SmallWalk {
  Side s;
  int32_t smin;               // threshold
  int32_t row_begin, row_end;
  const int32_t *map;         // CSC position of every CSR incidence
  const uint32_t *active;     // rows of size >= s (all with SLG_NO_PRUNE)
};

// [counters][survivor bits][active bits][tails NT x 8][ws][s_base][row, work][totals]
template <int LB>
size_t small_smem(int32_t R) {
  const size_t words = ((size_t)R + 31) / 32;
  const size_t cnt = (((size_t)R << LB) / 8 + 16) & ~(size_t)15;
  return cnt + ((2 * words + 3) & ~(size_t)3) * 4 + kSwNT * 8 + 16 * 4 + 32 + 9 * 8;
}

// LB: log2 of the counter width (4: rows of at most 65,535 vertices, 5).
template <int LB>
__global__ __launch_bounds__(kSwNT) void k_small_walk(SmallWalk w, EmitArgs a) {
  Meta *meta = a.meta;
  if (meta->err) return;
  constexpr int LW = 5 - LB;
  extern __shared__ __align__(16) unsigned char smem[];
  const int32_t R = w.s.R, nm = (R + 31) >> 5;
  const int32_t cnt_bytes = (int32_t)(((((size_t)R << LB) / 8) + 16) & ~(size_t)15);
  uint32_t *cnt = reinterpret_cast<uint32_t *>(smem);
  uint32_t *map = reinterpret_cast<uint32_t *>(smem + cnt_bytes);
  uint32_t *act = map + nm;
  int2 *s_tail = reinterpret_cast<int2 *>(map + ((2 * nm + 3) & ~3));
  int32_t *ws = reinterpret_cast<int32_t *>(s_tail + kSwNT);
  long long *s_base = reinterpret_cast<long long *>(ws + 16);
  int32_t *s_row = reinterpret_cast<int32_t *>(s_base + 1);  // [0] next row, [1] work
  // totals per bin (rows of <= 128, <= 1,024 and more wedges): rows, wedges, incidences
  unsigned long long *s_stat = reinterpret_cast<unsigned long long *>(s_base + 4);
  const int32_t tid = (int32_t)threadIdx.x, lane = tid & 31, wq = tid >> 5;
  for (int32_t i = tid; i < cnt_bytes / 16; i += kSwNT)
    reinterpret_cast<uint4 *>(cnt)[i] = make_uint4(0, 0, 0, 0);
  for (int32_t i = tid; i < nm; i += kSwNT) {
    map[i] = 0;
    act[i] = w.active[i];
  }
  if (tid < 9) s_stat[tid] = 0;
  const bool emit = a.mode != kCount;
  const bool unweighted = a.unweighted != 0;
  const uint32_t smin = (uint32_t)w.smin;
  int32_t max_work = 0;
  for (int32_t e = w.row_begin + (int32_t)blockIdx.x; e < w.row_end;) {
    if (tid == 0) {
      // the next row's ticket, fetched while this one is counted
      s_row[0] = w.row_begin + (int32_t)gridDim.x + (int32_t)atomicAdd(&meta->giant_ticket, 1u);
      s_row[1] = 0;
    }
    __syncthreads();  // (also: the counters and bits are clear)
    const int32_t next = s_row[0];
    if (!((act[e >> 5] >> (e & 31)) & 1u)) {  // uniform
      __syncthreads();  // `next` is read
      e = next;
      continue;
    }
    const int32_t k0 = w.s.r_off[e], k1 = w.s.r_off[e + 1];
    int32_t wedges = 0, c = 0;
    auto count = [&](int32_t f) {
      if (!((act[f >> 5] >> (f & 31)) & 1u)) return;
      ++wedges;
      const int sh = (f & ((1 << LW) - 1)) << LB;
      uint32_t old = atomicAdd(cnt + (f >> LW), 1u << sh);
      if (LB < 5) old = (old >> sh) & 0xFFFFu;
      if (old + 1 == smin) {
        if (emit) atomicOr(map + (f >> 5), 1u << (f & 31));
        else ++c;
      }
    };
    for (int32_t base = k0; base < k1; base += kSwNT) {
      // a batch of tails, then their entries: short tails by eight lanes, four
      // in flight, long ones by whole warps
      if (base > k0) __syncthreads();  // the batch before is read
      const int32_t k = base + tid;
      int2 tail = make_int2(0, 0);
      if (k < k1)
        tail = make_int2(__ldg(w.map + k) + 1, __ldg(w.s.c_off + __ldg(w.s.r_idx + k) + 1));
      s_tail[tid] = tail;
      __syncthreads();
      const int32_t n = min(kSwNT, k1 - base);
      const int l8 = lane & 7;
      for (int32_t x0 = tid >> 3; x0 < n; x0 += 4 * (kSwNT / 8)) {
        uint2 t[4];  // (unsigned: a place may lie beyond 2^31)
        int32_t f[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int32_t x = x0 + u * (kSwNT / 8);
          const int2 tail = x < n ? s_tail[x] : make_int2(0, 0);
          t[u] = make_uint2(tail.x, tail.y - tail.x > kSwLongMin ? tail.x : tail.y);
          f[u] = t[u].x + l8 < t[u].y ? __ldg(w.s.c_idx + t[u].x + l8) : -1;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          if (f[u] >= 0) count(f[u]);
          for (uint32_t i = t[u].x + l8 + 8; i < t[u].y; i += 8) count(__ldg(w.s.c_idx + i));
        }
      }
      for (int32_t x = wq; x < n; x += kSwNW) {
        const int2 t = s_tail[x];
        if (t.y - t.x <= kSwLongMin) continue;
        const uint32_t end = (uint32_t)t.y;
        for (uint32_t i = (uint32_t)t.x + lane; i < end; i += 128) {
          int32_t f[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) f[u] = i + 32 * u < end ? __ldg(w.s.c_idx + i + 32 * u) : -1;
#pragma unroll
          for (int u = 0; u < 4; ++u)
            if (f[u] >= 0) count(f[u]);
        }
      }
    }
    const int32_t ww = __reduce_add_sync(0xffffffffu, wedges);
    if (lane == 0 && ww) atomicAdd(s_row + 1, ww);
    __syncthreads();  // counts final
    const int32_t work = s_row[1];
    if (tid == 0 && work) {
      const int b = work <= kWarpMaxWork ? 0 : work <= kCtaSMaxWork ? 1 : 2;
      s_stat[3 * b] += 1;
      s_stat[3 * b + 1] += (unsigned long long)work;
      s_stat[3 * b + 2] += (unsigned long long)(k1 - k0);
      max_work = max(max_work, work);
    }
    if (work) {  // uniform
      // survivors: a thread owns consecutive words of the bits
      const int32_t wpt = (nm + kSwNT - 1) / kSwNT;
      const int32_t m0 = min(tid * wpt, nm), m1 = min(m0 + wpt, nm);
      if (emit)
        for (int32_t x = m0; x < m1; ++x) c += __popc(map[x]);
      int32_t total;
      const int32_t inc = block_inclusive_scan<kSwNT>(c, ws, &total);
      if (tid == 0 && total)
        *s_base = reserve(a, e, total,
                          work <= kWarpMaxWork ? kBinWarp : work <= kCtaSMaxWork ? kBinCtaS : kBinGiant);
      __syncthreads();
      const long long base = total ? *s_base : -1;
      if (emit)
        for_survivors(map, m0, m1, inc - c, total > kSurvDense * nm, [&](int32_t t, int32_t f) {
          const uint32_t word = cnt[f >> LW];
          const int32_t n = LB < 5 ? (int32_t)((word >> ((f & ((1 << LW) - 1)) << LB)) & 0xFFFFu)
                                   : (int32_t)word;
          if (base >= 0) put(a, base, t, e, f, unweighted ? 0 : n);
        });
      __syncthreads();  // the counters are read
      // far ends lie above e
      for (int32_t i = ((e >> LW) >> 2) + tid; i < cnt_bytes / 16; i += kSwNT)
        reinterpret_cast<uint4 *>(cnt)[i] = make_uint4(0, 0, 0, 0);
    } else {
      __syncthreads();  // the row's work is read
    }
    e = next;
  }
  __syncthreads();
  if (tid == 0) {
    const int bins[3] = {kBinWarp, kBinCtaS, kBinGiant};
    for (int b = 0; b < 3; ++b) {
      if (!s_stat[3 * b]) continue;
      atomicAdd(&meta->rows_bin[bins[b]], s_stat[3 * b]);
      atomicAdd(&meta->wedges_bin[bins[b]], s_stat[3 * b + 1]);
      atomicAdd(&meta->incid_bin[bins[b]], s_stat[3 * b + 2]);
      atomicAdd(&meta->wedges, s_stat[3 * b + 1]);
    }
    if (max_work) atomicMax(&meta->max_row_work, max_work);
  }
}

// A CTA owns kEmRows consecutive rows of the range: their places (the sum of
// the pair counts before them, taken by each CTA for itself), then their
// staged pairs.  The last CTA to finish copies the totals to the host.
__global__ __launch_bounds__(kEmNT) void k_small_emit(int32_t row_begin, int32_t rows,
                                                      const int32_t *__restrict__ n_e,
                                                      const uint32_t *__restrict__ active,
                                                      const long long *__restrict__ stage_pos,
                                                      const int32_t *__restrict__ stage_j,
                                                      const int32_t *__restrict__ stage_w,
                                                      int32_t *__restrict__ out_i,
                                                      int32_t *__restrict__ out_j,
                                                      int32_t *__restrict__ out_w, int unweighted,
                                                      long long *__restrict__ row_ptr,
                                                      long long out_cap, Meta *meta,
                                                      volatile uint32_t *host) {
  __shared__ long long ws[kEmNT / 32 + 1];
  __shared__ long long s_ptr[kEmRows + 1];
  __shared__ long long s_sp[kEmRows];
  __shared__ bool s_last;
  const int32_t tid = (int32_t)threadIdx.x;
  const int32_t r0 = (int32_t)blockIdx.x * kEmRows, nr = min(kEmRows, rows - r0);
  if (!meta->err) {
    long long before = 0, first;
    for (int32_t r = tid; r < r0; r += 4 * kEmNT) {
      int32_t x[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) x[u] = r + u * kEmNT < r0 ? __ldg(n_e + r + u * kEmNT) : 0;
      before += (long long)x[0] + x[1] + x[2] + x[3];
    }
    block_inclusive_scan64<kEmNT>(before, ws, &first);
    if (tid < 32) {
      const int32_t e = row_begin + r0 + tid;
      const long long x = tid < nr ? __ldg(n_e + r0 + tid) : 0;
      const long long inc = warp_inclusive_scan64(x);
      if (tid == 0) s_ptr[0] = first;
      s_ptr[tid + 1] = first + inc;
      s_sp[tid] = x > 0 && stage_j ? stage_pos[r0 + tid] : -1;
      const unsigned act =
          __ballot_sync(0xffffffffu, tid < nr && ((active[e >> 5] >> (e & 31)) & 1u));
      if (tid == 0 && act) atomicAdd(&meta->active, (unsigned long long)__popc(act));
      if (row_ptr && tid < nr) row_ptr[r0 + tid] = first + inc - x;
      if (tid == 31 && r0 + kEmRows >= rows) {  // the last rows
        if (row_ptr) row_ptr[rows] = first + inc;
        meta->pairs = (unsigned long long)(first + inc);
      }
    }
    __syncthreads();
    const long long end = s_ptr[kEmRows];
    if (stage_j) {
      int lo = 0;  // s_ptr[lo] <= p for every p still to come
      for (long long p0 = first + tid; p0 < end; p0 += kEmQ * kEmNT) {
        long long src[kEmQ];
        int row[kEmQ];
#pragma unroll
        for (int u = 0; u < kEmQ; ++u) {
          const long long p = p0 + u * kEmNT;
          src[u] = -1;
          row[u] = lo;
          if (p < end && p < out_cap) {  // (beyond: the call returns the capacity error)
            while (s_ptr[lo + 1] <= p) ++lo;
            row[u] = lo;
            if (s_sp[lo] >= 0) src[u] = s_sp[lo] + (p - s_ptr[lo]);
          }
        }
        int32_t vj[kEmQ], vw[kEmQ];
#pragma unroll
        for (int u = 0; u < kEmQ; ++u) {
          vj[u] = src[u] >= 0 ? stage_j[src[u]] : 0;
          vw[u] = src[u] >= 0 && !unweighted ? stage_w[src[u]] : 0;
        }
#pragma unroll
        for (int u = 0; u < kEmQ; ++u) {
          const long long p = p0 + u * kEmNT;
          if (src[u] < 0) continue;
          if (out_i) out_i[p] = row_begin + r0 + row[u];
          out_j[p] = vj[u];
          if (!unweighted) out_w[p] = vw[u];
        }
      }
    }
  }
  __threadfence();
  __syncthreads();
  if (tid == 0) s_last = atomicAdd(&meta->giant_huge, 1u) == gridDim.x - 1;
  __syncthreads();
  if (s_last) {
    __threadfence();
    const volatile uint32_t *src = reinterpret_cast<const volatile uint32_t *>(meta);
    for (int i = tid; i < (int)(sizeof(Meta) / 4); i += kEmNT) host[i] = src[i];
  }
}

int small_ctas(int lb, int32_t R, size_t *smem) {
  struct Occ {
    int dev = -1, sms = 0;
  };
  static Occ occ[64];
  static std::mutex mu;
  int dev = 0;
  cudaGetDevice(&dev);
  Occ &o = occ[dev & 63];
  {
    std::lock_guard<std::mutex> lock(mu);
    if (o.dev != dev) {
      cudaDeviceGetAttribute(&o.sms, cudaDevAttrMultiProcessorCount, dev);
      cudaFuncSetAttribute(k_small_walk<4>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)small_smem<4>(kSmallRows));
      cudaFuncSetAttribute(k_small_walk<5>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)small_smem<5>(kSmallRows));
      o.dev = dev;
    }
  }
  *smem = lb == 4 ? small_smem<4>(R) : small_smem<5>(R);
  // shared memory or 8 CTAs of 256 threads limit the residency
  const int per = (int)std::min<size_t>(8, (size_t)220 * 1024 / (*smem + 1024));
  return o.sms * std::max(per, 1);
}

// Places and totals, and (emit) the pairs.
cudaError_t small_emit(const SmallCall &c, bool emit, cudaStream_t st, int32_t *launches) {
  const int32_t rows = c.row_end - c.row_begin;
  const int grid = std::max((rows + kEmRows - 1) / kEmRows, 1);
  k_small_emit<<<grid, kEmNT, 0, st>>>(c.row_begin, rows, c.a.n_e, c.active, c.a.stage_pos,
                                       emit ? c.a.stage_j : nullptr, c.a.stage_w, c.out_i, c.out_j,
                                       c.out_w, c.a.unweighted, c.row_ptr, c.a.stage_cap, c.a.meta,
                                       reinterpret_cast<volatile uint32_t *>(c.host));
  ++*launches;
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_small(const SmallCall &c, cudaStream_t st, int32_t *launches, cudaEvent_t walk0,
                         cudaEvent_t walk1) {
  const int64_t warps = (int64_t)c.s.R / 4 + 1 +
                        (c.validate ? c.s.C / 4 + 1 + c.s.nnz / (32 * kCkK) + 1 : 0);
  const int64_t blocks = std::max<int64_t>((warps * 32 + kCkNT - 1) / kCkNT, 1);
  k_small_check<<<(int)std::min<int64_t>(blocks, 152 * 16), kCkNT, 0, st>>>(
      c.s, c.s_prune, c.validate ? c.map : nullptr, c.active, c.a.meta);
  ++*launches;
  if (walk0) cudaEventRecord(walk0, st);
  const int32_t rows = c.row_end - c.row_begin;
  if (rows > 0 && c.s.nnz > 0) {
    const int lb = std::min<int64_t>(c.s.C, c.s.nnz) <= 65535 ? 4 : 5;
    size_t smem = 0;
    const int ctas = std::min(small_ctas(lb, c.s.R, &smem), rows);
    SmallWalk w = {c.s, c.a.smin, c.row_begin, c.row_end, c.map, c.active};
    if (lb == 4) k_small_walk<4><<<ctas, kSwNT, smem, st>>>(w, c.a);
    else k_small_walk<5><<<ctas, kSwNT, smem, st>>>(w, c.a);
    ++*launches;
  }
  if (walk1) cudaEventRecord(walk1, st);
  return small_emit(c, !c.hold && c.a.mode != kCount, st, launches);
}

// The emission of a held call, once its outputs are there.
cudaError_t launch_small_emit(const SmallCall &c, cudaStream_t st, int32_t *launches) {
  return small_emit(c, true, st, launches);
}

}  // namespace slg
