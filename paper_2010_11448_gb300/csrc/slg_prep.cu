// Planning kernels of the s-overlap walk: input validation, the CSR->CSC
// position map, the CSC filtered by hyperedge size (degree-based pruning,
// Section IV-C: a hyperedge with |e| < s can be in no pair of L_s), the tail
// of every incidence (strict upper triangle, Section IV-C), and the binning of
// rows by wedge work (the GPU counterpart of the load balancing of
// Section IV-F).
#include <algorithm>

#include "slg_internal.cuh"

namespace slg {

namespace {

constexpr int kValNT = 256;

// Sides whose longest row matters to the map (k_csr2csc): k_validate notes it for
// these only, since a maximum over all warps costs it 10 us.
__host__ __device__ __forceinline__ bool long_rows(const Side &s) {
  return s.nnz >= 128ll * s.R;
}

// Offsets monotone inside [0, nnz], ids inside [0, cols), every row strictly
// ascending.  Eight lanes per row (rows hold 10 to 20 ids on average; a warp
// per row left two thirds of its lanes idle: 257 us for both sides of 500K x
// 1M, where this takes 123); a row of more than kValLong ids is read by the
// whole warp, four loads in flight.  Reports through meta (never traps).
constexpr int32_t kValLong = 128;

__global__ __launch_bounds__(kValNT) void k_validate(const int32_t *__restrict__ off,
                                                     const int32_t *__restrict__ idx,
                                                     int32_t rows, int32_t cols, int64_t nnz,
                                                     Meta *meta, int32_t where_off,
                                                     int32_t where_ids,
                                                     int32_t *longest) {
  const int lane = threadIdx.x & 31, sub = lane >> 3, l8 = lane & 7;
  const int64_t warp = ((int64_t)blockIdx.x * kValNT + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * kValNT) >> 5;
  if (warp == 0 && lane == 0) {
    if (off[0] != 0 || (int64_t)off[rows] != nnz) raise_error(meta, SLG_ERR_INVALID, where_off);
  }
  bool bad = false;
  int32_t most = 0;
  // ids k, k + step, ... of the row [lo, hi)
  // (unsigned: the last of the four may lie beyond 2^31)
  auto check = [&](uint32_t lo, uint32_t hi, uint32_t k0, uint32_t step) {
    for (; k0 < hi; k0 += 4 * step) {
      int32_t x[4], y[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const uint32_t k = k0 + u * step;
        x[u] = k < hi ? __ldg(idx + k) : 0;
        y[u] = k < hi && k > lo ? __ldg(idx + k - 1) : -1;
      }
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (k0 + u * step < hi) bad |= x[u] < 0 || x[u] >= cols || y[u] >= x[u];
    }
  };
  for (int64_t r0 = warp * 4; r0 < rows; r0 += nwarps * 4) {
    const int64_t r = r0 + sub;
    int32_t lo = 0, hi = 0;
    if (r < rows) {
      lo = __ldg(off + r);
      hi = __ldg(off + r + 1);
      if (lo < 0 || hi < lo || (int64_t)hi > nnz) {
        if (l8 == 0) raise_error(meta, SLG_ERR_INVALID, where_off);
        lo = hi = 0;
      }
    }
    most = max(most, hi - lo);
    if (hi - lo <= kValLong) check(lo, hi, lo + l8, 8);
    unsigned big = __ballot_sync(0xffffffffu, l8 == 0 && hi - lo > kValLong);
    while (big) {
      const int src = __ffs(big) - 1;
      big &= big - 1;
      const int32_t a = __shfl_sync(0xffffffffu, lo, src), b = __shfl_sync(0xffffffffu, hi, src);
      check(a, b, a + lane, 32);
    }
  }
  if (bad) raise_error(meta, SLG_ERR_INVALID, where_ids);
  if (longest) {
    most = __reduce_max_sync(0xffffffffu, most);
    if (lane == 0 && most > *(volatile int32_t *)longest) atomicMax(longest, most);
  }
}

// The CSC position of every incidence (v, f), found by binary search in the
// (validated, ascending) column v.  A miss means the CSR and CSC are not the
// same incidence.  With nnz equal on both sides and strictly ascending rows, a
// hit for every incidence makes the map a bijection.
// Incidences are dealt out evenly (a warp takes kMapK x 32 consecutive ones
// and finds their rows): with a warp per row, the kernel's time was that of
// its longest row (10,000 vertices, 312 dependent searches: 887 us on 500K x
// 1M, where this takes 211).  Where no row lasts that long beside the whole and
// the rows are long (all alike, mostly), a warp takes a row: all warps then pass
// through the column ids at the same pace and share their sectors (200K rows of 800
// of 30M columns 2.7 instead of 5.7 ms, 100K of 3,000 of 60M 4.0 instead of 11.8).
constexpr int kMapK = 8;
constexpr int64_t kMapRowShare = 5'000;   // incidences per vertex of the longest row
__global__ __launch_bounds__(kValNT) void k_csr2csc(Side s, int32_t *__restrict__ csr2csc,
                                                    Meta *meta) {
  if (meta->err) return;
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * kValNT + threadIdx.x) >> 5;
  if (long_rows(s) && meta->longest_row * kMapRowShare <= s.nnz) {
    const int64_t nwarps = ((int64_t)gridDim.x * kValNT) >> 5;
    bool bad = false;
    for (int64_t f = warp; f < s.R; f += nwarps) {
      const int32_t lo = s.r_off[f], hi = s.r_off[f + 1];
      for (int64_t k = (int64_t)lo + lane; k < hi; k += 32) {
        const int32_t v = s.r_idx[k];
        const int32_t q = find_sorted(s.c_idx, s.c_off[v], s.c_off[v + 1], (int32_t)f);
        if (q < 0) bad = true;
        else csr2csc[k] = q;
      }
    }
    if (bad) raise_error(meta, SLG_ERR_INVALID, kWhereMismatch);
    return;
  }
  const int64_t base = warp * (32 * kMapK);
  if (base >= s.nnz) return;
  int32_t f = 0;
  {
    int32_t hi = s.R;  // r_off[f] <= base < r_off[hi]
    while (hi - f > 1) {
      const int32_t mid = f + ((hi - f) >> 1);
      if (__ldg(s.r_off + mid) <= (int32_t)base) f = mid;
      else hi = mid;
    }
  }
  bool bad = false;
#pragma unroll 2
  for (int u = 0; u < kMapK; ++u) {
    const int64_t k = base + 32 * u + lane;
    if (k >= s.nnz) break;
    const int32_t v = s.r_idx[k];
    f = row_of(s.r_off, s.R, f, (int32_t)k);
    const int32_t q = find_sorted(s.c_idx, s.c_off[v], s.c_off[v + 1], f);
    if (q < 0) bad = true;
    else csr2csc[k] = q;
  }
  if (bad) raise_error(meta, SLG_ERR_INVALID, kWhereMismatch);
}

// ------------------------------------------ filtered CSC (reduce-then-scan) --

constexpr int kScanNT = 256;
constexpr int kScanIPT = 16;                    // items per thread
constexpr int kScanTile = kScanNT * kScanIPT;   // 4096 CSC entries per tile

__device__ __forceinline__ int32_t kept(const Side &s, int32_t q, int32_t smin) {
  const int32_t f = __ldg(s.c_idx + q);
  return (__ldg(s.r_off + f + 1) - __ldg(s.r_off + f)) >= s_of(s.row_s, smin, f);
}

__global__ __launch_bounds__(kScanNT) void k_filter_reduce(Side s, int32_t smin,
                                                           int32_t *__restrict__ tile,
                                                           const Meta *meta) {
  if (meta->err) return;
  __shared__ int32_t ws[kScanNT / 32 + 1];
  const int64_t base = (int64_t)blockIdx.x * kScanTile;
  int32_t c = 0;
#pragma unroll 4
  for (int i = 0; i < kScanIPT; ++i) {
    const int64_t q = base + (int64_t)i * kScanNT + threadIdx.x;
    if (q < s.nnz) c += kept(s, (int32_t)q, smin);
  }
  int32_t total;
  block_inclusive_scan<kScanNT>(c, ws, &total);
  if (threadIdx.x == 0) tile[blockIdx.x] = total;
}

// Exclusive scan of n int32 tile sums in place (one CTA); writes the grand
// total to tile[n] and, if given, to *total_out.
__global__ __launch_bounds__(1024) void k_scan_tiles(int32_t *tile, int32_t n,
                                                     int32_t *total_out, const Meta *meta) {
  if (meta->err) return;
  __shared__ int32_t ws[1024 / 32 + 1];
  __shared__ int32_t carry;
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  for (int32_t base = 0; base < n; base += 1024) {
    const int32_t i = base + threadIdx.x;
    const int32_t x = i < n ? tile[i] : 0;
    int32_t total;
    const int32_t inc = block_inclusive_scan<1024>(x, ws, &total);
    if (i < n) tile[i] = carry + inc - x;
    __syncthreads();
    if (threadIdx.x == 0) carry += total;
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    tile[n] = carry;
    if (total_out) *total_out = carry;
  }
}

// Per tile: qs[q] = number of kept entries before q; kept entries are copied
// to their place in the filtered CSC.  Items are strided by kScanNT inside
// the tile so reads stay coalesced; the scan order is item-major.
__global__ __launch_bounds__(kScanNT) void k_filter_scatter(Side s, int32_t smin,
                                                            const int32_t *__restrict__ tile,
                                                            int32_t *__restrict__ qs,
                                                            int32_t *__restrict__ c_idx_s,
                                                            const Meta *meta) {
  if (meta->err) return;
  __shared__ int32_t ws[kScanNT / 32 + 1];
  const int64_t base = (int64_t)blockIdx.x * kScanTile;
  int32_t carry = tile[blockIdx.x];
  for (int i = 0; i < kScanIPT; ++i) {
    const int64_t q = base + (int64_t)i * kScanNT + threadIdx.x;
    int32_t k = 0, f = 0;
    if (q < s.nnz) {
      f = __ldg(s.c_idx + q);
      k = (__ldg(s.r_off + f + 1) - __ldg(s.r_off + f)) >= s_of(s.row_s, smin, f);
    }
    int32_t total;
    const int32_t inc = block_inclusive_scan<kScanNT>(k, ws, &total);
    if (q < s.nnz) {
      const int32_t pos = carry + inc - k;
      qs[q] = pos;
      if (k) c_idx_s[pos] = f;
    }
    carry += total;
  }
}

__global__ void k_filter_offsets(Side s, const int32_t *__restrict__ qs,
                                 const int32_t *__restrict__ tile, int32_t ntiles,
                                 int32_t *__restrict__ c_off_s, const Meta *meta) {
  if (meta->err) return;
  const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (c > s.C) return;
  const int32_t q = s.c_off[c];
  c_off_s[c] = q < s.nnz ? qs[q] : tile[ntiles];
}

// ---------------------------------------------------- tails, work, bins --

constexpr int kRowsNT = 256;
constexpr int kRowsPerBlock = 64;

__device__ __forceinline__ int bin_of(int32_t work, const Bins &b) {
  if (work <= b.warp) return kBinWarp;
  if (work <= b.ctas) return kBinCtaS;
  if (work <= b.ctal) return kBinCtaL;
  return kBinGiant;
}

// The tail of every incidence (e, v): the filtered position of e in column v
// is qs[csr2csc[k]], so its tail starts one past it (for a row of size < s,
// which is not kept, nothing reads the tail).  Incidences are dealt out evenly,
// as in k_csr2csc.
__global__ __launch_bounds__(kRowsNT) void k_tails(int64_t k0, int64_t k1,
                                                   const int32_t *__restrict__ r_idx,
                                                   const int32_t *__restrict__ csr2csc,
                                                   const int32_t *__restrict__ qs,
                                                   const int32_t *__restrict__ c_off_s,
                                                   int32_t *__restrict__ tail_beg,
                                                   int32_t *__restrict__ tail_end,
                                                   const Meta *meta) {
  if (meta->err) return;
  const int64_t base = k0 + (int64_t)blockIdx.x * (kRowsNT * 4) + threadIdx.x;
  int32_t v[4], q[4], tb[4], te[4];
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int64_t k = base + u * kRowsNT;
    v[u] = k < k1 ? __ldg(r_idx + k) : 0;
    q[u] = k < k1 ? __ldg(csr2csc + k) : 0;
  }
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    tb[u] = __ldg(qs + q[u]) + 1;
    te[u] = __ldg(c_off_s + v[u] + 1);
  }
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int64_t k = base + u * kRowsNT;
    if (k < k1) {
      tail_beg[k] = tb[u];
      tail_end[k] = te[u];
    }
  }
}

// A block handles kRowsPerBlock consecutive rows, eight lanes each (long rows and
// core rows by whole warps).
// The row's work is the sum of its tail lengths (k_tails; core columns of core
// rows are set here).  Rows with
// work > 0 are appended to their bin's list (one global atomic per bin and
// block); rows outside the range or inactive get n_e = 0.
__global__ __launch_bounds__(kRowsNT) void k_rows_work(Side s, int32_t smin, int32_t row_begin,
                                                       int32_t row_end,
                                                       const int32_t *__restrict__ c_idx_s,
                                                       CoreInfo core, Bins bins,
                                                       int32_t *tail_beg,
                                                       int32_t *tail_end,
                                                       int32_t *__restrict__ n_e,
                                                       long long *__restrict__ stage_pos,
                                                       int32_t *__restrict__ row_work,
                                                       int32_t *__restrict__ bin_rows,
                                                       Meta *meta) {
  if (meta->err) return;
  __shared__ int32_t s_work[kRowsPerBlock], s_longest[kRowsPerBlock];  // wedges, longest tail
  // block maxima of the row work (all rows, giant-bin, sparse- or flat-bin, the dense
  // bin's two instances' rows) and size (dense-bin rows, all rows), and a plan's bounds: one
  // global atomicMax each per
  // block instead of one per row
  __shared__ int32_t s_max[10];
  __shared__ int32_t s_act;  // active rows (size >= s) of the block
  __shared__ int32_t s_cnt[kNumLists], s_base[kNumLists];
  __shared__ int32_t s_hcnt[4], s_hbase[4];  // giant / sparse / dense / flat rows handed out first
  __shared__ unsigned long long s_w[kNumLists], s_k[kNumLists];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int32_t r0 = row_begin + blockIdx.x * kRowsPerBlock;
  if (threadIdx.x < kNumLists) {
    s_cnt[threadIdx.x] = 0;
    s_w[threadIdx.x] = 0;
    s_k[threadIdx.x] = 0;
  }
  if (threadIdx.x < 4) s_hcnt[threadIdx.x] = 0;
  if (threadIdx.x < 10) s_max[threadIdx.x] = 0;
  if (threadIdx.x == 0) s_act = 0;
  __syncthreads();
  // eight lanes per row; long rows and core rows by the whole warp
  for (int i0 = warp * 4; i0 < kRowsPerBlock; i0 += kRowsNT / 8) {
    const int i = i0 + (lane >> 3), l8 = lane & 7;
    const int32_t e = r0 + i;
    int32_t work = 0, longest = 0, lo = 0, hi = 0;
    bool active = false, core_row = false;
    if (e < row_end) {
      lo = __ldg(s.r_off + e);
      hi = __ldg(s.r_off + e + 1);
      active = hi - lo >= s_of(s.row_s, smin, e);
      core_row = core.row_rank && core.row_rank[e + 1] != core.row_rank[e];
    }
    // tail lengths of incidences k0, k0 + step, ... of [.., b): their sum, the longest
    auto sum = [&](uint32_t k0, uint32_t b, uint32_t step) {
      int32_t n = 0;
      for (; k0 < b; k0 += 4 * step) {
        int32_t tb[4], te[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const uint32_t k = k0 + u * step;
          tb[u] = k < b ? tail_beg[k] : 0;
          te[u] = k < b ? tail_end[k] : 0;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          n += te[u] - tb[u];
          longest = max(longest, te[u] - tb[u]);
        }
      }
      return n;
    };
    const bool whole = active && (core_row || hi - lo > kValLong);
    if (active && !whole) work = sum(lo + l8, hi, 8);
#pragma unroll
    for (int d = 4; d > 0; d >>= 1) {
      work += __shfl_xor_sync(0xffffffffu, work, d);
      longest = max(longest, __shfl_xor_sync(0xffffffffu, longest, d));
    }
    unsigned big = __ballot_sync(0xffffffffu, l8 == 0 && whole);
    while (big) {
      const int src = __ffs(big) - 1;
      big &= big - 1;
      const int32_t x = __shfl_sync(0xffffffffu, e, src);
      const int32_t a = __shfl_sync(0xffffffffu, lo, src), b = __shfl_sync(0xffffffffu, hi, src);
      int32_t n = 0;
      const int32_t own = longest;  // of this lane's own row
      longest = 0;
      if (!__shfl_sync(0xffffffffu, (int)core_row, src)) {
        n = sum(a + lane, b, 32);
      } else {
        for (int32_t k = a + lane; k < b; k += 32) {
          const int32_t v = s.r_idx[k];
          if (core.col_rank[v + 1] != core.col_rank[v]) {
            // core row at a core column: its tail skips the core rows (their
            // shared core vertices are counted on the tensor cores)
            const int32_t cv = core.col_rank[v];
            int32_t p = core.x_base + core.x_off[cv], q = core.x_base + core.x_off[cv + 1];
            tail_end[k] = q;
            while (p < q) {  // first entry > x
              const int32_t mid = (p + q) >> 1;
              if (c_idx_s[mid] <= x) p = mid + 1;
              else q = mid;
            }
            tail_beg[k] = p;
          }
          n += tail_end[k] - tail_beg[k];
        }
      }
      n = __reduce_add_sync(0xffffffffu, n);
      const int32_t most = __reduce_max_sync(0xffffffffu, longest);
      longest = own;
      if ((lane & 24) == (src & 24)) {
        work = n;
        longest = most;
      }
    }
    if (l8 == 0) {
      if (e < row_end) {
        n_e[e - row_begin] = 0;
        stage_pos[e - row_begin] = -1;
        row_work[e - row_begin] = work;
        if (work) {
          atomicMax(&s_max[0], work);
          atomicMax(&s_max[5], hi - lo);
        }
        if (active) atomicAdd(&s_act, 1);
      }
      // core rows take part even without wedges (their tile counts are added
      // by the bin), marked by a negative work entry here
      s_work[i] = e < row_end ? (core_row && active ? -1 - work : work) : 0;
      s_longest[i] = longest;
    }
  }
  __syncthreads();
  int my_bin = -1, my_slot = 0;
  bool huge = false;
  int32_t my_work = 0;
  if (threadIdx.x < kRowsPerBlock) {
    my_work = s_work[threadIdx.x];
    const bool forced = my_work < 0;
    if (forced) my_work = -1 - my_work;
    if (my_work > 0 || forced) {
      const int32_t e = r0 + threadIdx.x;
      my_bin = forced ? (int)kBinGiant : bin_of(my_work, bins);
      const int32_t size = s.r_off[e + 1] - s.r_off[e];
      const int32_t se = s_of(s.row_s, smin, e);
      const int32_t span = (s.row_fhi ? s.row_fhi[e] : s.R) - 1 - e;  // far ends: (e, e + span]
      // a row whose far ends are dense in its span takes the dense bin; else
      // one with s >= 2 from bins.bloom up to bins.sparse wedges the sparse or
      // the flat bin
      const bool sparse = !forced && my_work > bins.bloom && my_work <= bins.sparse && se >= 2;
      if ((forced || my_work > kDenseMinWork) && is_dense(my_work, size, se, span, bins.dense, forced))
        my_bin = kBinDense;
      else if (!forced && my_work > bins.bloom && my_work <= bins.sparse && se >= 2) {
        if (!bins.flat || !short_tails(my_work, size, s_longest[threadIdx.x])) my_bin = kBinSparse;
        else if (my_work <= kFlatMaxWork) my_bin = kBinFlat;
      }
      else if (!forced && my_work <= bins.ctas && se >= 2)
        my_bin = size <= kRowsMaxSize ? kBinRows : kBinCtaS;
      if (s.row_s) {
        if (my_work > kDenseMinWork)
          atomicMax(&s_max[size > kDenseBigSize ? 7 : 8], max(my_work / se, 1));
        if (se >= 2 && my_work <= kSparseMaxWork) atomicMax(&s_max[9], my_work);
      }
      if (my_bin == kBinGiant) atomicMax(&s_max[1], my_work);
      if (my_bin == kBinSparse || my_bin == kBinFlat) atomicMax(&s_max[2], my_work);
      if (my_bin == kBinDense) {
        atomicMax(&s_max[size > kDenseBigSize ? 3 : 6], my_work);
        atomicMax(&s_max[4], size);
      }
      huge = (my_bin == kBinDense && size > kDenseBigSize) ||
             (my_bin == kBinGiant && my_work > kGiantHugeWork) ||
             ((my_bin == kBinSparse || my_bin == kBinFlat) && my_work > kSparseBigWork);
      my_slot = huge ? atomicAdd(&s_hcnt[my_bin - kBinGiant], 1) : atomicAdd(&s_cnt[my_bin], 1);
      atomicAdd(&s_w[my_bin], (unsigned long long)my_work);
      atomicAdd(&s_k[my_bin], (unsigned long long)size);
    }
  }
  __syncthreads();
  if (threadIdx.x < kNumLists) {
    const int b = threadIdx.x;
    if (b < kBinGiant || b == kBinRows) {
      s_base[b] = s_cnt[b] ? (int32_t)atomicAdd(&meta->rows_bin[b], (unsigned long long)s_cnt[b]) : 0;
    } else {
      // the huge rows of the giant, sparse, dense and flat bins fill their list from
      // the front, the others from the back (the kernels hand out the huge
      // ones first); rows_bin counts both
      const int q = b - kBinGiant;
      unsigned *rest = q == 0   ? &meta->giant_rest
                       : q == 1 ? &meta->sparse_rest
                       : q == 2 ? &meta->dense_rest
                                : &meta->flat_rest;
      unsigned *hge = q == 0   ? &meta->giant_huge
                      : q == 1 ? &meta->sparse_huge
                      : q == 2 ? &meta->dense_huge
                               : &meta->flat_huge;
      if (s_cnt[b] + s_hcnt[q])
        atomicAdd(&meta->rows_bin[b], (unsigned long long)(s_cnt[b] + s_hcnt[q]));
      s_base[b] = s_cnt[b] ? (int32_t)atomicAdd(rest, (unsigned)s_cnt[b]) : 0;
      s_hbase[q] = s_hcnt[q] ? (int32_t)atomicAdd(hge, (unsigned)s_hcnt[q]) : 0;
    }
    if (s_w[b]) {
      atomicAdd(&meta->wedges_bin[b], s_w[b]);
      atomicAdd(&meta->wedges, s_w[b]);
      atomicAdd(&meta->incid_bin[b], s_k[b]);
    }
  }
  if (threadIdx.x == kNumLists && s_act) atomicAdd(&meta->active, (unsigned long long)s_act);
  __syncthreads();
  if (threadIdx.x == 0) {
    if (s_max[0]) atomicMax(&meta->max_row_work, s_max[0]);
    if (s_max[1]) atomicMax(&meta->max_giant_work, s_max[1]);
    if (s_max[2]) atomicMax(&meta->max_sparse_work, s_max[2]);
    if (s_max[3]) atomicMax(&meta->max_dense_work[0], s_max[3]);
    if (s_max[6]) atomicMax(&meta->max_dense_work[1], s_max[6]);
    if (s_max[4]) atomicMax(&meta->max_dense_size, s_max[4]);
    if (s_max[5]) atomicMax(&meta->max_row_size, s_max[5]);
    if (s_max[7]) atomicMax(&meta->plan_pairs[0], s_max[7]);
    if (s_max[8]) atomicMax(&meta->plan_pairs[1], s_max[8]);
    if (s_max[9]) atomicMax(&meta->plan_sparse, s_max[9]);
  }
  if (my_bin >= 0) {
    const int64_t len = row_end - row_begin;
    int64_t pos = s_base[my_bin] + my_slot;
    if (huge) pos = s_hbase[my_bin - kBinGiant] + my_slot;
    else if (my_bin >= kBinGiant && my_bin != kBinRows) pos = len - 1 - pos;
    bin_rows[(int64_t)my_bin * len + pos] = r0 + threadIdx.x;
  }
}

inline int grid_for(int64_t items, int per_block, int cap = 1 << 20) {
  int64_t g = (items + per_block - 1) / per_block;
  if (g < 1) g = 1;
  if (g > cap) g = cap;
  return (int)g;
}

}  // namespace

cudaError_t launch_validate(const Side &s, Meta *meta, cudaStream_t st) {
  const int wpb = kValNT / 8;  // rows per block
  k_validate<<<grid_for(s.R, wpb, 65536), kValNT, 0, st>>>(s.r_off, s.r_idx, s.R, s.C, s.nnz, meta,
                                                          kWhereRowOffsets, kWhereRowIds,
                                                          long_rows(s) ? &meta->longest_row : nullptr);
  k_validate<<<grid_for(s.C, wpb, 65536), kValNT, 0, st>>>(s.c_off, s.c_idx, s.C, s.R, s.nnz, meta,
                                                          kWhereColOffsets, kWhereColIds,
                                                          nullptr);
  return cudaGetLastError();
}

// inv[map[k]] = k for k < n: the CSR->CSC map of the dual side from that of
// the primal side (the dual's CSR is the primal's CSC and vice versa).
__global__ void k_invert(const int32_t *__restrict__ map, int64_t n, int32_t *__restrict__ inv) {
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n;
       k += (int64_t)gridDim.x * blockDim.x) {
    const int32_t m = map[k];
    if (m >= 0 && m < n) inv[m] = (int32_t)k;  // a validated map is a permutation
  }
}

cudaError_t launch_invert(const int32_t *map, int64_t n, int32_t *inv, cudaStream_t st) {
  if (n > 0) k_invert<<<(int)std::min<int64_t>((n + 255) / 256, 152 * 16), 256, 0, st>>>(map, n, inv);
  return cudaGetLastError();
}

cudaError_t launch_csr2csc(const Side &s, int32_t *csr2csc, Meta *meta, cudaStream_t st) {
  if (s.nnz > 0)
    k_csr2csc<<<grid_for(s.nnz, kValNT * kMapK, 1 << 30), kValNT, 0, st>>>(s, csr2csc, meta);
  return cudaGetLastError();
}

cudaError_t launch_filter(const Side &s, int32_t smin, const Work &w, cudaStream_t st) {
  const int32_t ntiles = (int32_t)((s.nnz + kScanTile - 1) / kScanTile);
  if (ntiles > 0) {
    k_filter_reduce<<<ntiles, kScanNT, 0, st>>>(s, smin, w.tile, w.meta);
  }
  k_scan_tiles<<<1, 1024, 0, st>>>(w.tile, ntiles, &w.meta->kept, w.meta);
  if (ntiles > 0) {
    k_filter_scatter<<<ntiles, kScanNT, 0, st>>>(s, smin, w.tile, w.qs, w.c_idx_s, w.meta);
  }
  // (a column per thread: sides of up to 2^31 - 1 columns)
  k_filter_offsets<<<grid_for((int64_t)s.C + 1, 256, 1 << 30), 256, 0, st>>>(s, w.qs, w.tile, ntiles,
                                                                    w.c_off_s, w.meta);
  return cudaGetLastError();
}

cudaError_t launch_rows_work(const Side &s, int32_t smin, int32_t row_begin, int32_t row_end,
                             const Work &w, const CoreInfo &core, const Bins &bins,
                             cudaStream_t st) {
  const int32_t rows = row_end - row_begin;
  if (rows <= 0) return cudaSuccess;
  // (the tails of every row, also with a row range: its first incidence is
  // not known here)
  if (s.nnz > 0)
    k_tails<<<grid_for(s.nnz, kRowsNT * 4, 1 << 30), kRowsNT, 0, st>>>(
        0, s.nnz, s.r_idx, w.csr2csc, w.qs, w.c_off_s, w.tail_beg, w.tail_end, w.meta);
  const int grid = (rows + kRowsPerBlock - 1) / kRowsPerBlock;
  k_rows_work<<<grid, kRowsNT, 0, st>>>(s, smin, row_begin, row_end, w.c_idx_s, core, bins,
                                        w.tail_beg, w.tail_end, w.n_e, w.stage_pos, w.row_work,
                                        w.bin_rows, w.meta);
  return cudaGetLastError();
}

}  // namespace slg
