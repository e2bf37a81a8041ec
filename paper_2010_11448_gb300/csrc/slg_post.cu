// After the edge list: ID squeezing (Section IV-E), the line graph's
// adjacency, and s-connected components (the components of L_s, the
// motivating analysis of Section I).
//
// Squeezing numbers the ids that occur in the list 0 .. n_ids-1 in
// ascending order of their original id, so a canonical list stays
// canonical.  The adjacency is the symmetric CSR of L_s: row v lists its
// smaller neighbours and then its larger ones (its own segment of the
// canonical list), both ascending.  Components are found by lock-free
// union-find over the pairs: each root links to the smaller root, so every
// label ends as the smallest id of its component.
//
// All of it is bound by memory bandwidth and the random accesses per pair
// (L_2 of a 250K x 500K hypergraph, the three calls 3.95 -> 1.65 ms: ids
// marked in a shared-memory map 450 -> 54 us; degrees from the segments and
// groups instead of atomics 903 -> 162; one sort of the pairs themselves by
// two 9-bit digits instead of positions by three 8-bit ones and a gather,
// 1,080 -> 480; union-find after two hooking rounds 286 -> 235).
// The list is checked on the device by the first pass over it; the kernels
// after it stop at its error flag, and the host reads the flag with the
// result.
#include <algorithm>

#include "slg_internal.cuh"

namespace slg {

namespace {

constexpr int kNT = 256;

int grid_for(int64_t items, int64_t cap = 65536) {
  int64_t g = (items + kNT - 1) / kNT;
  if (g > cap) g = cap;
  return g < 1 ? 1 : (int)g;
}

int sm_count() {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms > 0 ? sms : 1;
}

// err = 1 if an id is outside [0, R) or i >= j.
__global__ __launch_bounds__(kNT) void k_check_pairs(const int32_t *__restrict__ a,
                                                     const int32_t *__restrict__ b, int64_t n,
                                                     int32_t R, int32_t *err) {
  const int64_t step = (int64_t)gridDim.x * kNT;
  bool bad = false;
  for (int64_t p = (int64_t)blockIdx.x * kNT + threadIdx.x; p < n; p += 4 * step) {
    int32_t i[4], j[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int64_t q = p + u * step;
      i[u] = q < n ? __ldg(a + q) : 0;
      j[u] = q < n ? __ldg(b + q) : 1;
      if (q < n) bad |= i[u] < 0 || j[u] >= R || i[u] >= j[u];
    }
  }
  if (bad) atomicExch(err, 1);
}

// ---------------------------------------------------------------- squeeze --

// Largest id map held in shared memory while marking, words (200 KB).
constexpr int32_t kMarkSmemWords = 51200;
constexpr int kMarkNT = 1024;

// Checks the pairs and marks their ids in `bits` (one bit per id).  SMEM: the
// map of the CTA's pairs is kept in shared memory (an id costs a shared read
// and seldom an atomic) and merged at the end; else the global map is read
// first and seldom written.  A list's i is mostly its predecessor's.
template <bool SMEM>
__global__ __launch_bounds__(kMarkNT) void k_mark(const int32_t *__restrict__ a,
                                                  const int32_t *__restrict__ b, int64_t n,
                                                  int32_t R, uint32_t *__restrict__ bits,
                                                  int32_t *err) {
  extern __shared__ uint32_t s_bits[];
  const int32_t words = (int32_t)(((int64_t)R + 31) >> 5);
  uint32_t *map = SMEM ? s_bits : bits;
  if (SMEM) {
    for (int32_t x = threadIdx.x; x < words; x += kMarkNT) s_bits[x] = 0;
    __syncthreads();
  }
  auto mark = [&](int32_t v) {
    const uint32_t m = 1u << (v & 31);
    if (!(*(volatile uint32_t *)(map + (v >> 5)) & m)) atomicOr(map + (v >> 5), m);
  };
  const int lane = threadIdx.x & 31;
  const int64_t step = (int64_t)gridDim.x * kMarkNT;
  bool bad = false;
  for (int64_t p0 = (int64_t)blockIdx.x * kMarkNT + threadIdx.x - lane; p0 < n; p0 += 4 * step) {
    int32_t i[4], j[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int64_t q = p0 + u * step + lane;
      i[u] = q < n ? __ldg(a + q) : -2;
      j[u] = q < n ? __ldg(b + q) : -2;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int32_t prev = __shfl_up_sync(0xffffffffu, i[u], 1);
      if (i[u] == -2 && j[u] == -2 && p0 + u * step + lane >= n) continue;
      if (i[u] < 0 || j[u] >= R || i[u] >= j[u]) {
        bad = true;
        continue;
      }
      if (lane == 0 || prev != i[u]) mark(i[u]);
      mark(j[u]);
    }
  }
  if (bad) atomicExch(err, 1);
  if (SMEM) {
    __syncthreads();
    for (int32_t x = threadIdx.x; x < words; x += kMarkNT)
      if (s_bits[x]) atomicOr(bits + x, s_bits[x]);
  }
}

// cnt[x] = ids marked in word x (cnt[words] = 0: the scan's total).
__global__ __launch_bounds__(kNT) void k_word_counts(const uint32_t *__restrict__ bits,
                                                     int32_t words, int32_t *__restrict__ cnt) {
  const int64_t x = (int64_t)blockIdx.x * kNT + threadIdx.x;
  if (x <= words) cnt[x] = x < words ? __popc(bits[x]) : 0;
}

// word[x] = (marked ids, rank of the word's first one); old_of_new[rank] = id.
__global__ __launch_bounds__(kNT) void k_squeeze_map(const uint32_t *__restrict__ bits,
                                                     const int32_t *__restrict__ rank,
                                                     int32_t words, int2 *__restrict__ word,
                                                     int32_t *__restrict__ old_of_new,
                                                     const int32_t *err) {
  if (*err) return;
  const int64_t x = (int64_t)blockIdx.x * kNT + threadIdx.x;
  if (x >= words) return;
  uint32_t m = bits[x];
  int32_t r = rank[x];
  word[x] = make_int2((int32_t)m, r);
  while (m) {
    const int k = __ffs(m) - 1;
    m &= m - 1;
    old_of_new[r++] = (int32_t)(x << 5) + k;
  }
}

__global__ __launch_bounds__(kNT) void k_squeeze_ids(const int32_t *__restrict__ a,
                                                     const int32_t *__restrict__ b, int64_t n,
                                                     const int2 *__restrict__ word,
                                                     int32_t *__restrict__ oa,
                                                     int32_t *__restrict__ ob,
                                                     const int32_t *err) {
  if (*err) return;
  auto rank = [&](int32_t v) {
    const int2 x = __ldg(word + (v >> 5));
    return x.y + __popc((uint32_t)x.x & ((1u << (v & 31)) - 1u));
  };
  const int64_t step = (int64_t)gridDim.x * kNT;
  for (int64_t p = (int64_t)blockIdx.x * kNT + threadIdx.x; p < n; p += 4 * step) {
    int32_t i[4], j[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int64_t q = p + u * step;
      i[u] = q < n ? __ldg(a + q) : 0;
      j[u] = q < n ? __ldg(b + q) : 0;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int64_t q = p + u * step;
      if (q < n) {
        oa[q] = rank(i[u]);
        ob[q] = rank(j[u]);
      }
    }
  }
}

// -------------------------------------------------------------- adjacency --
//
// U[v] = pairs (i, j) with i < v and L[v] = pairs with j < v.  Row v starts at
// off[v] = U[v] + L[v]: first its L[v+1] - L[v] smaller neighbours, then its
// larger ones.  So pair p of the list (i, j) puts j at p + L[i + 1], and the
// q-th pair in the stable order by j puts i at q + U[j].

// Checks that the list is canonical and notes where each i's segment starts
// and ends (first, last one past).
__global__ __launch_bounds__(kNT) void k_segments(const int32_t *__restrict__ a,
                                                  const int32_t *__restrict__ b, int64_t n,
                                                  int32_t V, int32_t *__restrict__ first,
                                                  int32_t *__restrict__ last, int32_t *err) {
  const int64_t step = (int64_t)gridDim.x * kNT;
  bool bad = false;
  for (int64_t p = (int64_t)blockIdx.x * kNT + threadIdx.x; p < n; p += step) {
    const int32_t i = __ldg(a + p), j = __ldg(b + p);
    const int32_t pi = p ? __ldg(a + p - 1) : -1, pj = p ? __ldg(b + p - 1) : -1;
    const int32_t ni = p + 1 < n ? __ldg(a + p + 1) : -1;
    if (i < 0 || j >= V || i >= j || pi > i || (pi == i && pj >= j)) {
      bad = true;
      continue;
    }
    if (pi != i) first[i] = (int32_t)p;
    if (ni != i) last[i] = (int32_t)p + 1;
  }
  if (bad) atomicExch(err, 1);
}

// The same for the ascending keys of the pairs in the order by j.
__global__ __launch_bounds__(kNT) void k_groups(const uint32_t *__restrict__ keys, int64_t n,
                                                int32_t *__restrict__ first,
                                                int32_t *__restrict__ last, const int32_t *err) {
  if (*err) return;
  const int64_t step = (int64_t)gridDim.x * kNT;
  for (int64_t q = (int64_t)blockIdx.x * kNT + threadIdx.x; q < n; q += step) {
    const uint32_t k = __ldg(keys + q);
    if (q == 0 || __ldg(keys + q - 1) != k) first[k] = (int32_t)q;
    if (q + 1 == n || __ldg(keys + q + 1) != k) last[k] = (int32_t)q + 1;
  }
}

// len[v] = last[v] - first[v], len[V] = 0 (in place of `last`).
__global__ __launch_bounds__(kNT) void k_lengths(const int32_t *__restrict__ first,
                                                 int32_t *__restrict__ last, int32_t V) {
  const int64_t v = (int64_t)blockIdx.x * kNT + threadIdx.x;
  if (v <= V) last[v] = v < V ? last[v] - first[v] : 0;
}

__global__ __launch_bounds__(kNT) void k_offsets(const int32_t *__restrict__ U,
                                                 const int32_t *__restrict__ L, int32_t V,
                                                 long long *__restrict__ off, const int32_t *err) {
  if (*err) return;
  const int64_t v = (int64_t)blockIdx.x * kNT + threadIdx.x;
  if (v <= V) off[v] = (long long)U[v] + L[v];
}

__global__ __launch_bounds__(kNT) void k_fill_upper(const int32_t *__restrict__ a,
                                                    const int32_t *__restrict__ b,
                                                    const int32_t *__restrict__ w, int64_t n,
                                                    const int32_t *__restrict__ L,
                                                    int32_t *__restrict__ adj,
                                                    int32_t *__restrict__ adj_w,
                                                    const int32_t *err) {
  if (*err) return;
  const int64_t step = (int64_t)gridDim.x * kNT;
  for (int64_t p = (int64_t)blockIdx.x * kNT + threadIdx.x; p < n; p += 2 * step) {
    int32_t i[2], j[2], x[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int64_t q = p + u * step;
      i[u] = q < n ? __ldg(a + q) : 0;
      j[u] = q < n ? __ldg(b + q) : 0;
      x[u] = q < n && adj_w ? __ldg(w + q) : 0;
    }
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int64_t q = p + u * step;
      if (q < n) {
        const long long dst = q + __ldg(L + i[u] + 1);
        adj[dst] = j[u];
        if (adj_w) adj_w[dst] = x[u];
      }
    }
  }
}

// The stable order by j: a radix sort by digits of at most 10 bits whose
// payload is the pair itself (i, and w), and whose last pass writes the
// smaller neighbours to their place in the adjacency.  Per pass and tile of
// 4,096 pairs: digit counts, their scan in (digit, tile) order, and a scatter
// that first orders the tile in shared memory, so that the writes of a digit
// are consecutive.
constexpr int kTsNT = 512;
constexpr int kTsIPT = 8;  // (16: 64 registers spill or one CTA per SM)
constexpr int kTsTile = kTsNT * kTsIPT;
constexpr int kTsNW = kTsNT / 32;
constexpr int kTsMaxBits = 10;
constexpr int kTsMaxBins = 1 << kTsMaxBits;

// [stage kTsTile][counts kTsNW x bins, 16 bits][digit start, digit base: bins each][ws]
constexpr size_t ts_smem(int bins) {
  return (size_t)kTsTile * 4 + (size_t)kTsNW * bins * 2 + (size_t)bins * 8 + (kTsNW + 1) * 4;
}

__global__ __launch_bounds__(kTsNT) void k_ts_hist(const uint32_t *__restrict__ keys, int64_t n,
                                                   int shift, int bits, int32_t ntiles,
                                                   int32_t *__restrict__ hist,
                                                   const int32_t *err) {
  if (*err) return;
  __shared__ int32_t h[kTsMaxBins];
  const int bins = 1 << bits;
  for (int d = threadIdx.x; d < bins; d += kTsNT) h[d] = 0;
  __syncthreads();
  const int64_t base = (int64_t)blockIdx.x * kTsTile + threadIdx.x;
  uint32_t k[kTsIPT];
#pragma unroll
  for (int r = 0; r < kTsIPT; ++r) {
    const int64_t q = base + (int64_t)r * kTsNT;
    k[r] = q < n ? __ldg(keys + q) : 0;
  }
#pragma unroll
  for (int r = 0; r < kTsIPT; ++r)
    if (base + (int64_t)r * kTsNT < n) atomicAdd(h + ((k[r] >> shift) & (bins - 1)), 1);
  __syncthreads();
  for (int d = threadIdx.x; d < bins; d += kTsNT) hist[(int64_t)d * ntiles + blockIdx.x] = h[d];
}

// U (last pass): key_out[q] = the key, i and w go to place q + U[key] of
// i_out and w_out; else to place q.
__global__ __launch_bounds__(kTsNT, 3) void k_ts_scatter(
    const uint32_t *__restrict__ keys, const int32_t *__restrict__ vi,
    const int32_t *__restrict__ vw, int64_t n, int shift, int bits, int32_t ntiles,
    const int32_t *__restrict__ hist, const int32_t *__restrict__ U,
    uint32_t *__restrict__ key_out, int32_t *__restrict__ i_out, int32_t *__restrict__ w_out,
    const int32_t *err) {
  if (*err) return;
  extern __shared__ __align__(16) unsigned char smem[];
  const int bins = 1 << bits;
  uint32_t *stage = reinterpret_cast<uint32_t *>(smem);
  uint16_t *cnt = reinterpret_cast<uint16_t *>(stage + kTsTile);
  int32_t *s_start = reinterpret_cast<int32_t *>(cnt + kTsNW * bins);
  int32_t *s_base = s_start + bins;
  int32_t *ws = s_base + bins;
  const int lane = threadIdx.x & 31, wq = threadIdx.x >> 5;
  const uint32_t mask = (uint32_t)bins - 1u;
  for (int d = threadIdx.x; d < kTsNW * bins / 2; d += kTsNT)
    reinterpret_cast<uint32_t *>(cnt)[d] = 0;
  // a warp owns kTsTile / kTsNW consecutive pairs, 32 per round
  const int64_t tile0 = (int64_t)blockIdx.x * kTsTile;
  const int32_t live = (int32_t)(n - tile0 < kTsTile ? n - tile0 : kTsTile);
  const int32_t q0 = wq * (kTsTile / kTsNW) + lane;
  uint32_t k[kTsIPT];
#pragma unroll
  for (int r = 0; r < kTsIPT; ++r)
    k[r] = q0 + 32 * r < live ? __ldg(keys + tile0 + q0 + 32 * r) : 0;
  __syncthreads();
  uint16_t *mine = cnt + wq * bins;
  uint16_t rank[kTsIPT];  // among the warp's pairs of the digit, in order
#pragma unroll
  for (int r = 0; r < kTsIPT; ++r) {
    const bool on = q0 + 32 * r < live;
    const uint32_t d = (k[r] >> shift) & mask;
    const unsigned peers = __match_any_sync(0xffffffffu, on ? d : (uint32_t)bins + lane);
    const int below = __popc(peers & ((1u << lane) - 1u));
    uint16_t c = 0;
    if (on) c = mine[d];
    rank[r] = (uint16_t)(c + below);
    __syncwarp();
    if (on && lane == 31 - __clz(peers)) mine[d] = (uint16_t)(c + __popc(peers));
    __syncwarp();
  }
  __syncthreads();
  // digit totals over the warps, their exclusive scan over the digits
  const int per = (bins + kTsNT - 1) / kTsNT;  // digits per thread (1 or 2)
  int32_t tot[2] = {0, 0}, sum = 0;
  for (int x = 0; x < per; ++x) {
    const int d = threadIdx.x * per + x;
    if (d < bins) {
      int32_t run = 0;
      for (int w = 0; w < kTsNW; ++w) {
        const int32_t c = cnt[w * bins + d];
        cnt[w * bins + d] = (uint16_t)run;
        run += c;
      }
      tot[x] = run;
      sum += run;
    }
  }
  int32_t total;
  int32_t start = block_inclusive_scan<kTsNT>(sum, ws, &total) - sum;
  for (int x = 0; x < per; ++x) {
    const int d = threadIdx.x * per + x;
    if (d < bins) {
      s_start[d] = start;
      s_base[d] = hist[(int64_t)d * ntiles + blockIdx.x] - start;
      start += tot[x];
    }
  }
  __syncthreads();
  uint16_t pos[kTsIPT];  // place in the ordered tile
#pragma unroll
  for (int r = 0; r < kTsIPT; ++r) {
    const uint32_t d = (k[r] >> shift) & mask;
    pos[r] = (uint16_t)(s_start[d] + mine[d] + rank[r]);
    if (q0 + 32 * r < live) stage[pos[r]] = k[r];
  }
  __syncthreads();
  int32_t dst[kTsIPT];
#pragma unroll
  for (int r = 0; r < kTsIPT; ++r) {
    const int32_t t = r * kTsNT + (int32_t)threadIdx.x;
    dst[r] = 0;
    if (t < live) {
      const uint32_t key = stage[t];
      const int32_t q = t + s_base[(key >> shift) & mask];
      key_out[q] = key;
      dst[r] = U ? q + __ldg(U + key) : q;
    }
  }
  auto move = [&](const int32_t *__restrict__ in, int32_t *__restrict__ out) {
    uint32_t v[kTsIPT];
#pragma unroll
    for (int r = 0; r < kTsIPT; ++r)
      v[r] = q0 + 32 * r < live ? (uint32_t)__ldg(in + tile0 + q0 + 32 * r) : 0;
    __syncthreads();  // the stage is read
#pragma unroll
    for (int r = 0; r < kTsIPT; ++r)
      if (q0 + 32 * r < live) stage[pos[r]] = v[r];
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kTsIPT; ++r) {
      const int32_t t = r * kTsNT + (int32_t)threadIdx.x;
      if (t < live) out[dst[r]] = (int32_t)stage[t];
    }
  };
  move(vi, i_out);
  if (vw) move(vw, w_out);
}

// ------------------------------------------------------------- components --

__global__ __launch_bounds__(kNT) void k_iota(int32_t *__restrict__ x, int64_t n,
                                              const int32_t *err) {
  if (*err) return;
  const int64_t step = (int64_t)gridDim.x * kNT;
  for (int64_t v = (int64_t)blockIdx.x * kNT + threadIdx.x; v < n; v += step) x[v] = (int32_t)v;
}

constexpr int kMaxUnionSteps = 1 << 25;  // above any path length (ids < 2^24): a guard

// Path halving; parents only decrease, so the walk ends at a root.
__device__ __forceinline__ int32_t find_root(int32_t *parent, int32_t v) {
  for (int step = 0; step < kMaxUnionSteps; ++step) {
    const int32_t p = parent[v];
    if (p == v) return v;
    const int32_t gp = parent[p];
    if (gp != p) atomicMin(parent + v, gp);
    v = gp;
  }
  return -1;
}

// Hooks without atomics, over a sample of the list: the larger of a pair's
// two parents, where it is a root, goes under the smaller one (whichever
// store is last: a root is always put under a smaller id of its component).
// The first time, parents are the ids themselves; the second, after a
// compression, the roots that the first left.
__global__ __launch_bounds__(kNT) void k_hook(const int32_t *__restrict__ a,
                                              const int32_t *__restrict__ b, int64_t n,
                                              int64_t stride, int32_t *__restrict__ parent,
                                              const int32_t *err) {
  if (*err) return;
  const int64_t step = (int64_t)gridDim.x * kNT * stride;
  for (int64_t p = ((int64_t)blockIdx.x * kNT + threadIdx.x) * stride; p < n; p += step) {
    const int32_t x = parent[__ldg(a + p)], y = parent[__ldg(b + p)];
    const int32_t hi = x > y ? x : y, lo = x > y ? y : x;
    if (hi != lo && parent[hi] == hi) parent[hi] = lo;
  }
}

// Most pairs of a list lie in one component that the sample already formed:
// two equal parents tell so at once (a parent, however old, is a member of
// the component).
__global__ __launch_bounds__(kNT) void k_union(const int32_t *__restrict__ a,
                                               const int32_t *__restrict__ b, int64_t n,
                                               int32_t *__restrict__ parent, int32_t *err) {
  if (*err) return;
  const int64_t step = (int64_t)gridDim.x * kNT;
  for (int64_t p = (int64_t)blockIdx.x * kNT + threadIdx.x; p < n; p += step) {
    int32_t x = __ldg(a + p), y = __ldg(b + p);
    if (parent[x] == parent[y]) continue;
    int tries = 0;
    for (; tries < kMaxUnionSteps; ++tries) {
      x = find_root(parent, x);
      y = find_root(parent, y);
      if (x < 0 || y < 0) break;
      if (x == y) break;
      if (x > y) {
        const int32_t t = x;
        x = y;
        y = t;
      }
      // link the larger root under the smaller one; fails if y stopped
      // being a root meanwhile, then retry from the new roots
      if (atomicCAS(parent + y, y, x) == y) break;
    }
    if (tries >= kMaxUnionSteps || x < 0 || y < 0) atomicExch(err, 2);
  }
}

// Every id's parent becomes its root; child[r] = 1 for a root with others
// (given `child`).
__global__ __launch_bounds__(kNT) void k_flatten(int32_t *parent, int32_t R,
                                                 int32_t *__restrict__ child, int32_t *err) {
  if (*err) return;
  const int64_t step = (int64_t)gridDim.x * kNT;
  for (int64_t v = (int64_t)blockIdx.x * kNT + threadIdx.x; v < R; v += step) {
    const int32_t r = find_root(parent, (int32_t)v);
    if (r < 0) {
      atomicExch(err, 2);
      continue;
    }
    if (r != v) {
      atomicMin(parent + v, r);
      if (child && !child[r]) child[r] = 1;
    }
  }
}

// Components of the ids in the list: the roots with others (an id of the
// list shares its component with the pair's other id).
__global__ __launch_bounds__(kNT) void k_count_roots(const int32_t *__restrict__ child, int32_t R,
                                                     unsigned long long *__restrict__ n_comp,
                                                     const int32_t *err) {
  if (*err) return;
  const int64_t step = (int64_t)gridDim.x * kNT;
  int32_t c = 0;
  for (int64_t v = (int64_t)blockIdx.x * kNT + threadIdx.x; v < R; v += step) c += child[v];
  c = __reduce_add_sync(0xffffffffu, c);
  if ((threadIdx.x & 31) == 0 && c) atomicAdd(n_comp, (unsigned long long)c);
}

}  // namespace

// bits: (R + 31) / 32 words, zeroed by the caller; cnt, rank: one int per
// word and one more; word: one int2 per word; tile: xscan_tiles(words + 1).
// rank[words] = number of ids.
cudaError_t launch_squeeze(const int32_t *a, const int32_t *b, int64_t n, int32_t R,
                           uint32_t *bits, int32_t *cnt, int32_t *rank, void *word,
                           int32_t *tile, int32_t *oa, int32_t *ob, int32_t *old_of_new,
                           int32_t *err, cudaStream_t st) {
  const int32_t words = (int32_t)(((int64_t)R + 31) >> 5);
  if (n > 0) {
    const int sms = sm_count();
    if (words <= kMarkSmemWords) {
      const size_t smem = (size_t)words * 4;
      cudaError_t e = cudaFuncSetAttribute(k_mark<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           kMarkSmemWords * 4);
      if (e != cudaSuccess) return e;
      const int64_t want = (n + kMarkNT - 1) / kMarkNT;
      const int64_t most = (int64_t)sms * (smem <= 100 * 1024 ? 2 : 1);
      k_mark<true><<<(unsigned)(want < most ? want : most), kMarkNT, smem, st>>>(a, b, n, R, bits,
                                                                                err);
    } else {
      k_mark<false><<<sms * 2, kMarkNT, 0, st>>>(a, b, n, R, bits, err);
    }
  }
  // (a word per thread: up to 2^26 + 1 of them, above grid_for's default cap)
  k_word_counts<<<grid_for((int64_t)words + 1, (int64_t)1 << 30), kNT, 0, st>>>(bits, words, cnt);
  cudaError_t e = launch_xscan(cnt, rank, (int64_t)words + 1, tile, st);
  if (e != cudaSuccess) return e;
  int2 *w2 = static_cast<int2 *>(word);
  if (words > 0)
    k_squeeze_map<<<grid_for(words, (int64_t)1 << 30), kNT, 0, st>>>(bits, rank, words, w2,
                                                                     old_of_new, err);
  if (n > 0) k_squeeze_ids<<<grid_for((n + 3) / 4), kNT, 0, st>>>(a, b, n, w2, oa, ob, err);
  return cudaGetLastError();
}

namespace {

int key_bits(int32_t V) {
  int bits = 0;
  while (bits < 31 && ((int64_t)(V > 0 ? V - 1 : 0) >> bits) != 0) ++bits;
  return bits < 1 ? 1 : bits;
}

int64_t ts_tiles(int64_t n) { return (n + kTsTile - 1) / kTsTile; }

}  // namespace

int adjacency_passes(int32_t V) { return (key_bits(V) + kTsMaxBits - 1) / kTsMaxBits; }

// Digit counts of a pass and their scan.
size_t adjacency_scratch_ints(int64_t n) {
  const int64_t nh = kTsMaxBins * std::max<int64_t>(ts_tiles(n), 1);
  return (size_t)(2 * nh + xscan_tiles(nh) + 1);
}

// first, last, U, L: V + 1 ints each, the first two zeroed by the caller;
// tile: xscan_tiles(V + 1) ints; hist: adjacency_scratch_ints(n).  key[2],
// vi[2], vw[2]: n entries each (vi and vw, and key[0], only with more than
// one pass; vi[1], vw[1] only with more than two).
cudaError_t launch_adjacency(const int32_t *a, const int32_t *b, const int32_t *w, int64_t n,
                             int32_t V, int32_t *first, int32_t *last, int32_t *U, int32_t *L,
                             int32_t *tile, uint32_t *const key[2], int32_t *const vi[2],
                             int32_t *const vw[2], int32_t *hist, long long *off, int32_t *adj,
                             int32_t *adj_w, int32_t *err, cudaStream_t st) {
  const int gv = grid_for((int64_t)V + 1, (int64_t)1 << 30);
  if (n > 0) k_segments<<<grid_for(n), kNT, 0, st>>>(a, b, n, V, first, last, err);
  k_lengths<<<gv, kNT, 0, st>>>(first, last, V);
  cudaError_t e = launch_xscan(last, U, (int64_t)V + 1, tile, st);
  if (e != cudaSuccess) return e;
  const size_t zero = ((size_t)V + 1) * sizeof(int32_t);
  e = cudaMemsetAsync(first, 0, zero, st);
  if (e == cudaSuccess) e = cudaMemsetAsync(last, 0, zero, st);
  if (e != cudaSuccess) return e;
  if (n > 0) {
    e = cudaFuncSetAttribute(k_ts_scatter, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)ts_smem(kTsMaxBins));
    if (e != cudaSuccess) return e;
    const int bits = key_bits(V), passes = adjacency_passes(V);
    const int32_t nt = (int32_t)ts_tiles(n);
    const uint32_t *ks = reinterpret_cast<const uint32_t *>(b);
    const int32_t *is = a, *wsrc = adj_w ? w : nullptr;
    int shift = 0;
    const uint32_t *sorted = nullptr;
    for (int p = 0; p < passes; ++p) {
      const int db = (bits - shift + passes - p - 1) / (passes - p);  // bits of this pass
      const bool fin = p + 1 == passes;
      const int64_t nh = (int64_t)nt << db;
      int32_t *counts = hist, *offs = hist + nh, *tl = hist + 2 * nh;
      k_ts_hist<<<nt, kTsNT, 0, st>>>(ks, n, shift, db, nt, counts, err);
      e = launch_xscan(counts, offs, nh, tl, st);
      if (e != cudaSuccess) return e;
      uint32_t *ko = fin && p == 0 ? key[1] : key[p & 1];  // never the pass's source
      int32_t *io = fin ? adj : vi[p & 1];
      int32_t *wo = fin ? adj_w : vw[p & 1];
      k_ts_scatter<<<nt, kTsNT, ts_smem(1 << db), st>>>(ks, is, wsrc, n, shift, db, nt, offs,
                                                       fin ? U : nullptr, ko, io, wo, err);
      sorted = ks = ko;
      is = io;
      if (wsrc) wsrc = wo;
      shift += db;
    }
    k_groups<<<grid_for(n), kNT, 0, st>>>(sorted, n, first, last, err);
  }
  k_lengths<<<gv, kNT, 0, st>>>(first, last, V);
  e = launch_xscan(last, L, (int64_t)V + 1, tile, st);
  if (e != cudaSuccess) return e;
  k_offsets<<<gv, kNT, 0, st>>>(U, L, V, off, err);
  if (n > 0)
    k_fill_upper<<<grid_for((n + 1) / 2), kNT, 0, st>>>(a, b, w, n, L, adj, adj_w, err);
  return cudaGetLastError();
}

// child: R ints, zeroed by the caller.  *err: 1 an invalid pair, 2 a bounded
// loop gave up.
cudaError_t launch_components(const int32_t *a, const int32_t *b, int64_t n, int32_t R,
                              int32_t *labels, int32_t *child, unsigned long long *n_comp,
                              int32_t *err, cudaStream_t st) {
  constexpr int64_t kSample = 16;  // pairs per sampled one
  constexpr int kHooks = 2;
  if (n > 0) k_check_pairs<<<grid_for((n + 3) / 4), kNT, 0, st>>>(a, b, n, R, err);
  if (R > 0) k_iota<<<grid_for(R), kNT, 0, st>>>(labels, R, err);
  if (n > 0 && R > 0) {
    if (n >= 65536) {
      for (int r = 0; r < kHooks; ++r) {
        k_hook<<<grid_for(n / kSample), kNT, 0, st>>>(a, b, n, kSample, labels, err);
        k_flatten<<<grid_for(R), kNT, 0, st>>>(labels, R, nullptr, err);
      }
    }
    k_union<<<grid_for(n), kNT, 0, st>>>(a, b, n, labels, err);
    k_flatten<<<grid_for(R), kNT, 0, st>>>(labels, R, child, err);
    k_count_roots<<<grid_for(R, 152 * 8), kNT, 0, st>>>(child, R, n_comp, err);
  }
  return cudaGetLastError();
}

}  // namespace slg
