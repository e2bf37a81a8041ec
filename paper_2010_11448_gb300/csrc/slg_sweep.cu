// Threshold filter over a canonical edge list: L_s from L_s' for s >= s'.
//
// Section III defines L_s by the overlap threshold alone, so a pair of L_s'
// belongs to L_s exactly when its weight is >= s: L_s is the sub-list of
// L_s' with w >= s, in the same (i, j) order.  One walk at the smallest
// threshold of a sweep therefore answers every larger one.
//
// Stable compaction in three launches: per tile of kTile triples the count
// of kept ones; an exclusive scan of the tile counts (64-bit); per tile the
// kept triples written in order.
//
// Bound by memory bandwidth: the count reads the weights (4 bytes per
// triple), the write pass reads them again with the 32-byte sectors of i and
// j that hold a kept triple.  In the write pass a warp owns 1,024 consecutive
// triples and loads all of its weights before it uses any; one ballot per 32
// of them gives every place, with one block barrier per tile.  (A block scan
// per 256 triples, with three barriers, took 630 us where this takes 284 us on
// the 1.4e8-pair L_2 list of a 200K x 400K dual at s = 6.)
#include "slg_internal.cuh"

namespace slg {

namespace {

constexpr int kNT = 512;
constexpr int kRounds = 32;                              // triples per thread
constexpr int64_t kTile = (int64_t)kNT * kRounds;        // 16,384 triples
constexpr int kWarpTriples = 32 * kRounds;

__global__ __launch_bounds__(kNT) void k_keep_count(const int32_t *__restrict__ w, int64_t n,
                                                    int32_t s, long long *__restrict__ tile) {
  __shared__ int32_t ws[kNT / 32];
  const int64_t base = (int64_t)blockIdx.x * kTile + threadIdx.x;
  int32_t c = 0;
  if (base - threadIdx.x + kTile <= n) {
#pragma unroll
    for (int r = 0; r < kRounds; ++r) c += __ldcs(w + base + r * kNT) >= s;
  } else {
    for (int r = 0; r < kRounds; ++r) {
      const int64_t p = base + (int64_t)r * kNT;
      if (p < n) c += __ldcs(w + p) >= s;
    }
  }
  c = __reduce_add_sync(0xffffffffu, c);
  if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = c;
  __syncthreads();
  if (threadIdx.x < 32) {
    const int32_t x = threadIdx.x < kNT / 32 ? ws[threadIdx.x] : 0;
    const int32_t total = __reduce_add_sync(0xffffffffu, x);
    if (threadIdx.x == 0) tile[blockIdx.x] = total;
  }
}

// Exclusive scan of the tile counts in place; tile[n] = total.
__global__ __launch_bounds__(1024) void k_keep_scan(long long *tile, int64_t n) {
  __shared__ long long ws[1024 / 32 + 1];
  __shared__ long long carry;
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  for (int64_t b = 0; b < n; b += 1024) {
    const int64_t i = b + threadIdx.x;
    const long long x = i < n ? tile[i] : 0;
    long long total;
    const long long inc = block_inclusive_scan64<1024>(x, ws, &total);
    if (i < n) tile[i] = carry + inc - x;
    __syncthreads();
    if (threadIdx.x == 0) carry += total;
    __syncthreads();
  }
  if (threadIdx.x == 0) tile[n] = carry;
}

// capacity: entries of the output arrays (nothing is written beyond them).
__global__ __launch_bounds__(kNT) void k_keep_write(const int32_t *__restrict__ in_i,
                                                    const int32_t *__restrict__ in_j,
                                                    const int32_t *__restrict__ in_w, int64_t n,
                                                    int32_t s, const long long *__restrict__ tile,
                                                    int32_t *__restrict__ out_i,
                                                    int32_t *__restrict__ out_j,
                                                    int32_t *__restrict__ out_w,
                                                    long long capacity) {
  __shared__ int32_t ws[kNT / 32];
  const int lane = threadIdx.x & 31, wq = threadIdx.x >> 5;
  const int64_t base = (int64_t)blockIdx.x * kTile + (int64_t)wq * kWarpTriples + lane;
  int32_t v[kRounds];
  if (base - lane + kWarpTriples <= n) {
#pragma unroll
    for (int r = 0; r < kRounds; ++r) v[r] = __ldcs(in_w + base + r * 32);
  } else {
#pragma unroll
    for (int r = 0; r < kRounds; ++r) {
      const int64_t p = base + r * 32;
      v[r] = p < n ? __ldcs(in_w + p) : 0;  // s >= 1: not kept
    }
  }
  unsigned mine = 0;  // lane r: the ballot of round r
#pragma unroll
  for (int r = 0; r < kRounds; ++r) {
    const unsigned bal = __ballot_sync(0xffffffffu, v[r] >= s);
    if (lane == r) mine = bal;
  }
  const int32_t cnt = __popc(mine);
  const int32_t inc = warp_inclusive_scan(cnt);
  if (lane == 31) ws[wq] = inc;
  __syncthreads();
  const int32_t x = lane < wq ? ws[lane] : 0;  // earlier warps
  const long long first = tile[blockIdx.x] + __reduce_add_sync(0xffffffffu, x);
  const int32_t before = inc - cnt;  // lane r: kept triples of the warp before round r
#pragma unroll
  for (int r0 = 0; r0 < kRounds; r0 += 4) {
    int32_t vi[4], vj[4];
    unsigned bal[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      bal[u] = __shfl_sync(0xffffffffu, mine, r0 + u);
      const bool keep = (bal[u] >> lane) & 1u;
      const int64_t p = base + (r0 + u) * 32;
      vi[u] = keep ? __ldg(in_i + p) : 0;
      vj[u] = keep ? __ldg(in_j + p) : 0;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const long long q = first + __shfl_sync(0xffffffffu, before, r0 + u) +
                          __popc(bal[u] & ((1u << lane) - 1u));
      if (((bal[u] >> lane) & 1u) && q < capacity) {
        out_i[q] = vi[u];
        out_j[q] = vj[u];
        if (out_w) out_w[q] = v[r0 + u];
      }
    }
  }
}

}  // namespace

int64_t keep_tiles(int64_t n) { return (n + kTile - 1) / kTile; }

cudaError_t launch_keep_count(const int32_t *w, int64_t n, int32_t s, long long *tile,
                              cudaStream_t st) {
  const int64_t nt = keep_tiles(n);
  if (nt > 0) k_keep_count<<<(unsigned)nt, kNT, 0, st>>>(w, n, s, tile);
  k_keep_scan<<<1, 1024, 0, st>>>(tile, nt);
  return cudaGetLastError();
}

cudaError_t launch_keep_write(const int32_t *in_i, const int32_t *in_j, const int32_t *in_w,
                              int64_t n, int32_t s, const long long *tile, int32_t *out_i,
                              int32_t *out_j, int32_t *out_w, int64_t capacity, cudaStream_t st) {
  const int64_t nt = keep_tiles(n);
  if (nt > 0)
    k_keep_write<<<(unsigned)nt, kNT, 0, st>>>(in_i, in_j, in_w, n, s, tile, out_i, out_j, out_w,
                                               capacity);
  return cudaGetLastError();
}

}  // namespace slg
