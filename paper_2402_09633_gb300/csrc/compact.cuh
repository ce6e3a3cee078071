// Edge filtering's compaction step: keep the edges whose score is above a
// threshold, in input order (a stable, deterministic stream compaction).
//
// At most kCompactMaxBlocks blocks, each with a run of consecutive edges: one
// launch counts the kept edges of every block; in the next, each block sums the
// counts before its own (and all of them: row 1 of the output starts behind row
// 0) and writes its kept edges there, ranked in input order (warp ballots within
// 1024 edges, a scan of the 32 ballots' counts, a running count from there on).
// The output is the kept edge list [2, n_kept], contiguous, plus the input id of
// every kept edge.
//
// The bytes (40 MB for 1.9M edges, half kept) take 6 us; what took the time was latency and launches.
// A launch of one block that scanned the counts stood between the two, and the scatter went through its
// 1024 edges in four dependent rounds of load, ballot and two block barriers.  1.9M edges: the filter call
// 439 -> 432 us (344 of them the MLP); 1,024, 1,216 or 4,096 blocks at most instead of 2,048: 430, 436, 429.
#pragma once
#include <cstdint>
#include "ptx.cuh"

namespace gnn {

constexpr int kCompactThreads = 256;
constexpr int kCompactRounds = 4;
constexpr int kCompactTile = kCompactThreads * kCompactRounds;    // edges a block takes at once
// More blocks would make the sums over their counts longer (8 loads a thread); fewer leave SMs idle.
constexpr int kCompactMaxBlocks = 2048;

// Tiles per block, and blocks.
__host__ __device__ inline int compact_tiles(int64_t m) {
  const int64_t tiles = (m + kCompactTile - 1) / kCompactTile;
  return (int)((tiles + kCompactMaxBlocks - 1) / kCompactMaxBlocks);
}
inline int compact_blocks(int64_t m) {
  const int64_t per = (int64_t)compact_tiles(m) * kCompactTile;
  return (int)((m + per - 1) / per);
}

__device__ __forceinline__ bool kept(float score, float threshold) { return score > threshold; }  // NaN: no

// The calling thread's scores of the tile at `base`: entry r is edge base + r * kCompactThreads + threadIdx.x.
__device__ __forceinline__ void compact_load(const float* __restrict__ scores, int64_t base, int m, float threshold,
                                             bool* keep) {
  float s[kCompactRounds];
#pragma unroll
  for (int r = 0; r < kCompactRounds; ++r) {
    const int64_t k = base + r * kCompactThreads + threadIdx.x;
    s[r] = k < m ? scores[k] : __int_as_float(0x7fffffff);           // NaN past the end
  }
#pragma unroll
  for (int r = 0; r < kCompactRounds; ++r) keep[r] = kept(s[r], threshold);
}

__global__ void __launch_bounds__(kCompactThreads) compact_count_kernel(const float* __restrict__ scores, int m,
                                                                        float threshold, int tiles,
                                                                        int* __restrict__ counts) {
  __shared__ int wsum[kCompactThreads / 32];
  pdl_wait();
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  int c = 0;
  for (int i = 0; i < tiles; ++i) {
    bool keep[kCompactRounds];
    compact_load(scores, ((int64_t)blockIdx.x * tiles + i) * kCompactTile, m, threshold, keep);
#pragma unroll
    for (int r = 0; r < kCompactRounds; ++r) c += keep[r] ? 1 : 0;
  }
  c = __reduce_add_sync(0xffffffffu, c);
  if (lane == 0) wsum[warp] = c;
  __syncthreads();
  if (t == 0) {
    int s = 0;
    for (int w = 0; w < kCompactThreads / 32; ++w) s += wsum[w];
    counts[blockIdx.x] = s;
  }
}

// Exclusive scan of a long int array in place, in two launches of compact_blocks(n) blocks, each with a run of
// `tiles` = compact_tiles(n) times 1024 consecutive entries: scan_reduce_kernel (sum of every block's entries,
// saturated at INT32_MAX), scan_apply_kernel (each block sums the sums before its own, and scans its entries
// from there; the total of all goes to *total).  At most 2,048 blocks, so that their sums over the block sums
// stay behind the entries themselves: with 1,024 entries a block whatever n, they grew with its square.
// Sums are taken in 64 bits and the total saturates at INT32_MAX, so a caller that compares it with its
// capacity (below INT32_MAX) sees an overflow as "too many"; the offsets are then meaningless and must not
// be used.
constexpr int kScanBlock = 1024;
static_assert(kScanBlock == kCompactTile, "compact_tiles and compact_blocks count in entries of a scan block");

__global__ void __launch_bounds__(kScanBlock) scan_reduce_kernel(const int* __restrict__ v, int n, int tiles,
                                                                 int* __restrict__ sums) {
  __shared__ long long wsum[32];
  pdl_wait();
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  long long x = 0;
  for (int k = 0; k < tiles; ++k) {
    const int64_t i = ((int64_t)blockIdx.x * tiles + k) * kScanBlock + t;
    x += i < n ? v[i] : 0;
  }
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  if (lane == 0) wsum[warp] = x;
  __syncthreads();
  if (t == 0) {
    long long s = 0;
    for (int w = 0; w < 32; ++w) s += wsum[w];
    sums[blockIdx.x] = s > 0x7fffffffLL ? 0x7fffffff : (int)s;
  }
}

__global__ void __launch_bounds__(kScanBlock) scan_apply_kernel(int* __restrict__ v, int n, int tiles,
                                                                const int* __restrict__ sums,
                                                                int* __restrict__ total) {
  __shared__ long long part[2][32];
  __shared__ int wsum[2][32];                            // two tiles' worth in turn
  pdl_wait();
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  long long before = 0, all = 0;
  for (int b = t; b < (int)gridDim.x; b += kScanBlock) {
    const long long s = sums[b];
    all += s;
    before += b < (int)blockIdx.x ? s : 0;
  }
  for (int o = 16; o > 0; o >>= 1) {
    before += __shfl_xor_sync(0xffffffffu, before, o);
    all += __shfl_xor_sync(0xffffffffu, all, o);
  }
  if (lane == 0) { part[0][warp] = before; part[1][warp] = all; }
  unsigned run = 0;                                      // offset of the tile's first entry (meaningless past 2^31)
  for (int k = 0; k < tiles; ++k) {
    const int64_t i = ((int64_t)blockIdx.x * tiles + k) * kScanBlock + t;
    const int c = i < n ? v[i] : 0;
    unsigned x = (unsigned)c;
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) wsum[k & 1][warp] = (int)x;
    __syncthreads();
    if (k == 0) {
      long long b = part[0][lane], a = part[1][lane];
      for (int o = 16; o > 0; o >>= 1) {
        b += __shfl_xor_sync(0xffffffffu, b, o);
        a += __shfl_xor_sync(0xffffffffu, a, o);
      }
      run = (unsigned)b;
      if (blockIdx.x == 0 && t == 0) *total = a > 0x7fffffffLL ? 0x7fffffff : (int)a;
    }
    unsigned w = (unsigned)wsum[k & 1][lane];            // inclusive scan over the warps' sums
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned y = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += y;
    }
    const unsigned first = __shfl_sync(0xffffffffu, w, warp > 0 ? warp - 1 : 0);
    if (i < n) v[i] = (int)(run + (warp > 0 ? first : 0u) + x - (unsigned)c);
    run += __shfl_sync(0xffffffffu, w, 31);
  }
}

// counts: of gridDim.x blocks, fewer than 2^31 edges in all.  The total goes to *total.
__global__ void __launch_bounds__(kCompactThreads) compact_scatter_kernel(
    const float* __restrict__ scores, const int32_t* __restrict__ ei, int m, float threshold, int tiles,
    const int* __restrict__ counts, int* __restrict__ total, int32_t* __restrict__ out_ei,
    int32_t* __restrict__ out_id) {
  constexpr int kWarps = kCompactThreads / 32;
  static_assert(kWarps * kCompactRounds == 32, "a lane per ballot of a tile");
  __shared__ int sums[2][kWarps];
  __shared__ int wcnt[2][32];                            // by round and warp; two tiles' worth in turn
  pdl_wait();
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  int before = 0, all = 0;
  for (int i = t; i < (int)gridDim.x; i += kCompactThreads) {
    const int c = counts[i];
    all += c;
    before += i < (int)blockIdx.x ? c : 0;
  }
  before = __reduce_add_sync(0xffffffffu, before);
  all = __reduce_add_sync(0xffffffffu, all);
  if (lane == 0) { sums[0][warp] = before; sums[1][warp] = all; }
  __syncthreads();
  int run = 0, n_kept = 0;
#pragma unroll
  for (int w = 0; w < kWarps; ++w) { run += sums[0][w]; n_kept += sums[1][w]; }
  if (blockIdx.x == 0 && t == 0) *total = n_kept;
  for (int i = 0; i < tiles; ++i) {
    const int64_t base = ((int64_t)blockIdx.x * tiles + i) * kCompactTile;
    bool keep[kCompactRounds];
    unsigned ball[kCompactRounds];
    compact_load(scores, base, m, threshold, keep);
    int u[kCompactRounds], v[kCompactRounds];
#pragma unroll
    for (int r = 0; r < kCompactRounds; ++r) {
      ball[r] = __ballot_sync(0xffffffffu, keep[r]);
      if (lane == 0) wcnt[i & 1][r * kWarps + warp] = __popc(ball[r]);
      const int64_t k = base + r * kCompactThreads + t;
      if (keep[r]) { u[r] = ei[k]; v[r] = ei[(size_t)m + k]; }
    }
    __syncthreads();
    const int own = wcnt[i & 1][lane];
    int x = own;                                         // inclusive scan over (round, warp)
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
#pragma unroll
    for (int r = 0; r < kCompactRounds; ++r) {
      const int first = __shfl_sync(0xffffffffu, x - own, r * kWarps + warp);
      if (!keep[r]) continue;
      const int pos = run + first + __popc(ball[r] & ((1u << lane) - 1u));
      out_ei[pos] = u[r];
      out_ei[(size_t)n_kept + pos] = v[r];
      if (out_id) out_id[pos] = (int)(base + r * kCompactThreads + t);
    }
    run += __shfl_sync(0xffffffffu, x, 31);
  }
}

}  // namespace gnn
