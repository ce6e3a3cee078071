// Destination-keyed CSR of the candidate edges, built on the device.
//
// The message-passing step sums every edge's message into its destination
// node.  Sorting the edges by destination turns that sum into a contiguous
// segment per node, read in a fixed order (deterministic, no float atomics),
// and lets the edge kernels stream the per-edge state in that order.
//
// Steps: a stable LSD radix sort of (key, input id), key = dst, or n_nodes for
// an edge with an endpoint out of range, whose first pass forms the keys from
// the edge index itself; then one kernel gathers the sources in sorted order
// and marks the first slot of every node (rowptr).  A stable sort of keys that
// only differ in input id gives the unique order "by destination, then input id".
//
// Each pass counts digits per tile, scans each digit's counts over the tiles
// and scatters.  Digits have up to 11 bits, as many as make the fewest passes
// (radix_digit_bits): 300k nodes take two passes of 10 bits, up to 2,047 nodes
// one.  What bounded the build was latency, not bytes (16 MB for 1M edges, 3 us
// at the copy rate): twelve launches, scatter rounds with four block barriers
// and a dependent load each, one block walking every tile's counts.  Here a
// thread's sixteen elements are loaded at once, a warp ranks its own 512 elements
// against its own counters without a block barrier, and a warp per digit scans
// the counts, in seven launches.  1M edges, 300k nodes: 131 -> 66 us, 58 with tiles
// sorted before they are written; 7,200 edges, 2,000 nodes (one pass): nine launches
// -> four, 45 us of the tiny event's 164 less.
#pragma once
#include <cstdint>
#include "ptx.cuh"

namespace gnn {

constexpr int kRadixThreads = 256;
constexpr int kRadixRounds = 16;
constexpr int kRadixTile = kRadixThreads * kRadixRounds;   // elements per tile
constexpr int kRadixWarps = kRadixThreads / 32;
constexpr int kRadixMaxBits = 11;
constexpr int kRadixMaxBins = 1 << kRadixMaxBits;

// Bits a key in [0, max_key] has, and the digits it is sorted by: `passes` digits of `digit` bits.
struct RadixPlan { int passes, digit; };
__host__ __device__ inline RadixPlan radix_plan(int max_key) {
  int bits = 0;
  while (bits < 31 && (max_key >> bits) != 0) ++bits;
  if (bits == 0) bits = 1;
  const int passes = (bits + kRadixMaxBits - 1) / kRadixMaxBits;
  return {passes, (bits + passes - 1) / passes};
}
// Ints of the per-tile digit counts of one pass, followed by the digit totals.
__host__ __device__ inline size_t radix_hist_ints(size_t n) {
  return ((n + kRadixTile - 1) / kRadixTile + 1) * (size_t)kRadixMaxBins;
}

// Where a pass reads its elements: the edge index (first pass of the CSR: key from the endpoints, value
// = input id), keys alone (first pass of another sort: value = position) or the previous pass's output.
struct RadixEdges {
  const int32_t* ei;
  int n_edges, n_nodes;
  uint32_t* err;
  __device__ __forceinline__ int key(int k) const {
    const int s = ei[k], d = ei[(size_t)n_edges + k];
    return ((s >= 0) & (s < n_nodes) & (d >= 0) & (d < n_nodes)) ? d : n_nodes;
  }
  __device__ __forceinline__ int val(int k) const { return k; }
  // An out-of-range edge sets DEV_ERR_INDEX_RANGE in *err (when err is not null); it sorts last.
  __device__ __forceinline__ void check(int key) const {
    if (key == n_nodes && err) atomicOr(err, DEV_ERR_INDEX_RANGE);
  }
};
struct RadixKeys {
  const int* keys;
  __device__ __forceinline__ int key(int k) const { return keys[k]; }
  __device__ __forceinline__ int val(int k) const { return k; }
  __device__ __forceinline__ void check(int) const {}
};
struct RadixPairs {
  const int* keys;
  const int* vals;
  __device__ __forceinline__ int key(int k) const { return keys[k]; }
  __device__ __forceinline__ int val(int k) const { return vals[k]; }
  __device__ __forceinline__ void check(int) const {}
};

// Digit counts per tile: hist[digit * n_tiles + tile].
template <typename Src>
__global__ void __launch_bounds__(kRadixThreads) radix_count_kernel(const Src src, int n, int shift, int bins, int n_tiles,
                                                                    int* __restrict__ hist) {
  pdl_wait();
  pdl_trigger_small();
  __shared__ int cnt[kRadixMaxBins];
  for (int d = threadIdx.x; d < bins; d += kRadixThreads) cnt[d] = 0;
  __syncthreads();
  const int base = blockIdx.x * kRadixTile + threadIdx.x;
  int key[kRadixRounds];
#pragma unroll
  for (int r = 0; r < kRadixRounds; ++r) key[r] = base + r * kRadixThreads < n ? src.key(base + r * kRadixThreads) : -1;
#pragma unroll
  for (int r = 0; r < kRadixRounds; ++r)
    if (key[r] >= 0) {
      src.check(key[r]);
      atomicAdd(&cnt[(key[r] >> shift) & (bins - 1)], 1);
    }
  __syncthreads();
  for (int d = threadIdx.x; d < bins; d += kRadixThreads) hist[(size_t)d * n_tiles + blockIdx.x] = cnt[d];
}

// One warp per digit: its counts over the tiles become exclusive offsets, in place; totals[d] = their sum.
__global__ void __launch_bounds__(kRadixThreads) radix_scan_kernel(int* __restrict__ hist, int bins, int n_tiles,
                                                                   int* __restrict__ totals) {
  pdl_wait();
  pdl_trigger_small();
  const int d = blockIdx.x * kRadixWarps + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (d >= bins) return;
  int* h = hist + (size_t)d * n_tiles;
  int run = 0;
  for (int t = lane; t - lane < n_tiles; t += 4 * 32) {
    int v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = t + 32 * k < n_tiles ? h[t + 32 * k] : 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      int x = v[k];                                        // inclusive scan inside the warp
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
      }
      if (t + 32 * k < n_tiles) h[t + 32 * k] = run + x - v[k];
      run += __shfl_sync(0xffffffffu, x, 31);
    }
  }
  if (lane == 0) totals[d] = run;
}

// Stable scatter of one pass.  Warp w of a tile's block owns the tile's elements [512 w, 512 w + 512) and
// takes them 32 at a time in input order: an element's rank among its warp's equal digits is the warp's
// count so far plus __match_any_sync.  Then the warps' counts are scanned per digit, on top of the digit's
// offset: keys with a smaller digit, plus those with this digit in earlier tiles.  The tile is put in digit
// order in shared memory first, so that neighbouring threads write neighbouring places of a digit's run.
template <typename Src>
__global__ void __launch_bounds__(kRadixThreads) radix_scatter_kernel(const Src src, int* __restrict__ keys_out,
                                                                      int* __restrict__ vals_out, int n, int shift,
                                                                      int bins, int n_tiles,
                                                                      const int* __restrict__ offs,
                                                                      const int* __restrict__ totals) {
  pdl_wait();
  pdl_trigger_small();
  __shared__ int first[kRadixMaxBins];                     // global position of the tile's first element per digit
  __shared__ uint16_t start[kRadixMaxBins];                // place of it inside the sorted tile
  __shared__ __align__(16) uint16_t wcnt[kRadixWarps][kRadixMaxBins];   // counts; later the sorted tile
  __shared__ int wsum[2][kRadixWarps];
  static_assert(sizeof(wcnt) == 2 * kRadixTile * sizeof(int), "the sorted tile takes the counts' place");
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const int base = blockIdx.x * kRadixTile + warp * (32 * kRadixRounds) + lane;
  int key[kRadixRounds], val[kRadixRounds];
#pragma unroll
  for (int r = 0; r < kRadixRounds; ++r) {
    const int k = base + 32 * r;
    key[r] = k < n ? src.key(k) : -1;
    val[r] = k < n ? src.val(k) : 0;
  }
  // digit bases: exclusive scan of the totals, bins / 256 (at least one) consecutive digits per thread
  const int per = bins > kRadixThreads ? bins / kRadixThreads : 1;
  int tot[kRadixMaxBins / kRadixThreads], sum = 0;
#pragma unroll
  for (int k = 0; k < kRadixMaxBins / kRadixThreads; ++k) {
    const int d = t * per + k;
    tot[k] = (k < per && d < bins) ? totals[d] : 0;
    sum += tot[k];
  }
  int x = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) wsum[0][warp] = x;
  const int half = bins >> 1, half_bits = __ffs(half) - 1;      // two 16-bit counts per word
  for (int i = t; i < kRadixWarps * half; i += kRadixThreads)
    reinterpret_cast<uint32_t*>(wcnt[i >> half_bits])[i & (half - 1)] = 0u;
  __syncthreads();
  int run = x - sum;
  for (int w = 0; w < warp; ++w) run += wsum[0][w];
#pragma unroll
  for (int k = 0; k < kRadixMaxBins / kRadixThreads; ++k) {
    const int d = t * per + k;
    if (k < per && d < bins) {
      first[d] = run + offs[(size_t)d * n_tiles + blockIdx.x];
      run += tot[k];
    }
  }
  // ranks inside the warp
  uint16_t rank[kRadixRounds];
  const unsigned below = (1u << lane) - 1u;
#pragma unroll
  for (int r = 0; r < kRadixRounds; ++r) {
    const int d = key[r] >= 0 ? (key[r] >> shift) & (bins - 1) : kRadixMaxBins;
    const unsigned peers = __match_any_sync(0xffffffffu, d);
    const int had = d < kRadixMaxBins ? wcnt[warp][d] : 0;
    rank[r] = (uint16_t)(had + __popc(peers & below));
    __syncwarp();
    if (d < kRadixMaxBins && (peers & below) == 0u) wcnt[warp][d] = (uint16_t)(had + __popc(peers));
    __syncwarp();
  }
  __syncthreads();
  int cnt = 0;                                             // this thread's digits: counts of the warps before
  int own[kRadixMaxBins / kRadixThreads];
#pragma unroll
  for (int k = 0; k < kRadixMaxBins / kRadixThreads; ++k) {
    const int d = t * per + k;
    own[k] = cnt;
    if (k < per && d < bins) {
      int c = 0;
#pragma unroll
      for (int w = 0; w < kRadixWarps; ++w) {
        const int v = wcnt[w][d];
        wcnt[w][d] = (uint16_t)c;
        c += v;
      }
      cnt += c;
    }
  }
  int y = cnt;                                             // ... and of the smaller digits
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int z = __shfl_up_sync(0xffffffffu, y, o);
    if (lane >= o) y += z;
  }
  if (lane == 31) wsum[1][warp] = y;
  __syncthreads();
  int before = y - cnt;
  for (int w = 0; w < warp; ++w) before += wsum[1][w];
#pragma unroll
  for (int k = 0; k < kRadixMaxBins / kRadixThreads; ++k) {
    const int d = t * per + k;
    if (k < per && d < bins) start[d] = (uint16_t)(before + own[k]);
  }
  __syncthreads();
  int place[kRadixRounds];
#pragma unroll
  for (int r = 0; r < kRadixRounds; ++r) {
    const int d = (key[r] >> shift) & (bins - 1);
    place[r] = key[r] >= 0 ? start[d] + wcnt[warp][d] + rank[r] : 0;
  }
  __syncthreads();                                         // the counts are read: their place takes the tile
  int* tile_key = reinterpret_cast<int*>(&wcnt[0][0]);
  int* tile_val = tile_key + kRadixTile;
#pragma unroll
  for (int r = 0; r < kRadixRounds; ++r)
    if (key[r] >= 0) {
      tile_key[place[r]] = key[r];
      tile_val[place[r]] = val[r];
    }
  __syncthreads();
  const int64_t left = (int64_t)n - (int64_t)blockIdx.x * kRadixTile;
  const int m = left < kRadixTile ? (int)left : kRadixTile;
  for (int i = t; i < m; i += kRadixThreads) {
    const int k = tile_key[i], d = (k >> shift) & (bins - 1);
    const int pos = first[d] + (i - start[d]);
    keys_out[pos] = k;
    vals_out[pos] = tile_val[i];
  }
}

// rowptr[j] = first sorted slot whose key >= j (binary search), for j in [0, n_nodes].
__global__ void csr_rowptr_kernel(const int* __restrict__ keys_sorted, int n_edges, int n_nodes,
                                  int* __restrict__ rowptr) {
  pdl_wait();
  pdl_trigger_small();
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j > n_nodes) return;
  int lo = 0, hi = n_edges;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (keys_sorted[mid] < j) lo = mid + 1; else hi = mid;
  }
  rowptr[j] = lo;
}

// Sorted order -> perm, src_sorted (0 for an invalid edge) and, when wanted, dst_sorted (clamped for
// invalid edges), one thread per slot; and the row pointers, one thread per node and one more.
__global__ void csr_finish_kernel(const int32_t* __restrict__ ei, const int* __restrict__ keys_sorted,
                                  const int* __restrict__ vals_sorted, int n_edges, int n_nodes, int* __restrict__ perm,
                                  int* __restrict__ src_sorted, int* __restrict__ dst_sorted, int* __restrict__ rowptr) {
  pdl_wait();
  pdl_trigger_small();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n_edges) {
    const int id = vals_sorted[i], key = keys_sorted[i];
    perm[i] = id;
    src_sorted[i] = key < n_nodes ? ei[id] : 0;
    if (dst_sorted) dst_sorted[i] = key < n_nodes ? key : 0;
  }
  if (i <= n_nodes) {
    int lo = 0, hi = n_edges;
    while (lo < hi) {
      const int mid = lo + ((hi - lo) >> 1);
      if (keys_sorted[mid] < i) lo = mid + 1; else hi = mid;
    }
    rowptr[i] = lo;
  }
}

}  // namespace gnn
