// Graph construction in the embedding space: every pair of hits whose
// embeddings lie within a fixed radius becomes a candidate edge (fixed-radius
// nearest neighbours).
//
// The embeddings are unit vectors, so each coordinate lies in [-1, 1].  Hits
// are binned on a uniform grid over their first K coordinates (K = 4 when the
// embedding has at least 4, else 3) with cells a little wider than half the
// radius (a coordinate outside [-1, 1] is clamped to the edge cells, which
// keeps the search exact, only slower), and sorted by cell (the library's
// stable radix sort); their embeddings and r values are then gathered into
// that order, zero-padded to a multiple of four coordinates.  A pair within
// the radius lies at most two cells apart on each axis, so the partners of a
// hit sit in the 5^(K-1) "rows" of cells around its own (rows over the first
// K-1 gridded coordinates), and in each row in one run of at most five
// consecutive cells along the last one, which is one contiguous range of
// sorted positions.  Rows before the hit's own row hold only earlier positions:
// each pair is visited once, by its earlier sorted position, which scans
// (5^(K-1) + 1) / 2 rows (its own row from the next position on).
//
// The test is the full squared distance, summed over the coordinates in order
// with one rounding per product and per sum (no fused multiply-add; the zero
// padding adds exact zeros), against radius^2 rounded to fp32; a tensor-core
// filter that never turns a pair down decides which pairs it is made for (many
// hits in up to three dimensions do without it).  Each pair becomes one edge,
// oriented from the hit with the smaller r (column 0 of the node features, hit
// id as tie-break).  A counting pass, an exclusive scan of the per-hit counts and
// a writing pass make the output order deterministic: by the visiting hit's
// sorted position, then by row and position of the partner.
// The counting pass also keeps the partners it finds, in the order it finds
// them, in a chain of 64-byte chunks per hit (its own first chunk, further ones
// from a pool), so the writing pass copies instead of searching again; a hit
// whose chain could not grow (pool exhausted) is searched again.
#pragma once
#include <climits>
#include <cstdint>
#include "ptx.cuh"

namespace gnn {

constexpr int kFrnnReach = 2;            // cells a partner can lie away on each axis
constexpr int kFrnnChunk = 16;           // ints per partner chunk: 15 sorted positions + the next chunk
constexpr int kFrnnLost = -2;            // link of a hit's first chunk: chain incomplete, search again

// Cells per axis for a grid over K coordinates (K = 3 or 4): cells 0.1 % wider than half the radius,
// so that the rounding of the cell coordinates and of the distance test never puts a pair within
// the radius three cells apart; at most 128 (K = 3) or 64 (K = 4) cells per axis.
__host__ __device__ inline int frnn_grid(float radius, int K) {
  const int max_grid = K == 4 ? 64 : 128;
  const float cells = 1.998f * (float)kFrnnReach / radius;
  return cells >= (float)max_grid ? max_grid : (cells < 1.0f ? 1 : (int)cells);
}

__device__ __forceinline__ int frnn_coord(float e, int grid) {
  int c = (int)floorf((e + 1.0f) * 0.5f * (float)grid);
  return c < 0 ? 0 : (c >= grid ? grid - 1 : c);
}

// Cell key of every hit: its cell over the first K coordinates (missing ones count as cell 0),
// row-major with the last gridded coordinate fastest.  Also zeroes the count of pool chunks taken.
template <int K>
__global__ void frnn_cell_kernel(const float* __restrict__ emb, int n, int dim, int grid, int* __restrict__ keys,
                                 int* __restrict__ next_chunk) {
  pdl_wait();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i == 0) *next_chunk = 0;
  if (i >= n) return;
  const float* e = emb + (size_t)i * dim;
  int key = 0;
#pragma unroll
  for (int k = 0; k < K; ++k) key = key * grid + (k < dim ? frnn_coord(e[k], grid) : 0);
  keys[i] = key;
}

// The tensor-core filter of the pair search.  With a = ah + al and b = bh + bl (bf16 parts) and the
// squared norms in three bf16 parts each, one product of K = 32 (dimensions 0-7; 32 more for eight
// further ones) gives
//   f = (1 - c)(|a|^2 + |b|^2) - 2 (ah bh + ah bl + al bh) - r2',  c = 2^-14, r2' slightly above r2.
// Against the squared distance d the parts left out, the splits' rounding and the accumulation are off
// by less than 3e-5 (|a|^2 + |b|^2) / 2 + 1e-5 (|a|^2 + |b|^2), under half of c (|a|^2 + |b|^2): a pair
// with d < r2 never gives f >= 0.  Only pairs with f < 0 are tested exactly.  A hit whose squared norm
// passes 1e18 is "wild": its operands are zero and its norm slot -1e30, so that f is finite everywhere and
// such a hit is tested exactly against every candidate.  A hit with an infinite or NaN coordinate is within
// no radius of any (its differences are infinite or NaN): its norm slot is one that no radius reaches.
// K slots: 0-7 -2ah.bh, 8-15 -2ah.bl, 16-23 -2al.bh, 24-26 |a|^2 parts x 1, 27-29 1 x |b|^2 parts.
constexpr float kFrnnSlack = 1.0f / 16384.0f;
constexpr float kFrnnWildNorm = 1e18f, kFrnnWild = -1e30f;

__device__ __forceinline__ uint32_t frnn_hi(float x, float y) { return pack_bf16x2(x, y); }
__device__ __forceinline__ uint32_t frnn_lo(float x, float y, uint32_t hi) {
  return pack_bf16x2(x - __uint_as_float(hi << 16), y - __uint_as_float(hi & 0xffff0000u));
}
// Three bf16 parts of v as float values.
__device__ __forceinline__ void frnn_parts(float v, float* q) {
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    q[k] = __bfloat162float(__float2bfloat16_rn(v));
    v -= q[k];
  }
}

// Whether any coordinate of this quad's hit is infinite or NaN (each lane holds some of them; called by whole warps).
template <int SETS>
__device__ __forceinline__ bool frnn_odd(const float2* v) {
  float z = 0.f;
#pragma unroll
  for (int s = 0; s < SETS; ++s) z += (v[s].x - v[s].x) + (v[s].y - v[s].y);         // 0 or NaN
  const unsigned odd = __ballot_sync(0xffffffffu, !(z == 0.f));
  return ((odd >> (threadIdx.x & 28)) & 15u) != 0u;
}

// What the search reads, from the sorted order, in one launch.  Blocks below frag_blocks: sorted copies
// emb_s [n, 4 * CH] (zero-padded) and r_s [n] = x[ids[t], 0], and the filter's B fragments, eight hits to
// a block: lane 4n + t of block b holds, for hit 8b + n and its dimensions 2t, 2t + 1 of each set of
// eight, (bh, bl) and, in the first set, the norm slots.  One uint4 per lane and set of eight dimensions
// (.x bh, .y bl, .z norm slots).  Lanes past the last hit get a norm that no radius reaches.  The other
// blocks: cell_start[j] = first sorted position whose cell is at least j, j in [0, n_cells].  The build
// is a chain of launches next to the search: this one was three, the scan of the counts three (now two),
// the reset of the chunk count one of its own, and none was a dependent launch.  2,000 hits 132 -> 104 us,
// 30,000 hits 230 -> 203, full event 839 -> 811.
template <int CH>
__global__ void frnn_layout_kernel(const float* __restrict__ emb, const float* __restrict__ x, int x_stride, int n,
                                   int dim, const int* __restrict__ ids, const int* __restrict__ cell_keys,
                                   int n_cells, int frag_blocks, float2* __restrict__ emb_s, float* __restrict__ r_s,
                                   uint4* __restrict__ frag, int* __restrict__ cell_start) {
  constexpr int SETS = (CH + 1) / 2;
  pdl_wait();
  if ((int)blockIdx.x >= frag_blocks) {
    const int64_t j = (int64_t)(blockIdx.x - frag_blocks) * blockDim.x + threadIdx.x;
    if (j > n_cells) return;
    int lo = 0, hi = n;
    while (lo < hi) {
      const int mid = lo + ((hi - lo) >> 1);
      if (cell_keys[mid] < j) lo = mid + 1; else hi = mid;
    }
    cell_start[j] = lo;
    return;
  }
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t pos = i >> 2;                        // blockDim is a multiple of 32: whole quads
  const int t = (int)(i & 3);
  if ((i >> 5) >= (n + 7) / 8) return;
  const int id = pos < n ? ids[pos] : 0;
  const float* e = emb + (size_t)id * dim;
  if (t == 0 && pos < n) r_s[pos] = x[(size_t)id * x_stride];
  float2 v[SETS];
#pragma unroll
  for (int s = 0; s < SETS; ++s) {
    const int d = 8 * s + 2 * t;
    v[s] = make_float2(pos < n && d < dim ? e[d] : 0.f, pos < n && d + 1 < dim ? e[d + 1] : 0.f);
  }
  float nb = 0.f;
#pragma unroll
  for (int s = 0; s < SETS; ++s) {
    if (pos < n && 8 * s + 2 * t < 4 * CH) emb_s[(size_t)pos * (2 * CH) + 4 * s + t] = v[s];
    nb = fmaf(v[s].x, v[s].x, fmaf(v[s].y, v[s].y, nb));
  }
  nb += __shfl_xor_sync(0xffffffffu, nb, 1);
  nb += __shfl_xor_sync(0xffffffffu, nb, 2);
  const bool wild = !(nb < kFrnnWildNorm), odd = frnn_odd<SETS>(v);
  nb = pos >= n || odd ? -kFrnnWild : wild ? kFrnnWild : nb * (1.0f - kFrnnSlack);
  float q[3];
  frnn_parts(nb, q);
#pragma unroll
  for (int s = 0; s < SETS; ++s) {
    uint4 w;
    if (wild) v[s] = make_float2(0.f, 0.f);
    w.x = frnn_hi(v[s].x, v[s].y);
    w.y = frnn_lo(v[s].x, v[s].y, w.x);
    w.z = s > 0 ? 0u : t == 0 ? pack_bf16x2(1.f, 1.f) : t == 1 ? pack_bf16x2(1.f, q[0]) : t == 2 ? pack_bf16x2(q[1], q[2]) : 0u;
    w.w = 0u;
    frag[((size_t)(i >> 5) * SETS + s) * 32 + (i & 31)] = w;
  }
}

// D = A B + C, bf16 operands, fp32 accumulators.
__device__ __forceinline__ void mma_m16n8k16(float* d, uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                             uint32_t b1, const float* c) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%11,%12,%13};"
      : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(c[0]), "f"(c[1]), "f"(c[2]), "f"(c[3]));
}

__device__ __forceinline__ float frnn_acc(float s, float a, float b) {
  const float d = a - b;
  return __fadd_rn(s, __fmul_rn(d, d));
}

// The pairs of every hit whose chain was kept, written oriented from the smaller r: four threads per hit,
// each a quarter of every chunk's entries (41 -> 26 us on the full event against a thread per hit with
// fifteen gathers at once; 4 pairs a hit).
constexpr int kFrnnCopyLanes = 4;
__global__ void __launch_bounds__(256) frnn_copy_kernel(const float* __restrict__ r_s, int n,
                                                        const int* __restrict__ ids, const int* __restrict__ offsets,
                                                        const int* __restrict__ total, int capacity,
                                                        const int* __restrict__ chunks, int32_t* __restrict__ out) {
  pdl_wait();
  const int64_t i4 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int t = (int)(i4 / kFrnnCopyLanes), q = (int)(i4 % kFrnnCopyLanes);
  if (i4 / kFrnnCopyLanes >= n) return;
  const int n_total = *total;
  if (n_total > capacity || chunks[(size_t)t * kFrnnChunk + kFrnnChunk - 1] == kFrnnLost) return;
  const int pos = offsets[t];
  const int cnt = (t + 1 < n ? offsets[t + 1] : n_total) - pos;
  const int i = ids[t];
  const float ri = r_s[t];
  int cur = t;
  for (int base = 0; base < cnt; base += kFrnnChunk - 1) {
    const int* c = chunks + (size_t)cur * kFrnnChunk;
    const int m = cnt - base < kFrnnChunk - 1 ? cnt - base : kFrnnChunk - 1;
    for (int k = q; k < m; k += kFrnnCopyLanes) {
      const int p = c[k];
      const int jj = ids[p];
      const float rj = r_s[p];
      const bool i_first = ri < rj || (ri == rj && i < jj);
      out[pos + base + k] = i_first ? i : jj;
      out[(size_t)n_total + pos + base + k] = i_first ? jj : i;
    }
    if (base + kFrnnChunk - 1 < cnt) cur = c[kFrnnChunk - 1];
  }
}

// The counting pass of many hits in at most three dimensions, a thread per hit: the runs of its own five cells in
// the 13 rows, every candidate tested exactly, partners kept as frnn_pairs_kernel keeps them (whose writing pass
// takes the hits that lost their chains).  An exact test is twelve operations there, and the filter of
// frnn_pairs_kernel lets much of what it sees through (it is right to about 0.01 between unit vectors, in cells of
// 1/64), so it only pays while threads are too few to fill the GPU.  Builds with the filter / by single hits: 2M
// hits D = 2 33.0 / 14.6 ms, D = 3 1.60 / 1.11; 300,000 hits D = 2 1.08 / 0.63; 100,000 hits D = 1 420 / 251 us,
// D = 2 257 / 199, D = 3 102 / 97; 65,000 hits 244 / 190, 163 / 154, 91 / 91; 16,000 hits D = 3 76 / 80.
// Above three dimensions the filter is ahead on unit vectors at every size (10M hits D = 4 10.2 ms, by single hits,
// with a slower sort, 12.9).  It is behind where hits fill the cube [-1, 1]^4, which an embedding's do not (2M hits
// with 10 edges each 1.81 ms, 1.46; one hit to two cells, no edges, 10M 8.4, 6.4).
constexpr int kFrnnSingleThreads = 128;
constexpr int kFrnnSingleHits = 65536;
__global__ void __launch_bounds__(kFrnnSingleThreads) frnn_single_kernel(
    const float4* __restrict__ emb_s, int n, float r2, int grid, const int* __restrict__ cell_keys,
    const int* __restrict__ cell_start, int* __restrict__ counts, int* __restrict__ chunks, int* __restrict__ next_chunk,
    int max_extra) {
  constexpr int C = kFrnnChunk - 1;                // entries per chunk
  pdl_wait();
  const int t = blockIdx.x * kFrnnSingleThreads + threadIdx.x;
  if (t >= n) return;
  const float4 x = emb_s[t];
  const int key = cell_keys[t], c2 = key % grid, c1 = key / grid % grid, c0 = key / grid / grid;
  const int lo = c2 < kFrnnReach ? 0 : c2 - kFrnnReach, hi = c2 + kFrnnReach >= grid ? grid : c2 + kFrnnReach + 1;
  int found = 0, cur = t, fill = 0;
  bool lost = false;
  chunks[(size_t)t * kFrnnChunk + C] = -1;         // link of the first chunk: none yet
  for (int a = 0; a <= kFrnnReach && c0 + a < grid; ++a)
    for (int b = a == 0 ? 0 : -kFrnnReach; b <= kFrnnReach; ++b) {
      if (c1 + b < 0 || c1 + b >= grid) continue;
      const int row = ((c0 + a) * grid + c1 + b) * grid, p1 = cell_start[row + hi];
      // 32 candidates at a time, so that the loop over them is free of the rare partner's work
      for (int p = a == 0 && b == 0 ? t + 1 : cell_start[row + lo]; p < p1; p += 32) {
        const int m = p1 - p < 32 ? p1 - p : 32;
        uint32_t hits = 0u;
        for (int k = 0; k < m; ++k) {
          const float4 y = emb_s[p + k];
          hits |= (frnn_acc(frnn_acc(frnn_acc(0.f, x.x, y.x), x.y, y.y), x.z, y.z) < r2 ? 1u : 0u) << k;
        }
        for (; hits; hits &= hits - 1) {
          if (fill == C && !lost) {
            const int next = atomicAdd(next_chunk, 1);
            lost = next < 0 || next >= max_extra;
            if (!lost) {
              chunks[(size_t)cur * kFrnnChunk + C] = n + next;
              cur = n + next;
              fill = 0;
            }
          }
          if (!lost) chunks[(size_t)cur * kFrnnChunk + fill++] = p + __ffs(hits) - 1;
          ++found;
        }
      }
    }
  counts[t] = found;
  if (lost) chunks[(size_t)t * kFrnnChunk + C] = kFrnnLost;
}

// A warp searches for sixteen consecutive sorted positions t (its queries).  write == 0: counts[t] =
// pairs visited from t, the partners kept in t's chain; write == 1: the pairs of the hits whose chain
// was lost, at offsets[t] (exclusive scan of counts), when the total fits (frnn_copy_kernel writes the
// others).  chunks: [n + max_extra][kFrnnChunk] ints; chunk t is hit t's first, pool chunks follow
// (next_chunk counts those taken, from zero).
//
// Queries in the same row of cells share their runs: the rows around it, each one contiguous range of
// sorted positions from two cells below the first query's to two above the last one's.  (A run wider
// than a query's own five cells holds no further partners of it, only pairs the exact test turns down.)
// The filter takes the run eight candidates and sixteen queries at a time, 32 candidates between
// votes.  The pairs it lets through wait in a queue, in ascending position for each query, until there
// are 32 for the warp's lanes to test exactly and append to the queries' lists.
//
// The bound is the filter's instructions and the latency of its MMAs: on the full event (D = 8, 2.5e9 pairs
// in the runs, 1.2e6 edges) 22 warp instructions for 128 pairs, two of them MMAs, with 24 warps per SM.  With
// one thread per hit and the exact test on every candidate the search took 24 fp32 operations a pair, 3.2-4.2
// ms; with each block's survivors tested on the spot by the lanes that held them 0.86 ms, queued 0.80, with
// 72 registers instead of 96 (seven blocks per SM) 0.74, and with the four blocks' loads and MMAs side by
// side at six blocks per SM 0.72.  32 queries per warp test more pairs than they save loads (0.77-0.85).
constexpr int kFrnnPairsThreads = 128;
constexpr int kFrnnQueries = 16;
constexpr int kFrnnBlockQueries = kFrnnPairsThreads / 32 * kFrnnQueries;
constexpr int kFrnnQueue = 32 + 8 * kFrnnQueries;                       // below 32 left over, and one block's

template <int CH, int K>
__global__ void __launch_bounds__(kFrnnPairsThreads, 6) frnn_pairs_kernel(
    const float4* __restrict__ emb_s, const uint4* __restrict__ frag, const float* __restrict__ r_s, int n, float r2,
    int grid, const int* __restrict__ cell_keys, const int* __restrict__ ids, const int* __restrict__ cell_start,
    int write, int* __restrict__ counts, const int* __restrict__ total, int capacity, int32_t* __restrict__ out,
    int* __restrict__ chunks, int* __restrict__ next_chunk, int max_extra, uint32_t* err) {
  constexpr int SETS = (CH + 1) / 2;
  constexpr int W = 2 * kFrnnReach + 1;
  constexpr int UNROLL = 4;                                              // blocks of eight candidates per vote
  constexpr unsigned FULL = 0xffffffffu;
  struct Warp {
    int pos[kFrnnQueue];                           // queued pairs: the candidate's sorted position, and
    unsigned char query[kFrnnQueue];               // the query
    int found[kFrnnQueries];                       // per query: partners so far (writing pass: next output slot)
    int cur[kFrnnQueries];                         // the chunk being filled
    int lost[kFrnnQueries];
  };
  __shared__ Warp warps[kFrnnPairsThreads / 32];
  pdl_wait();
  Warp& w = warps[threadIdx.x >> 5];
  const int lane = threadIdx.x & 31, g = lane >> 2, q = lane & 3;
  const unsigned below = (1u << lane) - 1u;
  const int t0 = (blockIdx.x * (kFrnnPairsThreads / 32) + (threadIdx.x >> 5)) * kFrnnQueries;
  if (t0 >= n) return;
  bool want = lane < kFrnnQueries && t0 + lane < n;                     // lane < 16: query t0 + lane is searched for
  int n_total = 0;
  if (write) {
    n_total = *total;
    if (n_total > capacity) {
      if (t0 == 0 && lane == 0) atomicOr(err, DEV_ERR_CAPACITY);
      return;
    }
    want = want && chunks[(size_t)(t0 + lane) * kFrnnChunk + kFrnnChunk - 1] == kFrnnLost;   // the others: frnn_copy_kernel's
    if (__ballot_sync(FULL, want) == 0u) return;
  } else if (want) {
    chunks[(size_t)(t0 + lane) * kFrnnChunk + kFrnnChunk - 1] = -1;   // link of the first chunk: none yet
  }
  if (lane < kFrnnQueries) {
    w.found[lane] = write && want ? counts[t0 + lane] : 0;
    w.cur[lane] = t0 + lane;
    w.lost[lane] = 0;
  }
  __syncwarp();

  // The exact test of the first m <= 32 queued pairs, and the partners to their queries' lists.
  auto drain = [&](int m) {
    int pf = 0, qi = kFrnnQueries;
    bool hit = false;
    if (lane < m) {
      pf = w.pos[lane];
      qi = w.query[lane];
      float s = 0.f;
#pragma unroll
      for (int k = 0; k < CH; ++k) {
        const float4 x = emb_s[(size_t)(t0 + qi) * CH + k], y = emb_s[(size_t)pf * CH + k];
        s = frnn_acc(s, x.x, y.x);
        s = frnn_acc(s, x.y, y.y);
        s = frnn_acc(s, x.z, y.z);
        s = frnn_acc(s, x.w, y.w);
      }
      hit = s < r2;
    }
    if (!__any_sync(FULL, hit)) return;            // usual where the radius is below the filter's resolution
    const unsigned peers = __match_any_sync(FULL, hit ? qi : kFrnnQueries);       // this query's partners
    const int rank = __popc(peers & below), cnt = __popc(peers), leader = __ffs(peers) - 1;
    const int had = hit ? w.found[qi] : 0, at = had + rank;
    int cur = 0;                                   // counting pass: the chunk being filled
    bool gone = false;
    if (write) {
      if (hit) {
        const int i = ids[t0 + qi], jj = ids[pf];
        const float ri = r_s[t0 + qi], rj = r_s[pf];
        const bool i_first = ri < rj || (ri == rj && i < jj);
        out[at] = i_first ? i : jj;
        out[(size_t)n_total + at] = i_first ? jj : i;
      }
    } else {
      constexpr int C = kFrnnChunk - 1;            // entries per chunk
      const int have = had > 0 ? (had - 1) / C : 0;                               // chunks filled or begun, less one
      const int more = hit ? (had + cnt - 1) / C - have : 0;                      // chunks this batch begins
      cur = hit ? w.cur[qi] : 0;
      gone = hit && w.lost[qi];
      int base = 0;
      if (hit && rank == 0 && more > 0 && !gone) {
        base = atomicAdd(next_chunk, more);
        if (base >= 0 && base <= max_extra - more) {
          for (int k = 0, c = cur; k < more; c = n + base + k, ++k) chunks[(size_t)c * kFrnnChunk + C] = n + base + k;
        } else {
          base = -1;
        }
      }
      base = __shfl_sync(FULL, base, leader);
      const bool keep = hit && !gone && base >= 0;
      if (keep) {
        const int k = at / C - have;               // 0: the chunk being filled
        chunks[(size_t)(k == 0 ? cur : n + base + k - 1) * kFrnnChunk + at % C] = pf;
      }
      if (keep && more > 0) cur = n + base + more - 1;
      gone = gone || base < 0;
    }
    __syncwarp();                                  // every lane has read found, cur and lost
    if (hit && rank == 0) {
      w.found[qi] = had + cnt;
      if (!write) {
        w.cur[qi] = cur;
        w.lost[qi] = gone;
      }
    }
    __syncwarp();
  };

  // A fragments of queries g and g + 8: rows r = 0, 1
  uint32_t ah[SETS][2], al[SETS][2], an[2];
  bool tame = true;                                // no query is wild
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    const int t = t0 + g + 8 * r < n ? t0 + g + 8 * r : n - 1;
    float2 v[SETS];
    float na = 0.f;
#pragma unroll
    for (int s = 0; s < SETS; ++s) {
      v[s] = make_float2(0.f, 0.f);
      if (8 * s + 2 * q < 4 * CH) v[s] = reinterpret_cast<const float2*>(emb_s)[(size_t)t * (2 * CH) + 4 * s + q];
      na = fmaf(v[s].x, v[s].x, fmaf(v[s].y, v[s].y, na));
    }
    na += __shfl_xor_sync(FULL, na, 1);
    na += __shfl_xor_sync(FULL, na, 2);
    const bool wild = !(na < kFrnnWildNorm), odd = frnn_odd<SETS>(v);
    tame = tame && !wild;
#pragma unroll
    for (int s = 0; s < SETS; ++s) {
      if (wild) v[s] = make_float2(0.f, 0.f);
      ah[s][r] = frnn_hi(-2.f * v[s].x, -2.f * v[s].y);
      al[s][r] = frnn_lo(-2.f * v[s].x, -2.f * v[s].y, ah[s][r]);
    }
    const float reach = fminf(r2 * (1.0f + 1.0f / 4096.0f) + 1e-35f, 1e29f);
    float u[3];
    frnn_parts(odd ? -kFrnnWild : wild ? kFrnnWild : na * (1.0f - kFrnnSlack) - reach, u);
    an[r] = q == 0 ? pack_bf16x2(u[0], u[1]) : q == 1 ? pack_bf16x2(u[2], 1.f) : q == 2 ? pack_bf16x2(1.f, 1.f) : 0u;
  }

  // Queries by row of cells (their keys ascend, so a row's queries are consecutive).  A row at level v is
  // the cells that agree in all but the last v + 1 gridded coordinates; its runs reach two cells beyond the
  // queries' first of those coordinates and over all of the others.  Level 0 tests the fewest pairs.  Where
  // hits are sparse a warp's queries lie in many rows, each with a search of its own for a handful of
  // candidates; a coarser level then puts them into fewer rows with longer runs.
  const int slot = lane & (kFrnnQueries - 1);
  const int key = cell_keys[t0 + slot < n ? t0 + slot : n - 1];
  const unsigned wanted = __ballot_sync(FULL, want);
  auto groups_at = [&](int d1) {                   // rows among the wanted queries, d1 = cells per row
    const int gid = key / d1, prev = __shfl_up_sync(FULL, gid, 1);
    return __popc(__ballot_sync(FULL, lane == 0 || gid != prev) & wanted) + ((wanted & 1u) ? 0 : 1);
  };
  // the run of this lane's row of cells (o-th at or after the queries' own), for queries first..last
  auto row_run = [&](int level, int d0, int d1, int first, int last, int o, int& p, int& p1) {
    const int gid = __shfl_sync(FULL, key / d1, first);
    const int c_lo = __shfl_sync(FULL, (key / d0) % grid, first) - kFrnnReach;
    const int c_hi = __shfl_sync(FULL, (key / d0) % grid, last) + kFrnnReach;
    p = p1 = 0;
    int rows = 1;
    for (int k = level + 1; k < K; ++k) rows *= W;
    if (o >= (rows + 1) / 2) return;
    int l = rows / 2 + o, rest = gid, row = 0, scale = 1;
    bool in = true;
    for (int k = level + 1; k < K; ++k) {
      const int c = rest % grid + l % W - kFrnnReach;
      in = in && c >= 0 && c < grid;
      row += c * scale;
      rest /= grid; l /= W; scale *= grid;
    }
    if (!in) return;
    const int lo = (c_lo < 0 ? 0 : c_lo) * d0, hi = (c_hi >= grid ? grid : c_hi + 1) * d0;
    p = o == 0 ? t0 + first + 1 : cell_start[row * d1 + lo];
    p1 = cell_start[row * d1 + hi];
  };
  int level = 0, d0 = 1;
  const int cells = __shfl_sync(FULL, key, 31 - __clz(wanted)) - __shfl_sync(FULL, key, __ffs(wanted) - 1);
  if (cells >= 2 && __all_sync(FULL, tame)) {      // (a wild query has every candidate tested: the fewest, then)
    // Two or more cells from the first query to the last.  A coarser level costs its blocks, by the first row's
    // runs; level 0 the time of about eight blocks (of one set of operands) for each run it looks up, however few
    // candidates that has.  Taken when it is cheaper, the finest first.  Builds of unit vectors with half of that
    // for a run, no notice of the sets and only where queries lay in three rows or more -> as it is: 2M hits D = 4
    // 2.04 -> 1.38 ms, D = 6 at small radius 2.20 -> 1.24; 300,000 hits D = 6 380 -> 289 us, D = 12 at small radius
    // 484 -> 328; 30,000 hits D = 8 234 -> 144 us; full event (queries in one cell) 0.74 ms both.  Half as much
    // again for a run: 300,000 hits D = 6 at large radius 574 -> 593 us, 2M 2.21 -> 2.35 ms.
    int runs0 = 1;
    for (int k = 1; k < K; ++k) runs0 *= W;
    const long long fine = 8LL * ((runs0 + 1) / 2) * groups_at(grid);
    for (int v = 1, e0 = grid; v < K; ++v, e0 *= grid) {
      const int e1 = e0 * grid, gs = groups_at(e1);
      const int first = __ffs(wanted) - 1;
      const unsigned same = __ballot_sync(FULL, key / e1 == __shfl_sync(FULL, key / e1, first)) & wanted;
      int p, p1;
      row_run(v, e0, e1, first, 31 - __clz(same), lane, p, p1);
      const int blocks = p < p1 ? (p1 - p) / 8 + 6 : 0;
      if ((long long)gs * (SETS * __reduce_add_sync(FULL, blocks) + 40) < fine) {
        level = v;
        d0 = e0;
        break;
      }
    }
  }
  const int d1 = d0 * grid;
  int rows = 1;
  for (int k = level + 1; k < K; ++k) rows *= W;
  rows = (rows + 1) / 2;
  unsigned todo = wanted;
  int queued = 0;
  while (todo) {
    const int first = __ffs(todo) - 1;
    const unsigned same = __ballot_sync(FULL, key / d1 == __shfl_sync(FULL, key / d1, first)) & todo;
    todo &= ~same;
    const int last = 31 - __clz(same);
    bool member[2];
    uint32_t norm[2];                              // a query of another row: a norm that no radius reaches
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      member[r] = ((same >> (g + 8 * r)) & 1u) != 0u;
      norm[r] = member[r] ? an[r] : q == 0 ? pack_bf16x2(-kFrnnWild, 0.f) : q == 1 ? pack_bf16x2(0.f, 1.f) : an[r];
    }
    for (int base = 0; base < rows; base += 32) {
      int p, p1;                                   // one row of cells per lane: its run of sorted positions
      row_run(level, d0, d1, first, last, base + lane, p, p1);
      for (unsigned runs = __ballot_sync(FULL, p < p1); runs; runs &= runs - 1) {
        const int from = __ffs(runs) - 1;
        const int rp = __shfl_sync(FULL, p, from), rp1 = __shfl_sync(FULL, p1, from);
        const int b1 = (rp1 + 7) >> 3;
        for (int b = rp >> 3; b < b1; b += UNROLL) {
          float c[UNROLL][4];
          uint32_t neg = 0u;                       // sign bits
          uint4 x[UNROLL], y[SETS == 2 ? UNROLL : 1];
#pragma unroll
          for (int u = 0; u < UNROLL; ++u) {
            const int blk = b + u < b1 ? b + u : b1 - 1;             // past the run's end: its last block again
            const uint4* f = frag + (size_t)blk * (32 * SETS) + lane;
            x[u] = f[0];
            if constexpr (SETS == 2) y[u] = f[32];
          }
          const float zero[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
          for (int u = 0; u < UNROLL; ++u) mma_m16n8k16(c[u], ah[0][0], ah[0][1], ah[0][0], ah[0][1], x[u].x, x[u].y, zero);
#pragma unroll
          for (int u = 0; u < UNROLL; ++u) mma_m16n8k16(c[u], al[0][0], al[0][1], norm[0], norm[1], x[u].x, x[u].z, c[u]);
          if constexpr (SETS == 2) {
#pragma unroll
            for (int u = 0; u < UNROLL; ++u) mma_m16n8k16(c[u], ah[1][0], ah[1][1], ah[1][0], ah[1][1], y[u].x, y[u].y, c[u]);
#pragma unroll
            for (int u = 0; u < UNROLL; ++u) mma_m16n8k16(c[u], al[1][0], al[1][1], 0u, 0u, y[u].x, 0u, c[u]);
          }
#pragma unroll
          for (int u = 0; u < UNROLL; ++u) {
            neg |= __float_as_uint(c[u][0]) | __float_as_uint(c[u][1]);
            neg |= __float_as_uint(c[u][2]) | __float_as_uint(c[u][3]);
          }
          if (!__any_sync(FULL, (int)neg < 0)) continue;
#pragma unroll
          for (int u = 0; u < UNROLL; ++u) {
            const uint32_t any = __float_as_uint(c[u][0]) | __float_as_uint(c[u][1]) | __float_as_uint(c[u][2]) |
                                 __float_as_uint(c[u][3]);
            if (b + u >= b1 || !__any_sync(FULL, (int)any < 0)) continue;
            // this block's pairs into the queue, by lane and then by column: ascending for each query
            unsigned ball[4];
            int before = 0;
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const int r = e >> 1, pf = 8 * (b + u) + 2 * q + (e & 1);
              ball[e] = __ballot_sync(FULL, c[u][e] < 0.f && member[r] && pf >= rp && pf < rp1 && pf > t0 + g + 8 * r);
              before += __popc(ball[e] & below);
            }
            int at = queued + before;
#pragma unroll
            for (int e = 0; e < 4; ++e)
              if ((ball[e] >> lane) & 1u) {
                w.pos[at] = 8 * (b + u) + 2 * q + (e & 1);
                w.query[at] = (unsigned char)(g + 8 * (e >> 1));
                ++at;
              }
            queued += __popc(ball[0]) + __popc(ball[1]) + __popc(ball[2]) + __popc(ball[3]);
            __syncwarp();
            while (queued >= 32) {
              drain(32);
              queued -= 32;
              for (int k = lane; k < queued; k += 32) {              // the rest to the front (a lane only
                w.pos[k] = w.pos[32 + k];                            // writes where it alone has read)
                w.query[k] = w.query[32 + k];
              }
              __syncwarp();
            }
          }
        }
      }
    }
  }
  if (queued > 0) drain(queued);
  if (!write && want) {
    counts[t0 + lane] = w.found[lane];
    if (w.lost[lane]) chunks[(size_t)(t0 + lane) * kFrnnChunk + kFrnnChunk - 1] = kFrnnLost;
  }
}

}  // namespace gnn
