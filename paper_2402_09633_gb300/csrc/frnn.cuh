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
// filter that never turns a pair down decides which pairs it is made for.  Each
// pair becomes one edge, oriented from the hit with the smaller r (column 0 of the
// node features, hit id as tie-break).  A counting pass, an exclusive scan of
// the per-hit counts and a writing pass make the output order deterministic: by
// the visiting hit's sorted position, then by row and position of the partner.
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
// row-major with the last gridded coordinate fastest.
template <int K>
__global__ void frnn_cell_kernel(const float* __restrict__ emb, int n, int dim, int grid, int* __restrict__ keys) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float* e = emb + (size_t)i * dim;
  int key = 0;
#pragma unroll
  for (int k = 0; k < K; ++k) key = key * grid + (k < dim ? frnn_coord(e[k], grid) : 0);
  keys[i] = key;
}

// Sorted copies: emb_s [n, 4 * CH] (zero-padded), r_s [n] = x[ids[t], 0].
template <int CH>
__global__ void frnn_gather_kernel(const float* __restrict__ emb, const float* __restrict__ x, int x_stride, int n,
                                   int dim, const int* __restrict__ ids, float4* __restrict__ emb_s,
                                   float* __restrict__ r_s) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  const int i = ids[t];
  const float* e = emb + (size_t)i * dim;
#pragma unroll
  for (int c = 0; c < CH; ++c) {
    float v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = 4 * c + k < dim ? e[4 * c + k] : 0.f;
    emb_s[(size_t)t * CH + c] = make_float4(v[0], v[1], v[2], v[3]);
  }
  r_s[t] = x[(size_t)i * x_stride];
}

// The tensor-core filter of the pair search.  With a = ah + al and b = bh + bl (bf16 parts) and the
// squared norms in three bf16 parts each, one product of K = 32 (dimensions 0-7; 16 more for each of two
// further sets of eight) gives
//   f = (1 - c)(|a|^2 + |b|^2) - 2 (ah bh + ah bl + al bh) - r2',  c = 2^-14, r2' slightly above r2.
// Against the squared distance d the parts left out, the splits' rounding and the accumulation are off
// by less than 3e-5 (|a|^2 + |b|^2) / 2 + 1e-5 (|a|^2 + |b|^2), under half of c (|a|^2 + |b|^2): a pair
// with d < r2 never gives f >= 0.  Pairs with !(f >= 0) (NaN from infinities among them) are tested
// exactly.  K slots: 0-7 -2ah.bh, 8-15 -2ah.bl, 16-23 -2al.bh, 24-26 |a|^2 parts x 1, 27-29 1 x |b|^2 parts.
constexpr float kFrnnSlack = 1.0f / 16384.0f;

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

// B fragments of the sorted hits, eight to a block: lane 4n + t of block b holds, for hit 8b + n and its
// dimensions 2t, 2t + 1 of each set of eight, (bh, bl) and, in the first set, the norm slots.  One uint4
// per lane and set of eight dimensions (.x bh, .y bl, .z norm slots).  Lanes past the last hit get a
// norm that no radius reaches.
template <int CH>
__global__ void frnn_fragments_kernel(const float4* __restrict__ emb_s, int n, uint4* __restrict__ frag) {
  constexpr int SETS = (CH + 1) / 2;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int pos = i >> 2, t = i & 3;                 // blockDim is a multiple of 32: whole quads
  if ((i >> 5) >= (n + 7) / 8) return;
  float2 v[SETS];
  float nb = 0.f;
#pragma unroll
  for (int s = 0; s < SETS; ++s) {
    v[s] = make_float2(0.f, 0.f);
    if (pos < n && 8 * s + 2 * t < 4 * CH)
      v[s] = reinterpret_cast<const float2*>(emb_s)[(size_t)pos * (2 * CH) + 4 * s + t];
    nb = fmaf(v[s].x, v[s].x, fmaf(v[s].y, v[s].y, nb));
  }
  nb += __shfl_xor_sync(0xffffffffu, nb, 1);
  nb += __shfl_xor_sync(0xffffffffu, nb, 2);
  nb = pos < n ? nb * (1.0f - kFrnnSlack) : 1e30f;
  float q[3];
  frnn_parts(nb, q);
#pragma unroll
  for (int s = 0; s < SETS; ++s) {
    uint4 w;
    w.x = frnn_hi(v[s].x, v[s].y);
    w.y = frnn_lo(v[s].x, v[s].y, w.x);
    w.z = s > 0 ? 0u : t == 0 ? pack_bf16x2(1.f, 1.f) : t == 1 ? pack_bf16x2(1.f, q[0]) : t == 2 ? pack_bf16x2(q[1], q[2]) : 0u;
    w.w = 0u;
    frag[((size_t)(i >> 5) * SETS + s) * 32 + (i & 31)] = w;
  }
}

__device__ __forceinline__ void mma_m16n8k16(float* d, uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                             uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ float min_nan(float a, float b) {       // NaN when either is
  float m;
  asm("min.NaN.f32 %0, %1, %2;" : "=f"(m) : "f"(a), "f"(b));
  return m;
}

__device__ __forceinline__ float frnn_acc(float s, float a, float b) {
  const float d = a - b;
  return __fadd_rn(s, __fmul_rn(d, d));
}

// The pairs of every hit whose chain was kept: the partners' sorted positions, read a chunk at a
// time, with their hit ids and r gathered together, written oriented from the smaller r.
__global__ void __launch_bounds__(256) frnn_copy_kernel(const float* __restrict__ r_s, int n,
                                                        const int* __restrict__ ids, const int* __restrict__ offsets,
                                                        const int* __restrict__ total, int capacity,
                                                        const int* __restrict__ chunks, int32_t* __restrict__ out) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  const int n_total = *total;
  if (n_total > capacity || chunks[(size_t)t * kFrnnChunk + kFrnnChunk - 1] == kFrnnLost) return;
  int pos = offsets[t];
  const int cnt = (t + 1 < n ? offsets[t + 1] : n_total) - pos;
  const int i = ids[t];
  const float ri = r_s[t];
  int cur = t;
  for (int base = 0; base < cnt; base += kFrnnChunk - 1) {
    const int4* c4 = reinterpret_cast<const int4*>(chunks + (size_t)cur * kFrnnChunk);
    const int4 w0 = c4[0], w1 = c4[1], w2 = c4[2], w3 = c4[3];
    const int w[kFrnnChunk] = {w0.x, w0.y, w0.z, w0.w, w1.x, w1.y, w1.z, w1.w,
                               w2.x, w2.y, w2.z, w2.w, w3.x, w3.y, w3.z, w3.w};
    const int m = cnt - base;
    int jj[kFrnnChunk - 1];
    float rr[kFrnnChunk - 1];
#pragma unroll
    for (int k = 0; k < kFrnnChunk - 1; ++k) {
      jj[k] = k < m ? ids[w[k]] : 0;
      rr[k] = k < m ? r_s[w[k]] : 0.f;
    }
#pragma unroll
    for (int k = 0; k < kFrnnChunk - 1; ++k) {
      if (k < m) {
        const bool i_first = ri < rr[k] || (ri == rr[k] && i < jj[k]);
        out[pos] = i_first ? i : jj[k];
        out[(size_t)n_total + pos] = i_first ? jj[k] : i;
        ++pos;
      }
    }
    cur = w[kFrnnChunk - 1];
  }
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
// votes; a vote that finds candidates tests them exactly and hands each query's partners, in ascending
// position, to the lane that keeps its list.  One thread per hit with the exact test on every candidate
// took 24 fp32 operations a pair (3.5e9 pairs on the full event, D = 8); the filter takes two MMAs and
// about five other warp instructions for 128 pairs.  The build of the full event: 4.25 -> 1.07 ms, of which
// this kernel takes 0.86.
constexpr int kFrnnPairsThreads = 128;
constexpr int kFrnnQueries = 16;
constexpr int kFrnnBlockQueries = kFrnnPairsThreads / 32 * kFrnnQueries;

template <int CH, int K>
__global__ void __launch_bounds__(kFrnnPairsThreads) frnn_pairs_kernel(
    const float4* __restrict__ emb_s, const uint4* __restrict__ frag, const float* __restrict__ r_s, int n, float r2,
    int grid, const int* __restrict__ cell_keys, const int* __restrict__ ids, const int* __restrict__ cell_start,
    int write, int* __restrict__ counts, const int* __restrict__ total, int capacity, int32_t* __restrict__ out,
    int* __restrict__ chunks, int* __restrict__ next_chunk, int max_extra, uint32_t* err) {
  constexpr int SETS = (CH + 1) / 2;
  constexpr int W = 2 * kFrnnReach + 1;
  constexpr int ROWS = K == 4 ? (W * W * W + 1) / 2 : (W * W + 1) / 2;   // rows at or after the queries' own
  constexpr int UNROLL = 4;                                              // blocks of eight candidates per vote
  constexpr unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31, g = lane >> 2, q = lane & 3;
  const int t0 = (blockIdx.x * (kFrnnPairsThreads / 32) + (threadIdx.x >> 5)) * kFrnnQueries;
  if (t0 >= n) return;
  // lanes 4g and 4g + 1 keep the lists of queries g and g + 8
  const int mine = t0 + g + 8 * (q & 1);
  bool want = q < 2 && mine < n;
  int pos = 0, n_total = 0, i = 0;
  float ri = 0.f;
  if (write) {
    n_total = *total;
    if (n_total > capacity) {
      if (t0 == 0 && lane == 0) atomicOr(err, DEV_ERR_CAPACITY);
      return;
    }
    want = want && chunks[(size_t)mine * kFrnnChunk + kFrnnChunk - 1] == kFrnnLost;   // the others: frnn_copy_kernel's
    if (__ballot_sync(FULL, want) == 0u) return;
    if (want) { pos = counts[mine]; i = ids[mine]; ri = r_s[mine]; }
  } else if (want) {
    chunks[(size_t)mine * kFrnnChunk + kFrnnChunk - 1] = -1;         // link of the first chunk: none yet
  }
  int cur = mine, fill = 0, found = 0;             // counting pass: the chain being filled
  bool lost = false;
  auto take = [&](int p) {                         // a partner of this lane's query
    if (write) {
      const int jj = ids[p];
      const float rj = r_s[p];
      const bool i_first = ri < rj || (ri == rj && i < jj);
      out[pos] = i_first ? i : jj;
      out[(size_t)n_total + pos] = i_first ? jj : i;
      ++pos;
      return;
    }
    ++found;
    if (lost) return;
    if (fill == kFrnnChunk - 1) {
      const int nc = atomicAdd(next_chunk, 1);
      if (nc >= max_extra) { lost = true; return; }
      chunks[(size_t)cur * kFrnnChunk + kFrnnChunk - 1] = n + nc;
      cur = n + nc;
      fill = 0;
    }
    chunks[(size_t)cur * kFrnnChunk + fill++] = p;
  };

  // A fragments of queries g and g + 8: rows r = 0, 1
  uint32_t ah[SETS][2], al[SETS][2], an[2];
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    const int t = t0 + g + 8 * r < n ? t0 + g + 8 * r : n - 1;
    float na = 0.f;
#pragma unroll
    for (int s = 0; s < SETS; ++s) {
      float2 v = make_float2(0.f, 0.f);
      if (8 * s + 2 * q < 4 * CH) v = reinterpret_cast<const float2*>(emb_s)[(size_t)t * (2 * CH) + 4 * s + q];
      na = fmaf(v.x, v.x, fmaf(v.y, v.y, na));
      ah[s][r] = frnn_hi(-2.f * v.x, -2.f * v.y);
      al[s][r] = frnn_lo(-2.f * v.x, -2.f * v.y, ah[s][r]);
    }
    na += __shfl_xor_sync(FULL, na, 1);
    na += __shfl_xor_sync(FULL, na, 2);
    float w[3];
    frnn_parts(na * (1.0f - kFrnnSlack) - (r2 * (1.0f + 1.0f / 4096.0f) + 1e-35f), w);
    an[r] = q == 0 ? pack_bf16x2(w[0], w[1]) : q == 1 ? pack_bf16x2(w[2], 1.f) : q == 2 ? pack_bf16x2(1.f, 1.f) : 0u;
  }
  const float4* ea[2] = {emb_s + (size_t)(t0 + g) * CH, emb_s + (size_t)(t0 + g + 8) * CH};

  // the candidates of one block whose filter value c is not clearly beyond the radius
  auto test_block = [&](const float* c, int blk, int p, int p1, const bool* member) {
    uint32_t hits[2] = {0u, 0u};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int r = e >> 1, pf = 8 * blk + 2 * q + (e & 1);
      if (!(c[e] >= 0.f) && member[r] && pf >= p && pf < p1 && pf > t0 + g + 8 * r) {
        float s = 0.f;
#pragma unroll
        for (int k = 0; k < CH; ++k) {
          const float4 x = ea[r][k], y = emb_s[(size_t)pf * CH + k];
          s = frnn_acc(s, x.x, y.x);
          s = frnn_acc(s, x.y, y.y);
          s = frnn_acc(s, x.z, y.z);
          s = frnn_acc(s, x.w, y.w);
        }
        hits[r] |= (s < r2 ? 1u : 0u) << (2 * q + (e & 1));
      }
    }
#pragma unroll
    for (int r = 0; r < 2; ++r) {                  // the quad's eight candidates of each query
      hits[r] |= __shfl_xor_sync(FULL, hits[r], 1);
      hits[r] |= __shfl_xor_sync(FULL, hits[r], 2);
    }
    if (q < 2)
      for (uint32_t m = hits[q]; m; m &= m - 1) take(8 * blk + __ffs(m) - 1);
  };

  // queries by row of cells (their keys ascend, so a row's queries are consecutive)
  const int key = cell_keys[t0 + (lane & 15) < n ? t0 + (lane & 15) : n - 1];
  const int row = key / grid, cl = key - row * grid;
  const bool wa = __shfl_sync(FULL, want, (lane & 7) * 4 + ((lane >> 3) & 1));      // query lane & 15 is wanted
  unsigned todo = __ballot_sync(FULL, wa && lane < 16);
  while (todo) {
    const int first = __ffs(todo) - 1;
    const int rid = __shfl_sync(FULL, row, first);
    const unsigned same = __ballot_sync(FULL, row == rid) & todo;
    todo &= ~same;
    const int last = 31 - __clz(same);
    const int c_lo = __shfl_sync(FULL, cl, first) - kFrnnReach, c_hi = __shfl_sync(FULL, cl, last) + kFrnnReach;
    const int lo = c_lo < 0 ? 0 : c_lo, hi = c_hi >= grid ? grid - 1 : c_hi;
    const bool member[2] = {((same >> g) & 1u) != 0u, ((same >> (g + 8)) & 1u) != 0u};
    for (int base = 0; base < ROWS; base += 32) {
      // one row of cells per lane: its run of sorted positions
      int p = 0, p1 = 0;
      const int o = base + lane;
      if (o < ROWS) {
        const int l = (K == 4 ? (W * W * W) / 2 : (W * W) / 2) + o;
        int ra, rb, rc = 0, rr;
        bool in;
        if constexpr (K == 4) {
          ra = rid / (grid * grid) + l / (W * W) - kFrnnReach;
          rb = (rid / grid) % grid + (l / W) % W - kFrnnReach;
          rc = rid % grid + l % W - kFrnnReach;
          in = ra < grid && rb >= 0 && rb < grid && rc >= 0 && rc < grid;
          rr = (ra * grid + rb) * grid + rc;
        } else {
          ra = rid / grid + l / W - kFrnnReach;
          rb = rid % grid + l % W - kFrnnReach;
          in = ra < grid && rb >= 0 && rb < grid;
          rr = ra * grid + rb;
        }
        if (in) {
          p = o == 0 ? t0 + first + 1 : cell_start[rr * grid + lo];
          p1 = cell_start[rr * grid + hi + 1];
        }
      }
      for (unsigned runs = __ballot_sync(FULL, p < p1); runs; runs &= runs - 1) {
        const int from = __ffs(runs) - 1;
        const int rp = __shfl_sync(FULL, p, from), rp1 = __shfl_sync(FULL, p1, from);
        const int b1 = (rp1 + 7) >> 3;
        for (int b = rp >> 3; b < b1; b += UNROLL) {
          float c[UNROLL][4];
          float m = 0.f;
#pragma unroll
          for (int u = 0; u < UNROLL; ++u) {
            const int blk = b + u < b1 ? b + u : b1 - 1;             // past the run's end: its last block again
            const uint4* f = frag + (size_t)blk * (32 * SETS) + lane;
            const uint4 w = f[0];
#pragma unroll
            for (int e = 0; e < 4; ++e) c[u][e] = 0.f;
            mma_m16n8k16(c[u], ah[0][0], ah[0][1], ah[0][0], ah[0][1], w.x, w.y);
            mma_m16n8k16(c[u], al[0][0], al[0][1], an[0], an[1], w.x, w.z);
            if constexpr (SETS == 2) {
              const uint4 w2 = f[32];
              mma_m16n8k16(c[u], ah[1][0], ah[1][1], ah[1][0], ah[1][1], w2.x, w2.y);
              mma_m16n8k16(c[u], al[1][0], al[1][1], 0u, 0u, w2.x, 0u);
            }
            m = min_nan(m, min_nan(min_nan(c[u][0], c[u][1]), min_nan(c[u][2], c[u][3])));
          }
          if (__any_sync(FULL, !(m >= 0.f))) {
#pragma unroll
            for (int u = 0; u < UNROLL; ++u) {
              const float mu = min_nan(min_nan(c[u][0], c[u][1]), min_nan(c[u][2], c[u][3]));
              if (b + u < b1 && __any_sync(FULL, !(mu >= 0.f))) test_block(c[u], b + u, rp, rp1, member);
            }
          }
        }
      }
    }
  }
  if (!write && want) {
    counts[mine] = found;
    if (lost) chunks[(size_t)mine * kFrnnChunk + kFrnnChunk - 1] = kFrnnLost;
  }
}

}  // namespace gnn
