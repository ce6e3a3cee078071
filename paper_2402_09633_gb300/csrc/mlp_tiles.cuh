// Fused MLP-tile kernels of the interaction network (tcgen05 / TMEM, sm_103a).
//
// One persistent CTA per SM walks 128-row tiles (edges in destination-sorted
// CSR order, or nodes).  Each tile runs a fixed program of "jobs": a job is one
// Linear layer D = A * W^T executed on the 5th-generation tensor cores with
// the activation tile A in tensor memory and the weight W in shared memory,
// followed by an epilogue in registers (bias or gathered projections,
// LayerNorm, ReLU) that writes the next layer's A back into tensor memory.
//
// Precision (template parameter BF):
//   * fp32 model (BF = false): fp32 weights and states; every product is
//     evaluated as hi*hi + hi*lo + lo*hi of bf16 splits (v = hi + lo, both bf16)
//     with fp32 accumulation, which keeps the relative product error near 2^-16;
//   * bf16 model (BF = true): bf16 weights, bf16 activations and stored states
//     (e, h, a), one bf16 product per K step, fp32 accumulation and fp32
//     LayerNorm; the first-layer projections P_s, P_d stay fp32 (they are
//     partial sums of one Linear layer).
//
// Organisation (one CTA per SM):
//   * NG worker groups of eight warps: three for the edge kernels, the edge encoder, the filter and the
//     embedding (72 registers a thread), two for the node kernels (96).  The issuing warp costs each worker
//     registers: 25 warps put seven on one of the SM's four schedulers, 17 put five, and ptxas shares out
//     its 16,384 registers by that.  The edge kernels spill 8 to 72 bytes at 72.  A group owns a tile at a time;
//     a warp owns 16 rows of it, a quad of threads shares two rows (each thread a quarter of the
//     columns), reads them from tensor memory with the 16-lane shapes and does the gathers, LayerNorm
//     and ReLU in registers, in packed fp32 pairs;
//   * tensor memory is cut into regions of H columns.  A region holds either a tile's D (H fp32 columns)
//     or its A operand: the epilogue reads D 32 columns at a time and writes A's bf16 hi and lo words
//     over the columns it has just read.  A tile so needs one region between jobs and two while a job
//     runs, and three tiles are in flight where fixed D and A columns for every tile allow two;
//   * biases are added by the tensor core: a job starts with D = ones * bias^T, one MMA of a K step, so
//     the epilogues read one vector less twice over.  The fp32 model's hidden layers need no gamma
//     either (the host folds it into the weights), which leaves beta;
//   * warp 0 issues the MMAs of whichever group has published its next A operand (24 tcgen05.mma and the
//     bias per layer; the warp runs in step, one elected lane issues: 0.7-0.8 us per layer against 1.3
//     from a lone lane, whose operands are moved to uniform registers one by one) and commits them to
//     the group's mbarrier; it also loads the weights with bulk copies (all at once, or streamed through
//     a ring of stages);
//   * one worker thread per group warms L2 (bulk prefetch) with the group's next tile.
//
// What bounds them (full event, 300k nodes / 1M edges, H = 128, L = 3): the chain of a tile, about 14 us
// for an edge update (edge state to A, gathers next to the layer-1 job, three epilogues, two more jobs of
// 0.7-0.8 us with their queueing, store), with three chains in flight: tensor pipe 47 % active, DRAM
// 54 %, issue 32 %.  Per launch, against two tiles in flight, biases and gammas in the
// epilogues and first layers on CUDA cores, fp32 / bf16 model: edge update 0.392 -> 0.288 / 0.313 -> 0.209
// ms, node update 0.193 -> 0.163 / 0.140 -> 0.118, classifier 0.373 -> 0.262 / 0.331 -> 0.216, edge encoder
// 0.284 -> 0.192 / 0.219 -> 0.150, node encoder 0.166 -> 0.114 / 0.139 -> 0.101; embedding of 300k hits
// 0.204 -> 0.078, filter on 1.9M edges 0.90 -> 0.344; the gammas' part in it is 0.5 to 0.8 % of a call.  Measured and not taken, in the edge update as it
// was at 0.32 ms: one thread per row and four warps per group (every thread then reads every parameter:
// 0.547 with shared memory, 0.371 through the constant cache); two groups with 104 registers (0.350);
// gathers of one or three 32-column chunks before the layer-1 wait instead of two (0.328, 0.342).
#pragma once
#include <climits>
#include <cstdint>
#include <type_traits>
#include <cuda_bf16.h>
#include "ptx.cuh"

namespace gnn {

enum class TileKind : int {
  NodeEncoder = 0,     // x -> h0, then P_s, P_d projections
  EdgeEncoder = 1,     // (dr, dphi) -> e0
  EdgeUpdate  = 2,     // e <- MLP_edge([h_src, h_dst, e]) via e*W_e + P_s[src] + P_d[dst]
  NodeUpdate  = 3,     // h <- MLP_node([h, sum of incoming e]); then P_s, P_d of new h
  Classifier  = 4,     // score = sigmoid(w_o . MLP_cls([h_src, h_dst, e]) + b_o)
  Filter      = 5,     // filtering step: score = sigmoid(w_o . MLP_f([x_src, x_dst]) + b_o), input edge order
  Embed       = 6,     // embedding step: y = normalize(W_out . MLP_emb(x) + b_out), D outputs per hit
};

constexpr int kMaxEmbedDim = 16;
constexpr int kTileRows = 128;
constexpr int kMaxJobs = 8;

// Kinds whose first job multiplies raw inputs (features, at most 32 of them).
__host__ __device__ constexpr bool has_input_job(TileKind k) {
  return k == TileKind::NodeEncoder || k == TileKind::EdgeEncoder || k == TileKind::Filter || k == TileKind::Embed;
}

// Worker groups and threads of a kernel: one warp that issues, and eight per group.
template <TileKind KIND>
struct TileRoles {
  static constexpr int NG = (KIND == TileKind::NodeEncoder || KIND == TileKind::NodeUpdate) ? 2 : 3;
  static constexpr int THREADS = 32 + 256 * NG;      // 800 (72 registers each) or 544 (96)
};

struct TileParams {
  int n_rows;                 // rows of this kernel: edges (E) or nodes (N)
  int n_tiles;
  int n_nodes;
  int n_layers;               // Linear layers per MLP (L)
  int n_feat;                 // node features (F_n)
  int n_in;                   // inputs of the first job of a kind with one (F_n, 2 or 2 F_n)
  int n_jobs;
  int job_mat[kMaxJobs];      // matrix index (into wmats) of each MMA job
  int job_acc[kMaxJobs];      // 1: accumulate into D (second half of a split layer 1)
  int job_areg[kMaxJobs];     // two groups: which of the group's two regions holds A (D is the other)
  int job_bias[kMaxJobs];     // bias tile (1-based, into consts) that the job's D starts from; 0: none
  int early;                  // 1: a small grid, let the next kernel start on the idle SMs (see pdl_trigger)
  int folded;                 // 1: gamma of every layer but the MLP's last is folded into the weights around it
  const uint8_t* consts;      // the ones tile, then the bias tiles (128 and H rows x 16 bf16, see gnn_api.cu)
  uint32_t const_bytes;
  uint32_t ring_bytes;        // weight ring (a stage per job where all jobs' weights fit)
  const uint8_t* wmats;       // packed matrices, mat_bytes apart (hi part then lo part)
  uint32_t mat_bytes;
  const float* vecs;          // per-kernel fp32 parameter vectors (layout per kind)
  int n_vec_floats;
  float eps;
  // graph data
  const float* x;             // [N, n_feat_total] node features
  int x_stride;
  const int* src_sorted;      // [E] source of CSR slot k
  const int* dst_sorted;      // [E] destination of CSR slot k (clamped to a valid id)
  const int* key_sorted;      // [E] destination key (== n_nodes for an invalid edge)
  const int* perm;            // [E] input edge id of CSR slot k
  const int* rowptr;          // [N+1]
  void* e;                    // [E, H] edge state, CSR order (updated in place); fp32 or bf16
  void* h;                    // [N, H] node state; fp32 or bf16
  float* ps;                  // [N, H] projections W_s h
  float* pd;                  // [N, H] projections W_d h + b1
  void* agg;                  // [N, H] row-tiled: sum of incoming messages per node; fp32 or bf16
  float* scores;              // [E] input order
  uint32_t* err;              // device error word
  const int32_t* ei_in;       // filter: [2, E] input edge index (rows in input order)
  float* emb;                 // embedding: [N, emb_dim] output
  int emb_dim;
#ifdef GNN_TRACE
  unsigned long long* trace;  // [3 roles][kTraceEvents] %globaltimer stamps of CTA 0
#endif
};

#ifdef GNN_TRACE
constexpr int kTraceEvents = 512;
#define GNN_TRACE_AT(role, idx)                                                               \
  do {                                                                                        \
    if (p.trace && blockIdx.x == 0 && (idx) < kTraceEvents) p.trace[(role) * kTraceEvents + (idx)] = global_timer_ns(); \
  } while (0)
#define GNN_TRACE_CTA(k)                                                                      \
  do {                                                                                        \
    if (p.trace && threadIdx.x == 0 && blockIdx.x < kTraceEvents / 2) p.trace[2 * kTraceEvents + 2 * blockIdx.x + (k)] = global_timer_ns(); \
  } while (0)
#define GNN_TRACE_W(label)                                                                    \
  do {                                                                                        \
    if (warp == 1 && lane == 0) GNN_TRACE_AT(1, tr_iter * 16 + (label));                      \
  } while (0)
#else
#define GNN_TRACE_AT(role, idx) do { } while (0)
#define GNN_TRACE_CTA(k) do { } while (0)
#define GNN_TRACE_W(label) do { } while (0)
#endif

template <int H, bool BF>
struct TileGeom {
  static constexpr int NCH = H / 32;                // 32-column chunks of a row
  static constexpr int TMEM_COLS = 512;
  static constexpr int NREG = TMEM_COLS / H;        // regions: 4 (H = 128) or 8 (H = 64)
  static constexpr uint32_t PART_BYTES = H * H * 2; // one bf16 H x H matrix part
  static constexpr uint32_t MAT_BYTES = BF ? PART_BYTES : 2 * PART_BYTES;  // hi [+ lo]
  static constexpr int STAGES = (192u * 1024u / MAT_BYTES) < 8 ? (192u * 1024u / MAT_BYTES) : 8;  // weight ring, at most
  static constexpr uint32_t IDESC = idesc_bf16_f32(128, H);
  static constexpr uint32_t ONES_BYTES = 128 * 32;  // 128 rows x 16 bf16
  static constexpr uint32_t BIAS_BYTES = H * 32;    // H rows x 16 bf16
};

// Byte offset of part w (0 hi, 1 mid, 2 lo) of an input matrix [H, 32] inside a weight block: parts 32 K
// elements apart along the block's K, the third in its own 64-column chunk.
template <int H>
__host__ __device__ constexpr uint32_t input_part_offset(int w) {
  return w < 2 ? 64u * w : (H == 128 ? H * 128u : TileGeom<H, false>::PART_BYTES);
}

// Parameter vectors are padded to 16 bytes so the mbarriers after them stay 8-byte aligned.
__host__ __device__ constexpr int padded_vec_floats(int n) { return (n + 3) & ~3; }

// Stages of a kernel's weight ring, at most; weights that need no more stay resident.  The node kernels of
// H = 128 stream their five to seven blocks through a shorter ring than would fit (two blocks in fp32, four in
// bf16): the L1 that it leaves is worth more (node update 0.179 -> 0.170 ms and 0.127 -> 0.118; a bf16 ring of
// five or three 0.127).  So is the fp32 edge update's and classifier's, whose gathers need it (three resident
// blocks 0.319 and 0.291 ms, two streamed 0.298 and 0.265; mid event 704 -> 670 us); the kernels without
// gathers keep three resident (filter 0.344, two streamed 0.366).  Stages of half a block (hi and lo parts
// apart) were slower at every depth (0.303-0.331).
template <TileKind KIND, int H, bool BF>
constexpr int tile_max_stages() {
  constexpr int most = TileGeom<H, BF>::STAGES;
  if (H == 128 && (KIND == TileKind::NodeUpdate || KIND == TileKind::NodeEncoder)) return BF ? 4 : 2;
  if (H == 128 && !BF && (KIND == TileKind::EdgeUpdate || KIND == TileKind::Classifier)) return 2;
  return most;
}
// Stages taken: one per job where they all fit, no more.  Shared memory that is not taken is L1: next to the
// full 192 KB it has about 230 lines left, too few for the loads that the worker warps have in flight (bf16
// edge update 0.240 -> 0.210 ms with 96 KB of weights instead of a 192 KB ring).  The fp32 kernels of H = 128
// need the full ring for three layers; they keep it, at a fixed offset, for two (a computed offset costs the
// edge update spills: 0.318 -> 0.338).
template <TileKind KIND, int H, bool BF>
constexpr int tile_stages(int n_jobs) {
  constexpr int most = tile_max_stages<KIND, H, BF>();
  return n_jobs < most && !(H == 128 && !BF) ? n_jobs : most;
}

template <int H, bool BF>
constexpr uint32_t tile_smem_bytes(int stages, int n_vec_floats, uint32_t const_bytes) {
  // ring (1024-aligned) + ones and bias tiles + vectors + barriers + alignment slack
  return stages * TileGeom<H, BF>::MAT_BYTES + const_bytes + (uint32_t)padded_vec_floats(n_vec_floats) * 4u + 320 + 1024;
}

// Launch geometry: dynamic shared memory of at least 120 KB, so that one CTA per SM runs (it owns
// the TMEM), and one persistent CTA per SM or per tile, whichever is fewer.  CTA b takes tiles b,
// b + grid, b + 2 grid, ...; its groups take them in turn.
template <int H, bool BF>
constexpr uint32_t tile_launch_smem(int stages, int n_vec_floats, uint32_t const_bytes) {
  const uint32_t b = tile_smem_bytes<H, BF>(stages, n_vec_floats, const_bytes);
  return b < 120u * 1024u ? 120u * 1024u : b;
}
inline int tile_grid(int n_tiles, int n_sm) { return n_tiles < n_sm ? n_tiles : n_sm; }

__device__ __forceinline__ float2 f2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 lo2(const float4& v) { return make_float2(v.x, v.y); }
__device__ __forceinline__ float2 hi2(const float4& v) { return make_float2(v.z, v.w); }
__device__ __forceinline__ float2 relu2(float2 v) { return make_float2(fmaxf(v.x, 0.f), fmaxf(v.y, 0.f)); }
__device__ __forceinline__ float2 round_bf16x2(float2 v) {
  return __bfloat1622float2(__floats2bfloat162_rn(v.x, v.y));
}
// ----------------------------------------------------------------- kernel
template <TileKind KIND, int H, bool BF>
__global__ void __launch_bounds__(TileRoles<KIND>::THREADS, 1) mlp_tile_kernel(const TileParams p) {
  using G = TileGeom<H, BF>;
  using SE = typename std::conditional<BF, __nv_bfloat16, float>::type;   // stored state element
  using R = TileRoles<KIND>;
  constexpr int NG = R::NG;
  constexpr int NCH = G::NCH;
  constexpr int STAGES = tile_max_stages<KIND, H, BF>();
  constexpr int NSPARE = G::NREG - NG;               // regions no group owns (three groups)
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* ring = smem;
  uint8_t* consts = smem + (H == 128 && !BF ? STAGES * G::MAT_BYTES : p.ring_bytes);
  float* vecs = reinterpret_cast<float*>(consts + p.const_bytes);
  uint64_t* bars = reinterpret_cast<uint64_t*>(vecs + padded_vec_floats(p.n_vec_floats));
  uint64_t* a_full = bars;                           // [3]  a group's eight warps published A
  uint64_t* d_full = bars + 3;                       // [3]  MMA of a group's current job completed
  uint64_t* spare_free = bars + 6;                   // [8]  the job that gave a spare region back completed
  uint64_t* c_full = bars + 14;                      // the constant tiles are loaded
  uint64_t* w_full = bars + 15;                      // [STAGES]  weight stage loaded
  uint64_t* w_empty = bars + 15 + STAGES;         // [STAGES]  all groups' MMAs on a stage completed
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 15 + 2 * STAGES);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  volatile int* d_region = abort_flag + 1;           // [3]  three groups: the region of a group's current D

  const int warp = uniform((int)threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  const bool resident = p.n_jobs <= STAGES;
  const int n_my = (p.n_tiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;   // this CTA's tiles
  const int n_rounds = (n_my + NG - 1) / NG;

  for (int i = threadIdx.x; i < p.n_vec_floats; i += R::THREADS) vecs[i] = p.vecs[i];
  if (threadIdx.x == 0) {
    for (int g = 0; g < NG; ++g) {
      mbar_init(&a_full[g], 8);
      mbar_init(&d_full[g], NG == 3 ? 2 : 1);        // three groups: the commit, and the issuer's region word
    }
    for (int s = 0; s < 8; ++s) mbar_init(&spare_free[s], 1);
    for (int s = 0; s < STAGES; ++s) { mbar_init(&w_full[s], 1); mbar_init(&w_empty[s], NG); }
    mbar_init(c_full, 1);
    *abort_flag = 0;
    fence_mbar_init();
    mbar_arrive_expect_tx(c_full, p.const_bytes);
    bulk_g2s(consts, p.consts, p.const_bytes, c_full);
    if (resident) {                                    // the weights are constant: load them at once
      mbar_arrive_expect_tx(&w_full[0], (uint32_t)p.n_jobs * G::MAT_BYTES);
      for (int j = 0; j < p.n_jobs; ++j)
        bulk_g2s(ring + j * G::MAT_BYTES, p.wmats + (size_t)p.job_mat[j] * p.mat_bytes, G::MAT_BYTES, &w_full[0]);
    }
  }
  if (warp == 0) { tmem_alloc(tmem_slot, G::TMEM_COLS); tmem_relinquish(); }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = (uint32_t)uniform((int)*tmem_slot);
  // Everything above (parameter vectors, barriers, tensor memory, the resident weights) depends on
  // no earlier kernel, so under a programmatic dependent launch it overlaps the previous kernel's
  // exit; from here on every thread may read what that kernel wrote.
  pdl_wait();
  if (p.early) pdl_trigger();
  GNN_TRACE_CTA(0);

  if (warp == 0) {
    // ------------------------------------------------ MMA issuer
    // The groups advance independently: each has its own job cursor, and the issuer serves
    // whichever has published its next A operand.  Three groups: a job writes D into a spare
    // region, and the region its A was in is spare once it has completed; the spares are taken in
    // the order they were given back, each with the mbarrier of the job that gave it back.  Two
    // groups: each has two regions of its own, and job_areg says which holds A.
    // In streamed-weight mode all groups walk the same (round, job) sequence of ring stages; a
    // stage is released after every group's MMAs on it completed (w_empty counts NG commits; a
    // group without a tile in the last round is covered by further commits of group 0).
    // The whole warp runs the loop in step, so that addresses and descriptors stay in uniform
    // registers; one elected lane issues.
    int i_g[NG], job_g[NG];
    uint32_t seq_g[NG], a_par[NG], reg_g[NG];
#pragma unroll
    for (int g = 0; g < NG; ++g) {
      i_g[g] = g; job_g[g] = 0; seq_g[g] = 0; a_par[g] = 0; reg_g[g] = g;
    }
    uint32_t spares = 0;                             // three groups: 4 bits per spare region
    if constexpr (NG == 3)
      for (int k = 0; k < NSPARE; ++k) spares |= (uint32_t)(NG + k) << (4 * k);
    uint32_t sp = 0, sp_uses = 0;                    // next spare, and how often the ring of spares was walked
    bool ok = warp_all(bounded_wait(c_full, 0, abort_flag, p.err));
    if (ok && resident) ok = warp_all(bounded_wait(&w_full[0], 0, abort_flag, p.err));
    uint32_t loaded = 0;                             // streamed weights: stages loaded so far
    const uint32_t to_load = resident ? 0 : (uint32_t)(n_rounds * p.n_jobs);
    uint64_t t_last = global_timer_ns();
    uint32_t spins = 0;
    int live = n_my < NG ? n_my : NG;
    while (ok && live > 0) {
      bool progressed = false;
      if (loaded < to_load) {
        const int st = loaded % STAGES;
        if (loaded < (uint32_t)STAGES || warp_all(mbar_test_wait(&w_empty[st], ((loaded / STAGES) - 1) & 1))) {
          const uint8_t* src = p.wmats + (size_t)p.job_mat[loaded % p.n_jobs] * p.mat_bytes;
          if (elect_one()) {
            mbar_arrive_expect_tx(&w_full[st], G::MAT_BYTES);
            bulk_g2s(ring + st * G::MAT_BYTES, src, G::MAT_BYTES, &w_full[st]);
          }
          __syncwarp();
          ++loaded;
          progressed = true;
        }
      }
#pragma unroll
      for (int g = 0; g < NG; ++g) {
        if (i_g[g] >= n_my) continue;
        const int j = job_g[g];
        const int st = resident ? j : (int)(seq_g[g] % STAGES);
        if (!resident && !warp_all(mbar_test_wait(&w_full[st], (seq_g[g] / STAGES) & 1))) continue;
        if (!warp_all(mbar_test_wait(&a_full[g], a_par[g]))) continue;
        a_par[g] ^= 1;
        uint32_t ra, rd;
        if constexpr (NG == 3) {
          if (sp_uses > 0 && !warp_all(bounded_wait(&spare_free[sp], (sp_uses - 1) & 1, abort_flag, p.err))) { ok = false; break; }
          ra = reg_g[g];
          rd = (spares >> (4 * sp)) & 15u;
          spares = (spares & ~(15u << (4 * sp))) | (ra << (4 * sp));
          reg_g[g] = rd;
        } else {
          ra = 2 * g + p.job_areg[j];
          rd = 2 * g + 1 - p.job_areg[j];
        }
        const uint32_t wb = smem_u32(ring + st * G::MAT_BYTES);
        const uint32_t d = tmem_base + rd * H, a = tmem_base + ra * H;
        const uint64_t bh0 = sdesc_kmajor_sw128(wb), bl0 = sdesc_kmajor_sw128(wb + G::PART_BYTES);
        const int bias = p.job_bias[j];
        const uint32_t acc0 = (p.job_acc[j] || bias) ? 1u : 0u;
        const uint64_t ones = sdesc_kmajor_plain(smem_u32(consts));
        const uint64_t bdesc = sdesc_kmajor_plain(smem_u32(consts) + G::ONES_BYTES + (bias ? bias - 1 : 0) * G::BIAS_BYTES);
        // covers for groups without a tile in the last round, at the streamed weights' stage
        const int covers = (!resident && g == 0 && i_g[0] + NG > n_my) ? i_g[0] + NG - n_my : 0;
        tc_fence_after();
        if (elect_one()) {
          GNN_TRACE_AT(0, 2 * (int)seq_g[g] + g * 160);
          if constexpr (NG == 3) {
            d_region[g] = (int)rd;
            mbar_arrive(&d_full[g]);
          }
          if (bias) mma_bf16_ss(d, ones, bdesc, G::IDESC, p.job_acc[j] ? 1u : 0u);   // D = 1 * bias^T
          bool input = false;
          if constexpr (has_input_job(KIND)) {
            // Raw inputs: A holds x = hi + mid + lo in three bf16 parts of up to 32 elements, 16 columns
            // apart; W likewise (one part in the bf16 model).  Products down to 2^-24 of the largest.
            input = j == 0;
            for (int ks = 0; input && ks < (p.n_in + 15) / 16; ++ks) {
              constexpr int PAIR[6][2] = {{0, 0}, {1, 0}, {2, 0}, {0, 1}, {1, 1}, {0, 2}};
#pragma unroll
              for (int q = 0; q < (BF ? 3 : 6); ++q) {
                const uint64_t off = (input_part_offset<H>(PAIR[q][1]) + ks * 32) >> 4;
                mma_bf16_ts(d, a + 16 * PAIR[q][0] + 8 * ks, bh0 + off, G::IDESC, 1u);
              }
            }
          }
#pragma unroll
          for (int ks = 0; !input && ks < H / 16; ++ks) {
            const uint64_t off = ((ks >> 2) * (H * 128) + (ks & 3) * 32) >> 4;
            const uint32_t ahi = a + (ks >> 1) * 32 + (ks & 1) * 8, alo = ahi + 16;
            mma_bf16_ts(d, ahi, bh0 + off, G::IDESC, ks > 0 ? 1u : acc0);
            if constexpr (!BF) {
              mma_bf16_ts(d, ahi, bl0 + off, G::IDESC, 1u);
              mma_bf16_ts(d, alo, bh0 + off, G::IDESC, 1u);
            }
          }
          mma_commit(&d_full[g]);
          if constexpr (NG == 3) mma_commit(&spare_free[sp]);
          if (!resident)
            for (int k = 0; k <= covers; ++k) mma_commit(&w_empty[st]);
          GNN_TRACE_AT(0, 2 * (int)seq_g[g] + 1 + g * 160);
        }
        __syncwarp();
        if constexpr (NG == 3)
          if (++sp == NSPARE) { sp = 0; ++sp_uses; }
        seq_g[g]++;
        if (++job_g[g] == p.n_jobs) {
          job_g[g] = 0;
          i_g[g] += NG;
          if (i_g[g] >= n_my) --live;
        }
        progressed = true;
      }
      if (progressed) {
        t_last = global_timer_ns();
        spins = 0;
      } else if ((++spins & 63u) == 0) {
        if (!warp_all(*abort_flag == 0)) break;
        if (!warp_all(global_timer_ns() - t_last <= kWaitLimitNs)) {
          if (lane == 0) atomicOr(p.err, DEV_ERR_TIMEOUT);
          *abort_flag = 1;
          break;
        }
      }
    }
    // Before teardown (and the TMEM release), every commit has arrived, not only the one of the same MMAs that
    // the workers wait for: an arrival after the block's exit could meet the next block's shared memory ...
#pragma unroll
    for (int g = 0; g < NG; ++g)
      if (seq_g[g] > 0) drain_wait(&d_full[g], (seq_g[g] - 1) & 1);
    if constexpr (NG == 3)
      for (uint32_t k = 0; k < (uint32_t)NSPARE; ++k)
        if (const uint32_t uses = sp_uses + (k < sp ? 1u : 0u)) drain_wait(&spare_free[k], (uses - 1) & 1);
    // ... and so has every weight copy (the last one per stage, and the release of its stage)
    drain_wait(c_full, 0);
    if (resident) drain_wait(&w_full[0], 0);
    for (uint32_t k = loaded > (uint32_t)STAGES ? loaded - STAGES : 0u; k < loaded; ++k) {
      drain_wait(&w_full[k % STAGES], (k / STAGES) & 1);
      drain_wait(&w_empty[k % STAGES], (k / STAGES) & 1);
    }
    __syncwarp();
  } else {
    // Worker groups: eight warps to a group, sixteen rows of its tile to a warp (half of a tensor-memory
    // lane quarter).  A quad of threads shares rows r0 = lane/4 and r0 + 8 of the warp's sixteen; thread
    // q = lane % 4 of it holds columns 8b + 2q and 8b + 2q + 1 of every 8-column block b.
    const int wq = warp - 1;
    const int grp = wq >> 3;
    const int quarter = warp & 3;              // TMEM lane quarter of this warp
    const int lane0 = quarter * 32 + ((wq >> 2) & 1) * 16;
    const int trow = lane0 + (lane >> 2);      // this thread's first row inside the tile; the second is trow + 8
    const int q4 = 4 * (lane & 3), q8 = 8 * (lane & 3);
    const bool leader = (wq & 7) == 0 && lane == 0;
    const uint32_t lane_base = tmem_base + ((uint32_t)lane0 << 16);
    uint32_t a_reg = lane_base + (NG == 3 ? grp : 2 * grp) * H;     // where this group's next A goes
    uint32_t d_reg = a_reg;
    uint32_t d_use = 0;
#ifdef GNN_TRACE
    int tr_iter = 0;
#endif
    int j = 0;                                 // job index inside the tile
    bool ok = true;

    auto publish = [&]() {                     // the A operand of job j is in place
      tmem_st_wait();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&a_full[grp]);
    };
    auto wait_job = [&]() {                    // job j's D is there; never early-exits a tile
      ok &= warp_all(bounded_wait(&d_full[grp], d_use & 1, abort_flag, p.err));
      d_use++;
      tc_fence_after();
      if constexpr (NG == 3) {
        d_reg = lane_base + (uint32_t)uniform(d_region[grp] & (G::NREG - 1)) * H;
        a_reg = d_reg;                         // the next A is written over D
      } else {
        d_reg = lane_base + (2 * grp + 1 - p.job_areg[j]) * H;
        a_reg = lane_base + (2 * grp + (j + 1 < p.n_jobs ? p.job_areg[j + 1] : p.job_areg[0])) * H;
      }
      ++j;
    };
    auto quad_sum = [&](float x) {
      x += __shfl_xor_sync(0xffffffffu, x, 1);
      x += __shfl_xor_sync(0xffffffffu, x, 2);
      return x;
    };
    // Row data, 32 columns (four blocks) at a time: t[2b] holds the pair of block b of row trow,
    // t[2b + 1] that of row trow + 8.
    //   row-tiled state "T16" (e, h, a): (r, c) at ((r/128)*(H/16) + c/16)*2048 + (r%128)*16 + x,
    //     x = 4*((c%8)/2) + 2*((c/8)%2) + c%2: a quad thread's pairs of two blocks are 16 (fp32) or 8
    //     (bf16) contiguous bytes, and a warp reads eight whole rows of 64 (32) bytes in a piece;
    //   row-major "RM32" (P_s, P_d, fp32): (r, c) at r*H + (c/32)*32 + 8*((c%8)/2) + 2*((c/8)%4) + c%2:
    //     a quad thread's pairs of four blocks are 32 contiguous bytes, a gathered row a whole line.
    auto t16 = [&](const void* base, int row, int bp) -> const SE* {
      return static_cast<const SE*>(base) + (((size_t)(row >> 7) * (H / 16) + bp) * 128 + (row & 127)) * 16 + q4;
    };
    auto st_state32 = [&](void* base, int row, int c, bool w0, bool w1, const float2* t) {
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          SE* a = const_cast<SE*>(t16(base, row + 8 * r, 2 * c + h));
          const float2 u = t[4 * h + r], v = t[4 * h + 2 + r];
          if (r ? w1 : w0) {
            if constexpr (BF) *reinterpret_cast<uint2*>(a) = make_uint2(pack_bf16x2(u.x, u.y), pack_bf16x2(v.x, v.y));
            else *reinterpret_cast<float4*>(a) = make_float4(u.x, u.y, v.x, v.y);
          }
        }
    };
    auto ld_p = [&](auto keep, const float* row, int c, float2* t) {      // one row's four pairs
      uint32_t m[8];
      ld_global_32b<decltype(keep)::value>(row + 32 * c + q8, m);
#pragma unroll
      for (int b = 0; b < 4; ++b) t[b] = make_float2(__uint_as_float(m[2 * b]), __uint_as_float(m[2 * b + 1]));
    };
    auto st_p32 = [&](float* base, int row, int c, bool w0, bool w1, const float2* t) {
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        uint32_t m[8];
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          m[2 * b] = __float_as_uint(t[2 * b + r].x);
          m[2 * b + 1] = __float_as_uint(t[2 * b + r].y);
        }
        if (r ? w1 : w0) st_global_32b(base + (size_t)(row + 8 * r) * H + 32 * c + q8, m);
      }
    };
    // A operand of 32 columns: bf16 hi words in the chunk's first 16 tensor-memory columns, lo words
    // in the other 16.  No wait: publish() waits for the stores.
    auto put_a = [&](uint32_t reg, int c, const float2* t) {
      uint32_t hi[8];
      if constexpr (BF) {
#pragma unroll
        for (int k = 0; k < 8; ++k) hi[k] = pack_bf16x2(t[k].x, t[k].y);
        tmem_st_16x16(reg + 32 * c, hi);
      } else {
        uint32_t lo[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) split_bf16x2(t[k], hi[k], lo[k]);
        tmem_st_16x16(reg + 32 * c, hi);
        tmem_st_16x16(reg + 32 * c + 16, lo);
      }
    };
    // Two T16 state rows -> A operand, AHEAD chunks of loads in flight: whole rows in the two-group kernels
    // (node update 0.170 -> 0.163 ms against three chunks), two chunks where registers are scarcer (edge update
    // 0.295 -> 0.291).  The edge kernels read the edge state, and the source's P_s rows, without keeping them in
    // L1, where the P_d rows of neighbouring edges are read again (0.292 -> 0.287); the node update's own rows
    // are better kept (0.163, 0.167 streamed).  Rows past the end lie in the buffers' padding to whole tiles.
    auto state_to_a = [&](uint32_t reg, const void* base, int row) {
      constexpr int AHEAD = NCH < 2 * (4 - NG) ? NCH : 2 * (4 - NG);
      using V = typename std::conditional<BF, uint2, float4>::type;
      V m[NCH][4];
#pragma unroll
      for (int c = 0; c < NCH + AHEAD; ++c) {
        if (c >= AHEAD) {
          const V* x = m[c - AHEAD];                       // [2h + r]: block pair h, row r
          if constexpr (BF) {                              // the stored words are A's words
            uint32_t hi[8];
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
              for (int r = 0; r < 2; ++r) { hi[4 * h + r] = x[2 * h + r].x; hi[4 * h + 2 + r] = x[2 * h + r].y; }
            tmem_st_16x16(reg + 32 * (c - AHEAD), hi);
          } else {
            float2 t[8];
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
              for (int r = 0; r < 2; ++r) { t[4 * h + r] = lo2(x[2 * h + r]); t[4 * h + 2 + r] = hi2(x[2 * h + r]); }
            put_a(reg, c - AHEAD, t);
          }
        }
        if (c < NCH)
#pragma unroll
          for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int r = 0; r < 2; ++r) {
              const V* a = reinterpret_cast<const V*>(t16(base, row + 8 * r, 2 * c + h));
              m[c][2 * h + r] = KIND == TileKind::NodeUpdate ? *a : __ldcs(a);
            }
      }
    };
    // Runs f(c, t) over the chunks of a region, the next chunk's load in flight meanwhile.
    auto each_chunk = [&](uint32_t reg, auto&& f) {
      float2 t[2][8];
      tmem_ld_16x32(reg, t[0]);
#pragma unroll
      for (int c = 0; c < NCH; ++c) {
        tmem_ld_wait(t[c & 1]);
        if (c + 1 < NCH) tmem_ld_16x32(reg + 32 * (c + 1), t[(c + 1) & 1]);
        f(c, t[c & 1]);
      }
    };
    // Per-column vectors lie in shared memory in the order the quads read them: column 8b + 2q + e of
    // an H-vector at 16*(b/2) + 4q + 2*(b%2) + e, so a thread reads its pairs of two blocks as 16 bytes
    // and the four quad positions read 64 contiguous bytes (no bank conflict).
    auto vec4 = [&](const float* v, int c, int h) { return *reinterpret_cast<const float4*>(v + 32 * c + 16 * h + q4); };
    // LayerNorm statistics of the two rows of D, chunk by chunk.  fp32 model: the host centred every
    // weight block and bias that feeds a LayerNorm (each output row minus the mean over output rows), so
    // the pre-activation has zero mean over the H features and only its variance is computed (the
    // subtraction of the mean is linear and sits in the MMA).  bf16 weights are not centred: the sum and
    // the squares about its own mean of each chunk's eight values, put together at the end.
    struct Stats { float mean[2], rstd[2]; };
    struct Moments { float2 q[2]; float m[2][BF ? NCH : 1]; };
    auto moments_zero = [&](Moments& m) { m.q[0] = m.q[1] = f2(0.f); };
    auto moments_add = [&](Moments& m, int c, const float2* t) {
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        float2 u[4] = {t[r], t[2 + r], t[4 + r], t[6 + r]};
        if constexpr (BF) {
          const float2 s = __fadd2_rn(__fadd2_rn(u[0], u[1]), __fadd2_rn(u[2], u[3]));
          m.m[r][c] = (s.x + s.y) * 0.125f;
#pragma unroll
          for (int k = 0; k < 4; ++k) u[k] = __fadd2_rn(u[k], f2(-m.m[r][c]));
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) m.q[r] = __ffma2_rn(u[k], u[k], m.q[r]);
      }
    };
    auto moments_done = [&](const Moments& m) -> Stats {
      Stats st{{0.f, 0.f}, {0.f, 0.f}};
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        float q = m.q[r].x + m.q[r].y;
        if constexpr (BF) {
          float s = 0.f;
#pragma unroll
          for (int c = 0; c < NCH; ++c) s += m.m[r][c];
          st.mean[r] = quad_sum(s) * (0.25f / NCH);
#pragma unroll
          for (int c = 0; c < NCH; ++c) {
            const float d = m.m[r][c] - st.mean[r];
            q = fmaf(8.f * d, d, q);
          }
        }
        st.rstd[r] = rsqrtf(quad_sum(q) * (1.0f / H) + p.eps);
      }
      return st;
    };
    auto stats = [&](uint32_t reg) -> Stats {
      Moments m;
      moments_zero(m);
      each_chunk(reg, [&](int c, float2* t) { moments_add(m, c, t); });
      return moments_done(m);
    };
    // LayerNorm + ReLU of the two rows of D, 32 columns at a time: emit(c, y).  vb: gamma, beta; without
    // unit_gamma, (v - m) * rstd * gamma + beta.
    auto norm_relu = [&](uint32_t reg, const Stats& st, auto unit_gamma, const float* vb, auto&& emit) {
      constexpr bool UG = decltype(unit_gamma)::value;
      each_chunk(reg, [&](int c, float2* t) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const float4 be = vec4(vb + H, c, h);
          const float4 g = UG ? be : vec4(vb, c, h);
#pragma unroll
          for (int r = 0; r < 2; ++r)
#pragma unroll
            for (int k = 0; k < 2; ++k) {
              float2& x = t[4 * h + 2 * k + r];
              const float2 bk = k ? hi2(be) : lo2(be), is = f2(st.rstd[r]);
              float2 a = x;
              if constexpr (BF) a = __fadd2_rn(a, f2(-st.mean[r]));
              if constexpr (UG) a = __ffma2_rn(a, is, bk);
              else a = __ffma2_rn(__fmul2_rn(a, is), k ? hi2(g) : lo2(g), bk);
              x = relu2(a);
            }
        }
        emit(c, t);
      });
    };
    using True = std::true_type;
    using False = std::false_type;
    // The next job's A from a layer's D: LayerNorm, ReLU.  vb: gamma, beta.
    auto norm_to_a = [&](const Stats& st, const float* vb) {
      auto put = [&](int c, const float2* t) { put_a(a_reg, c, t); };
      if (!BF && p.folded) norm_relu(d_reg, st, True{}, vb, put);
      else norm_relu(d_reg, st, False{}, vb, put);
      publish();
    };
    // Raw inputs of a kind with an input job: this thread's two rows, inputs 8b + 2q and 8b + 2q + 1 of
    // block b at x_in[2b + r].  They are loaded a tile ahead (and an edge's endpoints two), while the
    // current tile's first job runs: loaded at the tile's start, the two dependent loads stood at the head of
    // the chain (edge encoder 0.222 -> 0.190 ms, filter on 1.9M edges 0.412 -> 0.343, node encoder 0.126 ->
    // 0.118).  Not in the embedding, whose registers its outputs need (0.079 -> 0.084).
    constexpr bool AHEAD_INPUTS = KIND != TileKind::Embed;
    [[maybe_unused]] float2 x_in[8];
    [[maybe_unused]] int ends[2][2];           // rows' endpoints: source, destination
    [[maybe_unused]] int valid = 0, valid_next = 0;   // filter: bit r, endpoints of row r in range
    // This thread's row r of tile t, in arithmetic that wraps: rows of a tile past the end, which the loads
    // below are asked for and leave out, may not fit an int.
    auto tile_row = [&](int t, int r) { return (int)((uint32_t)t * kTileRows + (uint32_t)(trow + 8 * r)); };
    auto load_ends = [&](int t) {              // endpoints of this thread's two edges of tile t
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        const int k = tile_row(t, r);
        const bool in = t < p.n_tiles && k < p.n_rows;
        if constexpr (KIND == TileKind::Filter) {
          ends[r][0] = in ? p.ei_in[k] : -1;
          ends[r][1] = in ? p.ei_in[(size_t)p.n_rows + k] : -1;
        } else {
          ends[r][0] = in ? p.src_sorted[k] : 0;
          ends[r][1] = in ? p.dst_sorted[k] : 0;
        }
      }
    };
    auto load_inputs = [&](int t) {            // inputs of tile t (an edge's endpoints are in ends)
      valid_next = 0;
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        const float *xs, *xd;
        int split = p.n_in;
        if constexpr (KIND == TileKind::Filter) {
          const int s0 = ends[r][0], d0 = ends[r][1];
          const bool ok_ends = s0 >= 0 && s0 < p.n_nodes && d0 >= 0 && d0 < p.n_nodes;
          valid_next |= ok_ends ? 1 << r : 0;
          xs = p.x + (size_t)(ok_ends ? s0 : 0) * p.x_stride;
          xd = p.x + (size_t)(ok_ends ? d0 : 0) * p.x_stride;
          split = p.n_feat;
        } else if constexpr (KIND == TileKind::EdgeEncoder) {
          xs = p.x + (size_t)ends[r][0] * p.x_stride;
          xd = p.x + (size_t)ends[r][1] * p.x_stride;
        } else {
          const int k = tile_row(t, r);
          xs = xd = p.x + (size_t)(t < p.n_tiles && k < p.n_rows ? k : 0) * p.x_stride;
        }
        if constexpr (KIND == TileKind::EdgeEncoder) {       // columns 0 and 1 of both ends; (dr, dphi) at use
          x_in[r] = make_float2(xs[0], xs[1]);
          x_in[2 + r] = make_float2(xd[0], xd[1]);
        } else {
#pragma unroll
          for (int b = 0; b < 4; ++b) {
            const int i = 8 * b + 2 * (lane & 3);
            x_in[2 * b + r].x = i < split ? xs[i] : i < p.n_in ? xd[i - split] : 0.f;
            x_in[2 * b + r].y = i + 1 < split ? xs[i + 1] : i + 1 < p.n_in ? xd[i + 1 - split] : 0.f;
          }
        }
      }
    };
    // Inputs -> A operand of the first job, in three bf16 parts (24 bits: all of an fp32 value).  The next
    // tile's are loaded while the job runs.
    auto input_to_a = [&](int tile, int next) {
      float2 t[8];
      if constexpr (!AHEAD_INPUTS) load_inputs(tile);
      valid = valid_next;
      if constexpr (KIND == TileKind::EdgeEncoder) {
#pragma unroll
        for (int k = 0; k < 8; ++k) t[k] = f2(0.f);
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          float dphi = x_in[2 + r].y - x_in[r].y;
          if (dphi > 1.0f) dphi -= 2.0f;
          if (dphi <= -1.0f) dphi += 2.0f;
          if ((lane & 3) == 0) t[r] = make_float2(x_in[2 + r].x - x_in[r].x, dphi);
        }
      } else {
#pragma unroll
        for (int k = 0; k < 8; ++k) t[k] = x_in[k];
      }
#pragma unroll
      for (int part = 0; part < 3; ++part) {
        uint32_t w[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          w[k] = pack_bf16x2(t[k].x, t[k].y);
          t[k] = __fadd2_rn(t[k], make_float2(-__uint_as_float(w[k] << 16), -__uint_as_float(w[k] & 0xffff0000u)));
        }
        tmem_st_16x16(a_reg + 16 * part, w);
      }
      publish();
      if constexpr (AHEAD_INPUTS) load_inputs(next);
      if constexpr (KIND == TileKind::Filter || KIND == TileKind::EdgeEncoder) load_ends(next + NG * (int)gridDim.x);
      wait_job();
    };
    // w . y of the two rows, accumulated chunk by chunk (bf16 model: the input is a bf16 activation)
    auto dot_chunk = [&](int c, const float2* t, const float* w, float2* z) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const float4 ww = vec4(w, c, h);
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          const float2 u = BF ? round_bf16x2(t[4 * h + r]) : t[4 * h + r];
          const float2 v = BF ? round_bf16x2(t[4 * h + 2 + r]) : t[4 * h + 2 + r];
          z[r] = __ffma2_rn(v, hi2(ww), __ffma2_rn(u, lo2(ww), z[r]));
        }
      }
    };
    auto sigmoid = [&](float z) { return 1.0f / (1.0f + __expf(-z)); };

    const int L = p.n_layers;
    if (grp < n_my) {
      const int t = (int)blockIdx.x + grp * (int)gridDim.x;
      if constexpr (KIND != TileKind::NodeEncoder && KIND != TileKind::NodeUpdate && KIND != TileKind::Embed) load_ends(t);
      if constexpr (has_input_job(KIND) && AHEAD_INPUTS) {
        load_inputs(t);
        if constexpr (KIND == TileKind::Filter || KIND == TileKind::EdgeEncoder) load_ends(t + NG * (int)gridDim.x);
      }
    }
    for (int it = grp; ok && it < n_my; it += NG) {
      const int tile = (int)blockIdx.x + it * (int)gridDim.x;
      const int row = tile * kTileRows + trow;
      const bool in[2] = {row < p.n_rows, row + 8 < p.n_rows};
      const int next_tile = tile + NG * (int)gridDim.x;
      j = 0;

      if constexpr (KIND == TileKind::EdgeUpdate || KIND == TileKind::Classifier) {
        // vecs: [(gamma_l, beta_l) for l = 1..L, (w_o, b_o)]
        GNN_TRACE_W(0);
        // classifier: where each row's score goes (input order) and, in the sign bit, whether an
        // endpoint was out of range; read now so that the score store ending the tile waits on no load
        int out[2] = {0, 0};
        if constexpr (KIND == TileKind::Classifier)
#pragma unroll
          for (int r = 0; r < 2; ++r)
            if (in[r] && (lane & 3) == 0) out[r] = p.perm[row + 8 * r] | (p.key_sorted[row + 8 * r] < p.n_nodes ? 0 : INT_MIN);
        state_to_a(a_reg, p.e, row);
        publish();                                        // job: D = e * W_e^T
        GNN_TRACE_W(1);
        // layer-1 terms of the endpoints, loaded while the MMA runs: S = P_s[src] + P_d[dst] (P_d
        // carries b1), the first chunks before D is waited for, the others while those are added
        constexpr int EARLY = NCH < 2 ? NCH : 2;
        float2 S[NCH][8];
        auto gather = [&](int c) {
#pragma unroll
          for (int r = 0; r < 2; ++r) {
            float2 a[4], b[4];
            asm volatile("" : "+r"(ends[r][0]), "+r"(ends[r][1]));   // the row addresses are formed anew, not kept
            ld_p(std::false_type{}, p.ps + (size_t)ends[r][0] * H, c, a);
            ld_p(std::true_type{}, p.pd + (size_t)ends[r][1] * H, c, b);
#pragma unroll
            for (int k = 0; k < 4; ++k) S[c][2 * k + r] = __fadd2_rn(a[k], b[k]);
          }
#pragma unroll
          for (int k = 0; k < 8; ++k) asm volatile("" : "+f"(S[c][k].x), "+f"(S[c][k].y));
        };
#pragma unroll
        for (int c = 0; c < EARLY; ++c) gather(c);
        GNN_TRACE_W(2);
        wait_job();
        GNN_TRACE_W(3);
        Moments m;
        moments_zero(m);
#pragma unroll
        for (int c = 0; c < NCH; ++c) {                   // D += S, with the rows' moments
          float2 t[8];
          tmem_ld_16x32(d_reg + 32 * c, t);
          if (c >= EARLY) gather(c);
          tmem_ld_wait(t);
#pragma unroll
          for (int k = 0; k < 8; ++k) t[k] = __fadd2_rn(t[k], S[c][k]);
          moments_add(m, c, t);
          tmem_st_16x32(d_reg + 32 * c, t);
        }
        tmem_st_wait();
        norm_to_a(moments_done(m), vecs);
        GNN_TRACE_W(4);
        for (int l = 2; l <= L; ++l) {
          wait_job();
          GNN_TRACE_W(1 + 2 * l);
          if (l == 2) {
            // This group's next tile, a few microseconds before its load: its endpoints, and its
            // edge state into L2 (bulk prefetch: the copy engine, not the SM's load path).
            if (leader && next_tile < p.n_tiles)
              prefetch_l2_bulk(static_cast<const SE*>(p.e) + (size_t)next_tile * kTileRows * H, kTileRows * H * sizeof(SE));
            load_ends(next_tile);
          }
          if (l < L) norm_to_a(stats(d_reg), vecs + 2 * (l - 1) * H);
          GNN_TRACE_W(2 + 2 * l);
        }
        const float* vb = vecs + 2 * (L - 1) * H;
        const Stats sl = stats(d_reg);
        if constexpr (KIND == TileKind::EdgeUpdate) {
          norm_relu(d_reg, sl, False{}, vb, [&](int c, const float2* t) {
            st_state32(p.e, row, c, ok && in[0], ok && in[1], t);
          });
          GNN_TRACE_W(11);
        } else {
          const float* wo = vb + 2 * H;
          float2 z[2] = {f2(0.f), f2(0.f)};
          norm_relu(d_reg, sl, False{}, vb, [&](int c, const float2* t) { dot_chunk(c, t, wo, z); });
#pragma unroll
          for (int r = 0; r < 2; ++r) {
            const float zz = quad_sum(z[r].x + z[r].y) + wo[H];
            if (ok && in[r] && (lane & 3) == 0)
              p.scores[out[r] & INT_MAX] = out[r] >= 0 ? sigmoid(zz) : __int_as_float(0x7fc00000);
          }
        }
      } else if constexpr (KIND == TileKind::EdgeEncoder) {
        // vecs: [(gamma_l, beta_l) for l = 1..L]
        input_to_a(tile, next_tile);
        const float* vb = vecs;
        for (int l = 1; l < L; ++l, vb += 2 * H) {
          norm_to_a(stats(d_reg), vb);
          wait_job();
        }
        const Stats sl = stats(d_reg);
        norm_relu(d_reg, sl, False{}, vb, [&](int c, const float2* t) {
          st_state32(p.e, row, c, ok && in[0], ok && in[1], t);
        });
      } else if constexpr (KIND == TileKind::Embed) {
        // vecs: [(gamma_l, beta_l) for l = 1..L, W_out rows (D x H), b_out (D)]
        // L hidden layers, then the D outputs on CUDA cores, L2-normalised.
        input_to_a(tile, next_tile);
        const float* vb = vecs;
        for (int l = 1; l < L; ++l, vb += 2 * H) {
          norm_to_a(stats(d_reg), vb);
          wait_job();
        }
        const float* wout = vb + 2 * H;
        // the last layer's rows back into the region, then one pass over them per output: D is not
        // known to the compiler, and the rows do not fit in registers
        const Stats sl = stats(d_reg);
        norm_relu(d_reg, sl, False{}, vb, [&](int c, const float2* t) { tmem_st_16x32(d_reg + 32 * c, t); });
        tmem_st_wait();
        float nn[2] = {0.f, 0.f}, y[2] = {0.f, 0.f};       // thread q keeps outputs q, q + 4, ... of its rows
        float keep[2][kMaxEmbedDim / 4];
#pragma unroll
        for (int g = 0; g < kMaxEmbedDim / 4; ++g) {
          keep[0][g] = keep[1][g] = 0.f;
          for (int i = 4 * g; i < 4 * g + 4 && i < p.emb_dim; ++i) {
            float2 z[2] = {f2(0.f), f2(0.f)};
            each_chunk(d_reg, [&](int c, float2* t) { dot_chunk(c, t, wout + i * H, z); });
#pragma unroll
            for (int r = 0; r < 2; ++r) {
              y[r] = quad_sum(z[r].x + z[r].y) + wout[p.emb_dim * H + i];
              nn[r] = fmaf(y[r], y[r], nn[r]);
              if ((i & 3) == (lane & 3)) keep[r][g] = y[r];
            }
          }
        }
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          const float inv = nn[r] > 0.f ? rsqrtf(nn[r]) : 0.f;
#pragma unroll
          for (int g = 0; g < kMaxEmbedDim / 4; ++g) {
            const int i = 4 * g + (lane & 3);
            if (ok && in[r] && i < p.emb_dim) p.emb[(size_t)(row + 8 * r) * p.emb_dim + i] = keep[r][g] * inv;
          }
        }
      } else if constexpr (KIND == TileKind::Filter) {
        // vecs: [(gamma_l, beta_l) for l = 1..L, (w_o, b_o)]
        // The inputs are the raw features of both endpoints, [x_src, x_dst].
        input_to_a(tile, next_tile);
        const float* vb = vecs;
        for (int l = 1; l < L; ++l, vb += 2 * H) {
          norm_to_a(stats(d_reg), vb);
          wait_job();
        }
        const float* wo = vb + 2 * H;
        float2 z[2] = {f2(0.f), f2(0.f)};
        const Stats sl = stats(d_reg);
        norm_relu(d_reg, sl, False{}, vb, [&](int c, const float2* t) { dot_chunk(c, t, wo, z); });
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          const float zz = quad_sum(z[r].x + z[r].y) + wo[H];
          if (ok && in[r] && (lane & 3) == 0) {
            p.scores[row + 8 * r] = (valid >> r) & 1 ? sigmoid(zz) : __int_as_float(0x7fc00000);
            if (!((valid >> r) & 1)) atomicOr(p.err, DEV_ERR_INDEX_RANGE);
          }
        }
      } else {
        // NodeEncoder / NodeUpdate.
        // vecs: [(gamma_l, beta_l) for l = 1..L]
        const float* vb = vecs;
        const bool w0 = in[0], w1 = in[1];
        GNN_TRACE_W(0);
        if constexpr (KIND == TileKind::NodeEncoder) {
          input_to_a(tile, next_tile);
        } else {
          state_to_a(a_reg, p.h, row);
          publish();                                      // job: D = h * W_h^T
          GNN_TRACE_W(1);
          if (leader)                                     // this tile's aggregate rows
            prefetch_l2_bulk(static_cast<const SE*>(p.agg) + (size_t)tile * kTileRows * H, kTileRows * H * sizeof(SE));
          wait_job();                                     // A free again
          GNN_TRACE_W(2);
          state_to_a(a_reg, p.agg, row);                  // a_j, summed by the aggregation kernel
          publish();                                      // job: D += a * W_a^T
          GNN_TRACE_W(3);
          wait_job();
          GNN_TRACE_W(4);
        }
        for (int l = 1; l < L; ++l, vb += 2 * H) {
          norm_to_a(stats(d_reg), vb);
          GNN_TRACE_W(3 + 2 * l);
          wait_job();
          GNN_TRACE_W(4 + 2 * l);
        }
        {                                                 // last layer: new node state, and A for the P_s job
          if (KIND == TileKind::NodeUpdate && leader && next_tile < p.n_tiles)   // the next h tile
            prefetch_l2_bulk(static_cast<const SE*>(p.h) + (size_t)next_tile * kTileRows * H, kTileRows * H * sizeof(SE));
          const Stats sl = stats(d_reg);
          norm_relu(d_reg, sl, False{}, vb, [&](int c, const float2* t) {
            st_state32(p.h, row, c, ok && w0, ok && w1, t);
            put_a(a_reg, c, t);
          });
          publish();                                      // the P_s job
        }
        GNN_TRACE_W(11);
        wait_job();                                       // P_s = W_s h (no bias)
        GNN_TRACE_W(12);
        each_chunk(d_reg, [&](int c, const float2* t) { st_p32(p.ps, row, c, ok && w0, ok && w1, t); });
        publish();                                        // D read; A (= h) unchanged -> P_d job
        GNN_TRACE_W(13);
        wait_job();                                       // P_d = W_d h + b1 (edge-side bias)
        GNN_TRACE_W(14);
        each_chunk(d_reg, [&](int c, const float2* t) { st_p32(p.pd, row, c, ok && w0, ok && w1, t); });
        GNN_TRACE_W(15);
      }
#ifdef GNN_TRACE
      ++tr_iter;
#endif
    }
    __syncwarp();
  }

  // teardown: every warp reaches this point (waits are bounded)
  tc_fence_before();
  __syncthreads();
  GNN_TRACE_CTA(1);
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem_base, G::TMEM_COLS);
  }
}

// a_j = sum of the messages m_ij of the edges into node j (CSR segment of j,
// summed in slot order from zero, no atomics: deterministic, and identical for
// a node whether its event is scored alone or in a batch).  One warp serves one
// node (half a warp when H = 64): lane 4*bp + q owns the 16-byte vector q of
// block pair bp (row-tiled T16 layout of the tile kernels), so all lanes of a
// node run the same number of steps whatever the degree distribution, and
// every message row is read in whole 64-byte pieces.  Blocks take the nodes
// from the last one down: the edge update writes the messages in CSR (that is,
// destination) order and finishes with the highest tiles, which are then still
// in L2 when the first blocks here read them.
template <int H>
constexpr int agg_nodes_per_block() { return 256 / (H / 4); }

template <int H, bool BF>
__global__ void __launch_bounds__(256) aggregate_kernel(const void* __restrict__ e_, const int* __restrict__ rowptr,
                                                        int n_nodes, void* __restrict__ agg_) {
  using SE = typename std::conditional<BF, __nv_bfloat16, float>::type;
  constexpr int NBP = H / 16;
  constexpr int LPN = H / 4;                         // lanes per node
  const SE* e = static_cast<const SE*>(e_);
  SE* agg = static_cast<SE*>(agg_);
  pdl_wait();
  pdl_trigger_small();
  const int li = threadIdx.x % LPN;
  const int bp = li >> 2, q = li & 3;
  const int j = n_nodes - 1 - (blockIdx.x * agg_nodes_per_block<H>() + (int)threadIdx.x / LPN);
  if (j < 0) return;
  const int k0 = rowptr[j], k1 = rowptr[j + 1];
  auto at = [&](int k) -> float4 {
    const SE* a = e + (((size_t)(k >> 7) * NBP + bp) * 128 + (k & 127)) * 16 + 4 * q;
    if constexpr (BF) {
      const uint2 u = __ldcs(reinterpret_cast<const uint2*>(a));
      const float2 lo = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.x));
      const float2 hi = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.y));
      return make_float4(lo.x, lo.y, hi.x, hi.y);
    } else {
      return __ldcs(reinterpret_cast<const float4*>(a));
    }
  };
  float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
  int k = k0;
  for (; k + 4 <= k1; k += 4) {
    const float4 x0 = at(k), x1 = at(k + 1), x2 = at(k + 2), x3 = at(k + 3);
    a.x += x0.x; a.y += x0.y; a.z += x0.z; a.w += x0.w;
    a.x += x1.x; a.y += x1.y; a.z += x1.z; a.w += x1.w;
    a.x += x2.x; a.y += x2.y; a.z += x2.z; a.w += x2.w;
    a.x += x3.x; a.y += x3.y; a.z += x3.z; a.w += x3.w;
  }
  for (; k < k1; ++k) {
    const float4 x = at(k);
    a.x += x.x; a.y += x.y; a.z += x.z; a.w += x.w;
  }
  SE* out = agg + (((size_t)(j >> 7) * NBP + bp) * 128 + (j & 127)) * 16 + 4 * q;
  if constexpr (BF) {                                // the aggregate is a bf16 activation
    *reinterpret_cast<uint2*>(out) = make_uint2(pack_bf16x2(a.x, a.y), pack_bf16x2(a.z, a.w));
  } else {
    *reinterpret_cast<float4*>(out) = a;
  }
}

}  // namespace gnn
