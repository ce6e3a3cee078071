// C ABI and host orchestration of the interaction-network edge classifier.
//
// gnn_create parses the weight blob and repacks every H x H weight block into
// the layout the tensor-core kernels read straight into shared memory
// (bf16 hi and lo parts, K-major rows of 128 bytes, 128-byte swizzle).  The
// first Linear layer of the edge network and of the classifier acts on
// [h_src, h_dst, e]; it is split into three H x H blocks W_s, W_d, W_e so that
//   W1 [h_src; h_dst; e] + b1 = (W_s h_src) + (W_d h_dst + b1) + W_e e,
// where the two node terms are computed once per node (projections P_s, P_d)
// instead of once per edge.  The node network's first layer on [h, a] is
// split the same way into W_h and W_a.
//
// gnn_infer enqueues: CSR build (radix sort by destination, whose first pass
// validates the endpoints; one kernel gathers the sources and writes the row
// pointers) -> node encoder (+ projections) -> edge encoder -> T x (edge update,
// aggregation, node update + projections) -> classifier.
#include <cuda_runtime.h>
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <new>
#include <utility>
#include <vector>

#include "../../include/gnn.h"
#include "compact.cuh"
#include "components.cuh"
#include "csr.cuh"
#include "frnn.cuh"
#include "mlp_tiles.cuh"

using namespace gnn;

namespace {

constexpr uint32_t kBlobMagic = 0x57474E47u;
constexpr uint32_t kFilterMagic = 0x4C464E47u;   // "GNFL": the filtering MLP's weight blob
constexpr uint32_t kEmbedMagic = 0x4D454E47u;    // "GNEM": the embedding MLP's weight blob
constexpr int kHeaderBytes = 8 * 4 + 4 + 4 + 8;

struct Layer { const float* W; const float* b; const float* g; const float* be; int in; };

enum Mlp { NODE_ENC = 0, EDGE_ENC = 1, EDGE_NET = 2, NODE_NET = 3, CLASSIFIER = 4, N_MLP = 5 };

struct KernelPlan {          // job list and parameter vectors of one tile-kernel launch
  int n_jobs = 0;
  int job_mat[kMaxJobs] = {0};
  int job_acc[kMaxJobs] = {0};
  int job_bias[kMaxJobs] = {0};     // 1-based bias tile a job's D starts from, 0: none
  bool folded = false;              // gamma folded into the weights, but for the MLP's last layer
  std::vector<float> vecs;
  std::vector<const float*> biases; // the bias tiles' vectors, while the plan is made
  float* d_vecs = nullptr;          // vecs, and behind them the ones tile and the bias tiles
  uint8_t* d_consts = nullptr;
  uint32_t const_bytes = 0;
  const uint8_t* wmats = nullptr;   // its weight matrices (null: the context's)
};

}  // namespace

struct gnn_ctx {
  gnn_config cfg;
  int device = 0;
  int n_sm = 0;
  uint8_t* d_mats = nullptr;       // packed weight matrices
  uint32_t mat_bytes = 0;
  // plans: 0 node enc -> edge net, 1 node enc -> classifier, 2 edge enc,
  //        3 edge update, 4 node update -> edge net, 5 node update -> classifier, 6 classifier
  KernelPlan plan[7];
  // filtering step (gnn_filter_load): plan, packed deep-layer matrices, layers, LayerNorm eps
  KernelPlan filter_plan;
  uint8_t* d_filter_mats = nullptr;
  int filter_layers = 0;
  float filter_eps = 0.f;
  // embedding step (gnn_embed_load) and graph building scratch
  KernelPlan embed_plan;
  uint8_t* d_embed_mats = nullptr;
  int embed_layers = 0, embed_dim = 0;
  float embed_eps = 0.f;
  int* aux = nullptr;
  size_t aux_ints = 0;
  bool aux_tight = false;              // the scratch was made without the default pool of partner chunks
  int64_t graph_pool = -1;             // graph building: pool chunks for partner chains (-1: one per hit)
  uint32_t* d_err = nullptr;
  // workspace
  void* ws = nullptr;
  int64_t cap_nodes = -1, cap_edges = -1;
  int *keys_a = nullptr, *keys_b = nullptr, *vals_a = nullptr, *vals_b = nullptr;
  int *hist = nullptr, *perm = nullptr, *src_sorted = nullptr, *dst_sorted = nullptr, *rowptr = nullptr;
  int* key_sorted = nullptr;
  void *e = nullptr, *h = nullptr, *agg = nullptr;  // stored states (fp32 or bf16 per precision)
  float *ps = nullptr, *pd = nullptr;
  int64_t last_nodes = 0, last_edges = 0;
  // staging for gnn_infer_host
  void* stage = nullptr;
  size_t stage_bytes = 0;
  // profiling: event pairs around kernel groups
  struct ProfRec { int group; int launches; cudaEvent_t a, b; };
  bool prof_on = false;
  std::vector<ProfRec> prof;
  size_t prof_used = 0;
#ifdef GNN_TRACE
  unsigned long long* trace = nullptr;   // stamps of CTA 0 of the traced kernel kind
  int trace_kind = -1;
#endif
};

namespace {

inline uint16_t f32_to_bf16_rne(float f) {
  uint32_t u;
  std::memcpy(&u, &f, 4);
  if ((u & 0x7F800000u) == 0x7F800000u) return (uint16_t)((u >> 16) | ((u & 0xFFFFu) ? 0x40u : 0u));
  u += 0x7FFFu + ((u >> 16) & 1u);
  return (uint16_t)(u >> 16);
}
inline float bf16_to_f32(uint16_t h) {
  uint32_t u = (uint32_t)h << 16;
  float f;
  std::memcpy(&f, &u, 4);
  return f;
}

// Byte offset of element (n, k) of an H x H block in the K-major, 128-byte
// swizzled layout: 64-column chunks, 8-row atoms of 1024 bytes, 16-byte units
// of a row permuted by XOR with the row index inside the atom.
inline size_t swizzled_offset(int H, int n, int k) {
  const int kc = k / 64, kk = k % 64;
  return (size_t)kc * (H * 128) + (size_t)(n / 8) * 1024 + (n % 8) * 128 +
         (((kk / 8) ^ (n % 8)) * 16) + (kk % 8) * 2;
}

// Pack columns [col0, col0+H) of W [H, ld] into hi/lo bf16 parts (fp32 model), or
// into the single bf16 part (bf16 model: W holds bf16 values, hi == W exactly).
void pack_block(const float* W, int ld, int col0, int H, bool with_lo, uint8_t* out) {
  const size_t part = (size_t)H * H * 2;
  for (int n = 0; n < H; ++n)
    for (int k0 = 0; k0 < H; k0 += 8) {              // a 16-byte unit of the layout
      uint16_t hi[8], lo[8];
      for (int k = 0; k < 8; ++k) {
        const float v = W[(size_t)n * ld + col0 + k0 + k];
        hi[k] = f32_to_bf16_rne(v);
        lo[k] = f32_to_bf16_rne(v - bf16_to_f32(hi[k]));
      }
      const size_t off = swizzled_offset(H, n, k0);
      std::memcpy(out + off, hi, 16);
      if (with_lo) std::memcpy(out + part + off, lo, 16);
    }
}

// Pack a first layer's W [H, n_in], n_in <= 32, as an input matrix: its hi, mid and lo bf16 parts (fp32
// model) or its one part (bf16 model) at their places in a weight block of zeros.
void pack_input(const float* W, int n_in, int H, bool bf, uint8_t* out, size_t bytes) {
  std::memset(out, 0, bytes);
  for (int n = 0; n < H; ++n)
    for (int k = 0; k < n_in; ++k) {
      float v = W[(size_t)n * n_in + k];
      for (int w = 0; w < (bf ? 1 : 3); ++w) {
        const uint16_t part = f32_to_bf16_rne(v);
        // parts 0 and 1 share a 64-column chunk (columns 32 w + k); part 2 starts one of its own
        const size_t base = w < 2 ? 0 : (H == 128 ? input_part_offset<128>(2) : input_part_offset<64>(2));
        std::memcpy(out + base + swizzled_offset(H, n, (w < 2 ? 32 * w : 0) + k), &part, 2);
        v -= bf16_to_f32(part);
      }
    }
}

void push(std::vector<float>& v, const float* p, size_t n) { v.insert(v.end(), p, p + n); }

// W' = (I - 11^T/H) W and b' = b - mean(b): the LayerNorm after the layer then sees a
// zero-mean pre-activation (the fp32 model's kernels compute only the variance).
void centre_layer(const float* W, const float* b, int H, int in, std::vector<float>& Wc, std::vector<float>& bc) {
  Wc.resize((size_t)H * in);
  bc.resize(H);
  std::vector<double> mu(in, 0.0);
  for (int n = 0; n < H; ++n)
    for (int k = 0; k < in; ++k) mu[k] += W[(size_t)n * in + k];
  for (int k = 0; k < in; ++k) mu[k] /= H;
  for (int n = 0; n < H; ++n)
    for (int k = 0; k < in; ++k) Wc[(size_t)n * in + k] = (float)(W[(size_t)n * in + k] - mu[k]);
  double mb = 0.0;
  for (int n = 0; n < H; ++n) mb += b[n];
  mb /= H;
  for (int n = 0; n < H; ++n) bc[n] = (float)(b[n] - mb);
}

// LayerNorm vectors of one layer, as the kernels read them: gamma, beta.
void push_ln(std::vector<float>& v, const Layer& l, int H) {
  push(v, l.g, H);
  push(v, l.be, H);
}

// fp32 model: y_l = relu(gamma n + beta) of a hidden layer l < L equals |gamma| relu(s n + beta / |gamma|)
// with s = sign(gamma), so the kernels need no gamma when W_l's rows and b_l carry s and W_{l+1}'s columns
// carry |gamma| (a LayerNorm's variance does not see the sign, and the fp32 model's kernels compute no mean).  One
// vector less is read and one multiplication less made per element of every hidden layer.  Only for
// |gamma| in [2^-6, 2^6], where the scaling cannot overflow or lose a column; otherwise the MLP keeps
// its gammas (false).  `lay` points at copies of the model's arrays.
bool fold_gamma(std::vector<std::vector<float>*> W, std::vector<std::vector<float>*> b,
                std::vector<std::vector<float>*> g, std::vector<std::vector<float>*> be, const int* in, int H) {
  const int L = (int)W.size();
  for (int l = 0; l + 1 < L; ++l)
    for (int i = 0; i < H; ++i) {
      const float a = std::fabs((*g[l])[i]);
      if (!(a >= 0.015625f && a <= 64.f)) return false;
    }
  std::vector<float> scale((size_t)L * H);
  for (int l = 0; l + 1 < L; ++l)
    for (int i = 0; i < H; ++i) {
      const float s = (*g[l])[i] < 0.f ? -1.f : 1.f, a = std::fabs((*g[l])[i]);
      for (int k = 0; k < in[l]; ++k) (*W[l])[(size_t)i * in[l] + k] *= s;
      (*b[l])[i] *= s;
      (*be[l])[i] /= a;
      (*g[l])[i] = 1.f;
      scale[l * H + i] = a;
    }
  for (int l = 0; l + 1 < L; ++l)
    for (int n = 0; n < H; ++n)
      for (int i = 0; i < H; ++i) (*W[l + 1])[(size_t)n * in[l + 1] + i] *= scale[l * H + i];
  return true;
}

// Copies of one MLP's arrays, centred and folded for the fp32 model; the Layers are pointed at them.
struct MlpCopy {
  std::vector<std::vector<float>> W, b, g, be;
  bool folded = false;
};
void prepare_mlp(Layer* lay, int L, int H, bool bf, bool fold, MlpCopy& c) {
  if (bf) return;                                    // bf16 weights stay on the bf16 grid, as given
  c.W.resize(L); c.b.resize(L); c.g.resize(L); c.be.resize(L);
  std::vector<std::vector<float>*> W, b, g, be;
  int in[4];
  for (int l = 0; l < L; ++l) {
    in[l] = lay[l].in;
    centre_layer(lay[l].W, lay[l].b, H, lay[l].in, c.W[l], c.b[l]);
    c.g[l].assign(lay[l].g, lay[l].g + H);
    c.be[l].assign(lay[l].be, lay[l].be + H);
    W.push_back(&c.W[l]); b.push_back(&c.b[l]); g.push_back(&c.g[l]); be.push_back(&c.be[l]);
  }
  c.folded = fold && fold_gamma(W, b, g, be, in, H);
  for (int l = 0; l < L; ++l) lay[l] = {c.W[l].data(), c.b[l].data(), c.g[l].data(), c.be[l].data(), in[l]};
}

// A job's D starts from this bias.
void set_bias(KernelPlan& pl, int job, const float* b) {
  pl.biases.push_back(b);
  pl.job_bias[job] = (int)pl.biases.size();
}

// The constant tiles a plan's biases are added with: D = ones * tile^T, one K step of 16.  Every row of
// the ones tile [128, 16] is (1, 1, 1, 0, ...); row n of a bias tile [H, 16] is b[n] in three bf16 parts
// (24 bits, all of an fp32 value), then zeros.  K-major without a swizzle: element (r, k) at byte
// (r / 8) * 256 + (k / 8) * 128 + (r % 8) * 16 + (k % 8) * 2.
// Appended to `block`.
void const_tiles(const KernelPlan& pl, int H, std::vector<uint8_t>& block) {
  const size_t base = block.size();
  block.resize(base + 128 * 32 + pl.biases.size() * H * 32, 0);
  auto put = [&](size_t tile, int r, int k, uint16_t v) {
    std::memcpy(block.data() + base + tile + (r / 8) * 256 + (k / 8) * 128 + (r % 8) * 16 + (k % 8) * 2, &v, 2);
  };
  for (int r = 0; r < 128; ++r)
    for (int k = 0; k < 3; ++k) put(0, r, k, f32_to_bf16_rne(1.0f));
  for (size_t i = 0; i < pl.biases.size(); ++i)
    for (int n = 0; n < H; ++n) {
      float v = pl.biases[i][n];
      for (int k = 0; k < 3; ++k) {
        const uint16_t part = f32_to_bf16_rne(v);
        put(128 * 32 + i * H * 32, n, k, part);
        v -= bf16_to_f32(part);
      }
    }
}

// Every whole H-float segment of a plan's vector block is one per-column vector (bias, gamma,
// beta, head weights, a first-layer weight row); the kernels read them in block-pair order:
// column 8b + 2q + e at 16*(b/2) + 4q + 2*(b%2) + e.  A trailing partial segment (the head
// bias) stays as is.  Then padded to 16 bytes.
void finish_vecs(std::vector<float>& v, int H) {
  std::vector<float> seg(H);
  for (size_t base = 0; base + H <= v.size(); base += H) {
    for (int q = 0; q < 4; ++q)
      for (int b = 0; b < H / 8; ++b)
        for (int e = 0; e < 2; ++e) seg[16 * (b / 2) + 4 * q + 2 * (b % 2) + e] = v[base + 8 * b + 2 * q + e];
    std::copy(seg.begin(), seg.end(), v.begin() + base);
  }
  v.resize(padded_vec_floats((int)v.size()), 0.f);
}

// Test hook: the next g_fail_allocs device allocations made by the library fail (host-side fault
// injection for the allocation-failure paths; see gnn_debug_fail_allocs).
std::atomic<int> g_fail_allocs{0};

cudaError_t dev_alloc(void** p, size_t bytes) {
  int n = g_fail_allocs.load();
  while (n > 0 && !g_fail_allocs.compare_exchange_weak(n, n - 1)) {
  }
  if (n > 0) {
    *p = nullptr;
    return cudaErrorMemoryAllocation;
  }
  return cudaMalloc(p, bytes);
}

// A plan's vectors and constant tiles to the device.
cudaError_t upload_plan(KernelPlan& pl, int H) {
  const size_t vb = (pl.vecs.size() * 4 + 255) & ~size_t(255);
  std::vector<uint8_t> block(vb, 0);
  std::memcpy(block.data(), pl.vecs.data(), pl.vecs.size() * 4);
  const_tiles(pl, H, block);
  pl.biases.clear();
  pl.const_bytes = (uint32_t)(block.size() - vb);
  cudaError_t err = dev_alloc((void**)&pl.d_vecs, block.size());
  if (err != cudaSuccess) { pl.d_vecs = nullptr; return err; }
  pl.d_consts = (uint8_t*)pl.d_vecs + vb;
  err = cudaMemcpy(pl.d_vecs, block.data(), block.size(), cudaMemcpyHostToDevice);
  return err;
}

// A kernel that waits, through the library's bounded wait, on an mbarrier nothing arrives on.
__global__ void wait_timeout_kernel(uint64_t limit_ns, uint32_t* err) {
  __shared__ uint64_t bar;
  __shared__ int abort_flag;
  if (threadIdx.x != 0) return;
  mbar_init(&bar, 1);
  abort_flag = 0;
  fence_mbar_init();
  bounded_wait(&bar, 0, &abort_flag, err, limit_ns);
}

int cuda_fail(cudaError_t e) {
  (void)cudaGetLastError();
  return e == cudaErrorMemoryAllocation ? GNN_ERR_OOM : GNN_ERR_CUDA;
}

// Every count a call accepts (nodes, edges, output capacity) lies in [0, GNN_MAX_COUNT], so that
// the kernels' 32-bit row indices stay in range after rounding up to a whole block or radix tile
// (at most 8192 rows).
inline bool count_ok(int64_t n) { return n >= 0 && n <= (int64_t)GNN_MAX_COUNT; }

// Blocks of `per_block` threads (or rows) covering n, computed in 64 bits.
inline unsigned blocks_for(int64_t n, int64_t per_block) { return (unsigned)((n + per_block - 1) / per_block); }

// Launch as a programmatic dependent of the previous kernel in the stream: the kernel may start
// while that one finishes its last CTAs, and waits for it (pdl_wait) before touching its data.
// Every kernel launched this way calls pdl_wait before its first access to data an earlier
// kernel writes.  Returns the launch status.
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*kernel)(KArgs...), unsigned grid, unsigned block, size_t smem, cudaStream_t st,
                       Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

constexpr int kProfGroups = 10;

// Returns the record index, or -1 when profiling is off.
int prof_begin(gnn_ctx* c, int group, int launches, cudaStream_t st) {
  if (!c->prof_on) return -1;
  if (c->prof_used == c->prof.size()) {
    gnn_ctx::ProfRec r{};
    if (cudaEventCreate(&r.a) != cudaSuccess || cudaEventCreate(&r.b) != cudaSuccess) return -1;
    c->prof.push_back(r);
  }
  gnn_ctx::ProfRec& r = c->prof[c->prof_used];
  r.group = group;
  r.launches = launches;
  cudaEventRecord(r.a, st);
  return (int)c->prof_used++;
}
void prof_end(gnn_ctx* c, int idx, cudaStream_t st) {
  if (idx >= 0) cudaEventRecord(c->prof[idx].b, st);
}

template <TileKind K, int H, bool BF>
cudaError_t set_smem_attr() {
  return cudaFuncSetAttribute(mlp_tile_kernel<K, H, BF>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              227 * 1024);
}

template <int H, bool BF>
cudaError_t set_all_attrs() {
  cudaError_t e;
  if ((e = set_smem_attr<TileKind::NodeEncoder, H, BF>()) != cudaSuccess) return e;
  if ((e = set_smem_attr<TileKind::EdgeEncoder, H, BF>()) != cudaSuccess) return e;
  if ((e = set_smem_attr<TileKind::EdgeUpdate, H, BF>()) != cudaSuccess) return e;
  if ((e = set_smem_attr<TileKind::NodeUpdate, H, BF>()) != cudaSuccess) return e;
  if ((e = set_smem_attr<TileKind::Filter, H, BF>()) != cudaSuccess) return e;
  if ((e = set_smem_attr<TileKind::Embed, H, BF>()) != cudaSuccess) return e;
  return set_smem_attr<TileKind::Classifier, H, BF>();
}

template <TileKind K, int H, bool BF>
cudaError_t launch_tile(gnn_ctx* c, const KernelPlan& pl, TileParams p, cudaStream_t st) {
  p.n_jobs = pl.n_jobs;
  // A lies in the region the previous job's D was written to, except where a job keeps its predecessor's
  // regions: it accumulates into the same D, or (the P_d job, last of a node plan) reads the same A.
  const bool node = K == TileKind::NodeEncoder || K == TileKind::NodeUpdate;
  for (int j = 0, areg = 0; j < kMaxJobs; ++j) {
    p.job_mat[j] = pl.job_mat[j];
    p.job_acc[j] = pl.job_acc[j];
    if (j > 0 && !(pl.job_acc[j] || (node && j == pl.n_jobs - 1))) areg ^= 1;
    p.job_areg[j] = areg;
    p.job_bias[j] = pl.job_bias[j];
  }
  p.folded = pl.folded ? 1 : 0;
  p.consts = pl.d_consts;
  p.const_bytes = pl.const_bytes;
  p.vecs = pl.d_vecs;
  p.n_vec_floats = (int)pl.vecs.size();
  p.wmats = pl.wmats ? pl.wmats : c->d_mats;
  p.mat_bytes = c->mat_bytes;
  p.n_tiles = (p.n_rows + kTileRows - 1) / kTileRows;
  if (p.n_tiles == 0) return cudaSuccess;
  const int stages = tile_stages<K, H, BF>(p.n_jobs);
  p.ring_bytes = stages * TileGeom<H, BF>::MAT_BYTES;
  const uint32_t smem = tile_launch_smem<H, BF>(stages, p.n_vec_floats, p.const_bytes);
  const int grid = tile_grid(p.n_tiles, c->n_sm);
  p.early = 2 * grid <= c->n_sm;
#ifdef GNN_TRACE
  p.trace = ((int)K == c->trace_kind) ? c->trace : nullptr;
#endif
  static const int group[7] = {1, 2, 3, 4, 5, 8, 9};   // NodeEncoder, EdgeEncoder, EdgeUpdate, NodeUpdate, Classifier, Filter, Embed
  const int pr = prof_begin(c, group[(int)K], 1, st);
  const cudaError_t err = launch_pdl(mlp_tile_kernel<K, H, BF>, grid, TileRoles<K>::THREADS, smem, st, p);
  prof_end(c, pr, st);
  return err;
}

template <int H, bool BF>
int run_network(gnn_ctx* c, const float* x, int N, int E, float* scores, cudaStream_t st) {
  TileParams p{};
  p.n_nodes = N;
  p.n_layers = c->cfg.mlp_layers;
  p.eps = c->cfg.ln_eps;
  p.x = x;
  p.x_stride = c->cfg.n_node_feat;
  p.src_sorted = c->src_sorted;
  p.dst_sorted = c->dst_sorted;
  p.key_sorted = c->key_sorted;
  p.perm = c->perm;
  p.rowptr = c->rowptr;
  p.e = c->e; p.h = c->h; p.ps = c->ps; p.pd = c->pd; p.agg = c->agg;
  p.scores = scores;
  p.err = c->d_err;
  const int T = c->cfg.n_iters;

  cudaError_t le = cudaSuccess;                        // first launch error
  auto chk = [&](cudaError_t e) { if (le == cudaSuccess) le = e; };
  TileParams pn = p; pn.n_rows = N; pn.n_feat = pn.n_in = c->cfg.n_node_feat;
  chk(launch_tile<TileKind::NodeEncoder, H, BF>(c, c->plan[T > 0 ? 0 : 1], pn, st));
  TileParams pe = p; pe.n_rows = E; pe.n_in = 2;
  chk(launch_tile<TileKind::EdgeEncoder, H, BF>(c, c->plan[2], pe, st));
  for (int t = 1; t <= T; ++t) {
    chk(launch_tile<TileKind::EdgeUpdate, H, BF>(c, c->plan[3], pe, st));
    {
      const int pr = prof_begin(c, 7, 1, st);
      chk(launch_pdl(aggregate_kernel<H, BF>, blocks_for(N, agg_nodes_per_block<H>()), 256, 0, st, (const void*)c->e,
                     (const int*)c->rowptr, N, c->agg));
      prof_end(c, pr, st);
    }
    chk(launch_tile<TileKind::NodeUpdate, H, BF>(c, c->plan[t < T ? 4 : 5], pn, st));
  }
  chk(launch_tile<TileKind::Classifier, H, BF>(c, c->plan[6], pe, st));
  const cudaError_t err = le != cudaSuccess ? le : cudaGetLastError();
  return err == cudaSuccess ? GNN_OK : cuda_fail(err);
}

int64_t state_bytes(const gnn_ctx* c) { return c->cfg.precision == GNN_PRECISION_BF16 ? 2 : 4; }

void free_workspace(gnn_ctx* c) {
  if (c->ws) cudaFree(c->ws);
  c->ws = nullptr;
  c->cap_nodes = c->cap_edges = -1;
}

int ensure_workspace(gnn_ctx* c, int64_t N, int64_t E) {
  if (N <= c->cap_nodes && E <= c->cap_edges) return GNN_OK;
  const int64_t n = N > c->cap_nodes ? N : c->cap_nodes;
  const int64_t e = E > c->cap_edges ? E : c->cap_edges;
  const int64_t H = c->cfg.hidden;
  const int64_t hist_bytes = 4 * (int64_t)radix_hist_ints((size_t)e);
  auto al = [](int64_t b) { return (b + 255) & ~int64_t(255); };
  const int64_t sz_e_int = al(4 * (e > 0 ? e : 1));
  // edge and node state use the row-tiled layout: rows padded to whole 128-row tiles
  const int64_t e_pad = (e + kTileRows - 1) / kTileRows * kTileRows;
  const int64_t n_pad = (n + kTileRows - 1) / kTileRows * kTileRows;
  const int64_t se = state_bytes(c);                   // stored-state element: fp32 or bf16
  const int64_t total = 7 * sz_e_int + al(hist_bytes) + al(4 * (n + 1)) +
                        al(se * e_pad * H) + 2 * al(se * n_pad * H) + 2 * al(4 * n * H);
  free_workspace(c);
  void* ws = nullptr;
  cudaError_t err = dev_alloc(&ws, (size_t)total);
  if (err != cudaSuccess) return cuda_fail(err);
  c->ws = ws;
  uint8_t* q = (uint8_t*)ws;
  auto take = [&](int64_t bytes) { uint8_t* r = q; q += al(bytes); return r; };
  c->keys_a = (int*)take(4 * e); c->keys_b = (int*)take(4 * e);
  c->vals_a = (int*)take(4 * e); c->vals_b = (int*)take(4 * e);
  c->perm = (int*)take(4 * e);
  c->src_sorted = (int*)take(4 * e); c->dst_sorted = (int*)take(4 * e);
  c->hist = (int*)take(hist_bytes);
  c->rowptr = (int*)take(4 * (n + 1));
  c->e = take(se * e_pad * H);
  c->h = take(se * n_pad * H);
  c->agg = take(se * n_pad * H);
  c->ps = (float*)take(4 * n * H);
  c->pd = (float*)take(4 * n * H);
  c->cap_nodes = n;
  c->cap_edges = e;
  return GNN_OK;
}

// Stable sort of n keys in [0, max_key] read through `src` (first pass), values = positions in it, by
// passes that write keys_out[0], keys_out[1], ... in turn (two buffers each).  Returns the index of the
// buffers that hold the result.
template <typename Src>
int launch_radix_sort(const Src& src, int n, int max_key, int* const* keys, int* const* vals, int* hist, cudaStream_t st,
                      cudaError_t* err) {
  auto chk = [&](cudaError_t e) { if (*err == cudaSuccess) *err = e; };
  const RadixPlan plan = radix_plan(max_key);
  const int tiles = (int)blocks_for(n, kRadixTile), bins = 1 << plan.digit;
  int* totals = hist + (size_t)tiles * bins;
  for (int ps = 0; ps < plan.passes; ++ps) {
    const int shift = plan.digit * ps, out = ps & 1;
    const RadixPairs pairs{keys[out ^ 1], vals[out ^ 1]};
    if (ps == 0) chk(launch_pdl(radix_count_kernel<Src>, tiles, kRadixThreads, 0, st, src, n, shift, bins, tiles, hist));
    else chk(launch_pdl(radix_count_kernel<RadixPairs>, tiles, kRadixThreads, 0, st, pairs, n, shift, bins, tiles, hist));
    chk(launch_pdl(radix_scan_kernel, blocks_for(bins, kRadixWarps), kRadixThreads, 0, st, hist, bins, tiles, totals));
    if (ps == 0)
      chk(launch_pdl(radix_scatter_kernel<Src>, tiles, kRadixThreads, 0, st, src, keys[out], vals[out], n, shift, bins,
                     tiles, (const int*)hist, (const int*)totals));
    else
      chk(launch_pdl(radix_scatter_kernel<RadixPairs>, tiles, kRadixThreads, 0, st, pairs, keys[out], vals[out], n, shift,
                     bins, tiles, (const int*)hist, (const int*)totals));
  }
  return (plan.passes - 1) & 1;
}

// The destination-keyed CSR of ei [2, E] into perm, src_sorted, dst_sorted (may be null) and rowptr;
// returns the sorted keys through key_sorted.
cudaError_t launch_csr(const int32_t* ei, int N, int E, int* const* keys, int* const* vals, int* hist, int* perm,
                       int* src_sorted, int* dst_sorted, int* rowptr, uint32_t* d_err, int** key_sorted, cudaStream_t st) {
  constexpr int tb = 256;
  cudaError_t err = cudaSuccess;                       // first launch error
  const int k = launch_radix_sort(RadixEdges{ei, E, N, d_err}, E, N, keys, vals, hist, st, &err);
  const int64_t threads = E > (int64_t)N + 1 ? E : (int64_t)N + 1;
  const cudaError_t e = launch_pdl(csr_finish_kernel, blocks_for(threads, tb), tb, 0, st, ei, (const int*)keys[k],
                                   (const int*)vals[k], E, N, perm, src_sorted, dst_sorted, rowptr);
  if (key_sorted) *key_sorted = keys[k];
  return err != cudaSuccess ? err : e;
}

int build_csr(gnn_ctx* c, const int32_t* ei, int N, int E, cudaStream_t st) {
  const int pr = prof_begin(c, 0, 3 * radix_plan(N).passes + 1, st);
  int* const keys[2] = {c->keys_a, c->keys_b};
  int* const vals[2] = {c->vals_a, c->vals_b};
  const cudaError_t le = launch_csr(ei, N, E, keys, vals, c->hist, c->perm, c->src_sorted, c->dst_sorted, c->rowptr,
                                    c->d_err, &c->key_sorted, st);
  prof_end(c, pr, st);
  const cudaError_t err = le != cudaSuccess ? le : cudaGetLastError();
  return err == cudaSuccess ? GNN_OK : cuda_fail(err);
}

}  // namespace

extern "C" {

const char* gnn_error_string(int code) {
  switch (code) {
    case GNN_OK: return "ok";
    case GNN_ERR_INVALID_ARG: return "invalid argument";
    case GNN_ERR_BAD_WEIGHTS: return "bad weight blob";
    case GNN_ERR_OOM: return "device out of memory";
    case GNN_ERR_CUDA: return "CUDA error";
    case GNN_ERR_INDEX_RANGE: return "edge endpoint out of range";
    case GNN_ERR_DEVICE_TIMEOUT: return "device pipeline wait timed out";
    case GNN_ERR_CAPACITY: return "output buffer too small";
    default: return "unknown status";
  }
}

int gnn_create(const gnn_config* cfg, const void* weights_host, size_t weights_bytes, gnn_ctx** out) {
  if (!cfg || !weights_host || !out) return GNN_ERR_INVALID_ARG;
  *out = nullptr;
  const int H = cfg->hidden, L = cfg->mlp_layers, Fn = cfg->n_node_feat;
  if (cfg->version != 1 || (H != 64 && H != 128) || L < 2 || L > 4 || Fn < 2 || Fn > 16 ||
      cfg->n_edge_feat != 2 || cfg->n_iters < 0 || cfg->n_iters > 64 ||
      (cfg->precision != GNN_PRECISION_FP32 && cfg->precision != GNN_PRECISION_BF16) || !(cfg->ln_eps > 0.f))
    return GNN_ERR_INVALID_ARG;
  if (weights_bytes < (size_t)kHeaderBytes) return GNN_ERR_BAD_WEIGHTS;
  const uint8_t* blob = (const uint8_t*)weights_host;
  int32_t hdr[8];
  float eps;
  int64_t n_floats;
  std::memcpy(hdr, blob, 32);
  std::memcpy(&eps, blob + 32, 4);
  std::memcpy(&n_floats, blob + 40, 8);
  if ((uint32_t)hdr[0] != kBlobMagic || hdr[1] != 1 || hdr[2] != Fn || hdr[3] != 2 || hdr[4] != H ||
      hdr[5] != cfg->n_iters || hdr[6] != L || hdr[7] != cfg->precision || eps != cfg->ln_eps)
    return GNN_ERR_BAD_WEIGHTS;
  const int in1[N_MLP] = {Fn, 2, 3 * H, 2 * H, 3 * H};
  int64_t want = H + 1;
  for (int m = 0; m < N_MLP; ++m) want += (int64_t)H * in1[m] + 3 * H + (int64_t)(L - 1) * (H * H + 3 * H);
  if (n_floats != want || weights_bytes != (size_t)kHeaderBytes + 4 * (size_t)want) return GNN_ERR_BAD_WEIGHTS;

  // locate arrays
  const float* f = (const float*)(blob + kHeaderBytes);
  Layer lay[N_MLP][4];
  for (int m = 0; m < N_MLP; ++m)
    for (int l = 0; l < L; ++l) {
      const int in = l == 0 ? in1[m] : H;
      lay[m][l] = {f, f + (size_t)H * in, f + (size_t)H * in + H, f + (size_t)H * in + 2 * H, in};
      f += (size_t)H * in + 3 * H;
    }
  const float* head_w = f;
  const float* head_b = f + H;

  // Every Linear layer here feeds a LayerNorm, whose first step subtracts the
  // mean over the H outputs.  That subtraction is linear, so it is folded into
  // the layer: each weight column and the bias are centred over the output
  // rows (W' = (I - 11^T/H) W, b' = b - mean(b)).  The kernels then receive
  // zero-mean pre-activations and compute only the variance.  The hidden layers'
  // gammas go into the weights around them (fold_gamma).  Centred and folded
  // copies are kept in `copies` and the Layer pointers redirected to them.
  // The bf16 model keeps its weights as given (bf16 values): centring would take them off the
  // bf16 grid, so its kernels subtract the LayerNorm mean themselves.
  const bool bf = cfg->precision == GNN_PRECISION_BF16;
  MlpCopy copies[N_MLP];
  for (int m = 0; m < N_MLP; ++m) prepare_mlp(lay[m], L, H, bf, true, copies[m]);

  gnn_ctx* c = new (std::nothrow) gnn_ctx();
  if (!c) return GNN_ERR_OOM;
  c->cfg = *cfg;
  cudaError_t err = cudaGetDevice(&c->device);
  if (err == cudaSuccess) err = cudaDeviceGetAttribute(&c->n_sm, cudaDevAttrMultiProcessorCount, c->device);
  if (err == cudaSuccess)
    err = bf ? ((H == 128) ? set_all_attrs<128, true>() : set_all_attrs<64, true>())
             : ((H == 128) ? set_all_attrs<128, false>() : set_all_attrs<64, false>());
  if (err != cudaSuccess) { delete c; return cuda_fail(err); }

  // matrices
  std::vector<std::pair<const Layer*, int>> mats;   // (layer, column offset)
  auto add_mat = [&](const Layer* ly, int col0) { mats.push_back({ly, col0}); return (int)mats.size() - 1; };
  const int en_s = add_mat(&lay[EDGE_NET][0], 0), en_d = add_mat(&lay[EDGE_NET][0], H),
            en_e = add_mat(&lay[EDGE_NET][0], 2 * H);
  const int cl_s = add_mat(&lay[CLASSIFIER][0], 0), cl_d = add_mat(&lay[CLASSIFIER][0], H),
            cl_e = add_mat(&lay[CLASSIFIER][0], 2 * H);
  const int nn_h = add_mat(&lay[NODE_NET][0], 0), nn_a = add_mat(&lay[NODE_NET][0], H);
  int deep[N_MLP][4];
  for (int m = 0; m < N_MLP; ++m)
    for (int l = 1; l < L; ++l) deep[m][l] = add_mat(&lay[m][l], 0);
  const int in_node = add_mat(&lay[NODE_ENC][0], -1), in_edge = add_mat(&lay[EDGE_ENC][0], -1);   // input matrices
  c->mat_bytes = (bf ? 1u : 2u) * H * H * 2u;
  std::vector<uint8_t> packed((size_t)c->mat_bytes * mats.size());
  for (size_t i = 0; i < mats.size(); ++i) {
    uint8_t* out = packed.data() + i * c->mat_bytes;
    if (mats[i].second < 0) pack_input(mats[i].first->W, mats[i].first->in, H, bf, out, c->mat_bytes);
    else pack_block(mats[i].first->W, mats[i].first->in, mats[i].second, H, !bf, out);
  }

  // kernel plans
  auto jobs = [](KernelPlan& pl, std::initializer_list<int> ids, int acc_mask = 0) {
    pl.n_jobs = 0;
    for (int id : ids) { pl.job_acc[pl.n_jobs] = (acc_mask >> pl.n_jobs) & 1; pl.job_mat[pl.n_jobs++] = id; }
  };
  auto add_deep = [&](KernelPlan& pl, int m) {
    pl.folded = copies[m].folded;
    for (int l = 1; l < L; ++l) {
      set_bias(pl, pl.n_jobs, lay[m][l].b);
      pl.job_acc[pl.n_jobs] = 0;
      pl.job_mat[pl.n_jobs++] = deep[m][l];
    }
  };
  auto gb = [&](std::vector<float>& v, int m) {
    for (int l = 0; l < L; ++l) push_ln(v, lay[m][l], H);
  };
  for (int target = 0; target < 2; ++target) {           // node encoder -> edge net / classifier
    KernelPlan& pl = c->plan[target];
    jobs(pl, {in_node});
    set_bias(pl, 0, lay[NODE_ENC][0].b);
    add_deep(pl, NODE_ENC);
    pl.job_mat[pl.n_jobs++] = target == 0 ? en_s : cl_s;
    pl.job_mat[pl.n_jobs++] = target == 0 ? en_d : cl_d;
    gb(pl.vecs, NODE_ENC);
    set_bias(pl, pl.n_jobs - 1, lay[target == 0 ? EDGE_NET : CLASSIFIER][0].b);   // P_d carries it
  }
  {  // edge encoder
    KernelPlan& pl = c->plan[2];
    jobs(pl, {in_edge});
    set_bias(pl, 0, lay[EDGE_ENC][0].b);
    add_deep(pl, EDGE_ENC);
    gb(pl.vecs, EDGE_ENC);
  }
  {  // edge update
    KernelPlan& pl = c->plan[3];
    jobs(pl, {en_e});
    add_deep(pl, EDGE_NET);
    gb(pl.vecs, EDGE_NET);
  }
  for (int target = 0; target < 2; ++target) {           // node update -> edge net / classifier
    KernelPlan& pl = c->plan[4 + target];
    jobs(pl, {nn_h, nn_a}, 0b10);
    set_bias(pl, 0, lay[NODE_NET][0].b);
    add_deep(pl, NODE_NET);
    pl.job_acc[pl.n_jobs] = 0; pl.job_mat[pl.n_jobs++] = target == 0 ? en_s : cl_s;
    pl.job_acc[pl.n_jobs] = 0; pl.job_mat[pl.n_jobs++] = target == 0 ? en_d : cl_d;
    gb(pl.vecs, NODE_NET);
    set_bias(pl, pl.n_jobs - 1, lay[target == 0 ? EDGE_NET : CLASSIFIER][0].b);   // P_d carries it
  }
  {  // classifier
    KernelPlan& pl = c->plan[6];
    jobs(pl, {cl_e});
    add_deep(pl, CLASSIFIER);
    gb(pl.vecs, CLASSIFIER);
    push(pl.vecs, head_w, H);
    push(pl.vecs, head_b, 1);
  }

  for (int i = 0; i < 7; ++i) finish_vecs(c->plan[i].vecs, H);
  err = dev_alloc((void**)&c->d_mats, packed.size());
  if (err == cudaSuccess) err = cudaMemcpy(c->d_mats, packed.data(), packed.size(), cudaMemcpyHostToDevice);
  for (int i = 0; i < 7 && err == cudaSuccess; ++i) err = upload_plan(c->plan[i], H);
#ifdef GNN_TRACE
  if (err == cudaSuccess) err = cudaMalloc(&c->trace, 3 * kTraceEvents * 8);
  if (err == cudaSuccess) err = cudaMemset(c->trace, 0, 3 * kTraceEvents * 8);
  if (const char* k = getenv("GNN_TRACE_KIND")) c->trace_kind = atoi(k);
#endif
  if (err == cudaSuccess) err = dev_alloc((void**)&c->d_err, 4);
  if (err == cudaSuccess) err = cudaMemset(c->d_err, 0, 4);
  if (err != cudaSuccess) { gnn_destroy(c); return cuda_fail(err); }
  *out = c;
  return GNN_OK;
}

int gnn_reserve(gnn_ctx* ctx, int64_t max_nodes, int64_t max_edges) {
  if (!count_ok(max_nodes) || !count_ok(max_edges) || !ctx) return GNN_ERR_INVALID_ARG;
  return ensure_workspace(ctx, max_nodes, max_edges);
}

int gnn_infer(gnn_ctx* ctx, const float* node_feats, const int32_t* edge_index, int64_t n_nodes,
              int64_t n_edges, float* edge_scores, gnn_stream_t stream) {
  if (!count_ok(n_nodes) || !count_ok(n_edges) || !ctx) return GNN_ERR_INVALID_ARG;
  if (n_edges == 0) return GNN_OK;
  if (n_nodes == 0 || !node_feats || !edge_index || !edge_scores) return GNN_ERR_INVALID_ARG;
  int rc = ensure_workspace(ctx, n_nodes, n_edges);
  if (rc != GNN_OK) return rc;
  cudaStream_t st = (cudaStream_t)stream;
  const int N = (int)n_nodes, E = (int)n_edges;
  rc = build_csr(ctx, edge_index, N, E, st);
  if (rc != GNN_OK) return rc;
  ctx->last_nodes = N;
  ctx->last_edges = E;
  const bool bf = ctx->cfg.precision == GNN_PRECISION_BF16;
  if (ctx->cfg.hidden == 128)
    return bf ? run_network<128, true>(ctx, node_feats, N, E, edge_scores, st)
              : run_network<128, false>(ctx, node_feats, N, E, edge_scores, st);
  return bf ? run_network<64, true>(ctx, node_feats, N, E, edge_scores, st)
            : run_network<64, false>(ctx, node_feats, N, E, edge_scores, st);
}

int gnn_infer_host(gnn_ctx* ctx, const float* node_feats, const int32_t* edge_index, int64_t n_nodes,
                   int64_t n_edges, float* edge_scores, gnn_stream_t stream) {
  if (!count_ok(n_nodes) || !count_ok(n_edges) || !ctx) return GNN_ERR_INVALID_ARG;
  if (n_edges == 0) return GNN_OK;
  if (n_nodes == 0 || !node_feats || !edge_index || !edge_scores) return GNN_ERR_INVALID_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  const size_t bx = (size_t)n_nodes * ctx->cfg.n_node_feat * 4, be = (size_t)n_edges * 8,
               bs = (size_t)n_edges * 4;
  auto al = [](size_t b) { return (b + 255) & ~size_t(255); };
  const size_t need = al(bx) + al(be) + al(bs);
  if (need > ctx->stage_bytes) {
    if (ctx->stage) { cudaStreamSynchronize(st); cudaFree(ctx->stage); ctx->stage = nullptr; ctx->stage_bytes = 0; }
    const cudaError_t err = dev_alloc(&ctx->stage, need);
    if (err != cudaSuccess) return cuda_fail(err);
    ctx->stage_bytes = need;
  }
  uint8_t* q = (uint8_t*)ctx->stage;
  float* dx = (float*)q;
  int32_t* de = (int32_t*)(q + al(bx));
  float* ds = (float*)(q + al(bx) + al(be));
  int pr = prof_begin(ctx, 6, 2, st);
  cudaError_t err = cudaMemcpyAsync(dx, node_feats, bx, cudaMemcpyHostToDevice, st);
  if (err == cudaSuccess) err = cudaMemcpyAsync(de, edge_index, be, cudaMemcpyHostToDevice, st);
  prof_end(ctx, pr, st);
  if (err != cudaSuccess) return cuda_fail(err);
  int rc = gnn_infer(ctx, dx, de, n_nodes, n_edges, ds, stream);
  if (rc != GNN_OK) return rc;
  pr = prof_begin(ctx, 6, 1, st);
  err = cudaMemcpyAsync(edge_scores, ds, bs, cudaMemcpyDeviceToHost, st);
  prof_end(ctx, pr, st);
  if (err != cudaSuccess) return cuda_fail(err);
  return gnn_status(ctx, stream);
}

int gnn_filter_load(gnn_ctx* ctx, const void* weights_host, size_t weights_bytes) {
  if (!ctx || !weights_host) return GNN_ERR_INVALID_ARG;
  const int H = ctx->cfg.hidden, Fn = ctx->cfg.n_node_feat;
  const bool bf = ctx->cfg.precision == GNN_PRECISION_BF16;
  if (weights_bytes < (size_t)kHeaderBytes) return GNN_ERR_BAD_WEIGHTS;
  const uint8_t* blob = (const uint8_t*)weights_host;
  int32_t hdr[8];
  float eps;
  int64_t n_floats;
  std::memcpy(hdr, blob, 32);
  std::memcpy(&eps, blob + 32, 4);
  std::memcpy(&n_floats, blob + 40, 8);
  const int L = hdr[4];
  if ((uint32_t)hdr[0] != kFilterMagic || hdr[1] != 1 || hdr[2] != Fn || hdr[3] != H || L < 2 || L > 4 ||
      hdr[5] != ctx->cfg.precision || !(eps > 0.f))
    return GNN_ERR_BAD_WEIGHTS;
  const int64_t want = (int64_t)H * 2 * Fn + 3 * H + (int64_t)(L - 1) * (H * H + 3 * H) + H + 1;
  if (n_floats != want || weights_bytes != (size_t)kHeaderBytes + 4 * (size_t)want) return GNN_ERR_BAD_WEIGHTS;
  const float* f = (const float*)(blob + kHeaderBytes);
  std::vector<Layer> lay(L);
  for (int l = 0; l < L; ++l) {
    const int in = l == 0 ? 2 * Fn : H;
    lay[l] = {f, f + (size_t)H * in, f + (size_t)H * in + H, f + (size_t)H * in + 2 * H, in};
    f += (size_t)H * in + 3 * H;
  }
  const float* head = f;
  MlpCopy copy;
  prepare_mlp(lay.data(), L, H, bf, true, copy);
  KernelPlan pl;
  pl.folded = copy.folded;
  for (int l = 0; l < L; ++l) {                       // job and matrix l: layer l, the first an input matrix
    set_bias(pl, l, lay[l].b);
    pl.job_mat[l] = l;
  }
  pl.n_jobs = L;
  for (int l = 0; l < L; ++l) push_ln(pl.vecs, lay[l], H);
  push(pl.vecs, head, H + 1);
  finish_vecs(pl.vecs, H);
  std::vector<uint8_t> packed((size_t)ctx->mat_bytes * L);
  pack_input(lay[0].W, lay[0].in, H, bf, packed.data(), ctx->mat_bytes);
  for (int l = 1; l < L; ++l) pack_block(lay[l].W, H, 0, H, !bf, packed.data() + (size_t)l * ctx->mat_bytes);
  // replace a previous filter
  if (ctx->filter_plan.d_vecs) { cudaFree(ctx->filter_plan.d_vecs); ctx->filter_plan.d_vecs = nullptr; }
  if (ctx->d_filter_mats) { cudaFree(ctx->d_filter_mats); ctx->d_filter_mats = nullptr; }
  ctx->filter_layers = 0;
  cudaError_t err = dev_alloc((void**)&ctx->d_filter_mats, packed.size());
  if (err == cudaSuccess) err = cudaMemcpy(ctx->d_filter_mats, packed.data(), packed.size(), cudaMemcpyHostToDevice);
  if (err == cudaSuccess) err = upload_plan(pl, H);
  if (err != cudaSuccess) {
    if (pl.d_vecs) cudaFree(pl.d_vecs);
    if (ctx->d_filter_mats) { cudaFree(ctx->d_filter_mats); ctx->d_filter_mats = nullptr; }
    return cuda_fail(err);
  }
  pl.wmats = ctx->d_filter_mats;
  ctx->filter_plan = std::move(pl);
  ctx->filter_layers = L;
  ctx->filter_eps = eps;
  return GNN_OK;
}

int gnn_filter_edges(gnn_ctx* ctx, const float* node_feats, const int32_t* edge_index, int64_t n_nodes,
                     int64_t n_edges, float threshold, float* edge_scores, int32_t* kept_index, int32_t* kept_id,
                     int32_t* n_kept, gnn_stream_t stream) {
  if (!count_ok(n_nodes) || !count_ok(n_edges) || !ctx || !n_kept) return GNN_ERR_INVALID_ARG;
  if (ctx->filter_layers == 0) return GNN_ERR_INVALID_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  if (n_edges == 0) {
    const cudaError_t err = cudaMemsetAsync(n_kept, 0, sizeof(int32_t), st);
    return err == cudaSuccess ? GNN_OK : cuda_fail(err);
  }
  if (n_nodes == 0 || !node_feats || !edge_index || !edge_scores || !kept_index) return GNN_ERR_INVALID_ARG;
  int rc = ensure_workspace(ctx, n_nodes, n_edges);          // block counts live in the sort keys' buffer
  if (rc != GNN_OK) return rc;
  const int N = (int)n_nodes, E = (int)n_edges;
  TileParams p{};
  p.n_rows = E;
  p.n_nodes = N;
  p.n_layers = ctx->filter_layers;
  p.n_feat = ctx->cfg.n_node_feat;
  p.n_in = 2 * p.n_feat;
  p.eps = ctx->filter_eps;
  p.x = node_feats;
  p.x_stride = ctx->cfg.n_node_feat;
  p.ei_in = edge_index;
  p.scores = edge_scores;
  p.err = ctx->d_err;
  const bool bf = ctx->cfg.precision == GNN_PRECISION_BF16;
  if (ctx->cfg.hidden == 128) {
    if (bf) launch_tile<TileKind::Filter, 128, true>(ctx, ctx->filter_plan, p, st);
    else launch_tile<TileKind::Filter, 128, false>(ctx, ctx->filter_plan, p, st);
  } else {
    if (bf) launch_tile<TileKind::Filter, 64, true>(ctx, ctx->filter_plan, p, st);
    else launch_tile<TileKind::Filter, 64, false>(ctx, ctx->filter_plan, p, st);
  }
  const int tiles = compact_tiles(E), nb = compact_blocks(E);
  int* counts = ctx->keys_a;
  cudaError_t err = launch_pdl(compact_count_kernel, nb, kCompactThreads, 0, st, (const float*)edge_scores, E, threshold,
                               tiles, counts);
  if (err == cudaSuccess)
    err = launch_pdl(compact_scatter_kernel, nb, kCompactThreads, 0, st, (const float*)edge_scores, edge_index, E,
                     threshold, tiles, (const int*)counts, n_kept, kept_index, kept_id);
  if (err != cudaSuccess) return cuda_fail(err);
  err = cudaGetLastError();
  return err == cudaSuccess ? GNN_OK : cuda_fail(err);
}

int gnn_embed_load(gnn_ctx* ctx, const void* weights_host, size_t weights_bytes) {
  if (!ctx || !weights_host) return GNN_ERR_INVALID_ARG;
  const int H = ctx->cfg.hidden, Fn = ctx->cfg.n_node_feat;
  const bool bf = ctx->cfg.precision == GNN_PRECISION_BF16;
  if (weights_bytes < (size_t)kHeaderBytes) return GNN_ERR_BAD_WEIGHTS;
  const uint8_t* blob = (const uint8_t*)weights_host;
  int32_t hdr[8];
  float eps;
  int64_t n_floats;
  std::memcpy(hdr, blob, 32);
  std::memcpy(&eps, blob + 32, 4);
  std::memcpy(&n_floats, blob + 40, 8);
  const int L = hdr[4], D = hdr[6];
  if ((uint32_t)hdr[0] != kEmbedMagic || hdr[1] != 1 || hdr[2] != Fn || hdr[3] != H || L < 2 || L > 4 ||
      hdr[5] != ctx->cfg.precision || D < 1 || D > kMaxEmbedDim || !(eps > 0.f))
    return GNN_ERR_BAD_WEIGHTS;
  const int64_t want = (int64_t)H * Fn + 3 * H + (int64_t)(L - 1) * (H * H + 3 * H) + (int64_t)D * H + D;
  if (n_floats != want || weights_bytes != (size_t)kHeaderBytes + 4 * (size_t)want) return GNN_ERR_BAD_WEIGHTS;
  const float* f = (const float*)(blob + kHeaderBytes);
  std::vector<Layer> lay(L);
  for (int l = 0; l < L; ++l) {
    const int in = l == 0 ? Fn : H;
    lay[l] = {f, f + (size_t)H * in, f + (size_t)H * in + H, f + (size_t)H * in + 2 * H, in};
    f += (size_t)H * in + 3 * H;
  }
  const float* wout = f;                                  // [D, H] then b_out [D]
  MlpCopy copy;
  prepare_mlp(lay.data(), L, H, bf, false, copy);
  KernelPlan pl;
  pl.folded = copy.folded;
  for (int l = 0; l < L; ++l) {                       // job and matrix l: layer l, the first an input matrix
    set_bias(pl, l, lay[l].b);
    pl.job_mat[l] = l;
  }
  pl.n_jobs = L;
  for (int l = 0; l < L; ++l) push_ln(pl.vecs, lay[l], H);
  push(pl.vecs, wout, (size_t)D * H + D);
  finish_vecs(pl.vecs, H);
  std::vector<uint8_t> packed((size_t)ctx->mat_bytes * L);
  pack_input(lay[0].W, lay[0].in, H, bf, packed.data(), ctx->mat_bytes);
  for (int l = 1; l < L; ++l) pack_block(lay[l].W, H, 0, H, !bf, packed.data() + (size_t)l * ctx->mat_bytes);
  if (ctx->embed_plan.d_vecs) { cudaFree(ctx->embed_plan.d_vecs); ctx->embed_plan.d_vecs = nullptr; }
  if (ctx->d_embed_mats) { cudaFree(ctx->d_embed_mats); ctx->d_embed_mats = nullptr; }
  ctx->embed_layers = 0;
  cudaError_t err = dev_alloc((void**)&ctx->d_embed_mats, packed.size());
  if (err == cudaSuccess) err = cudaMemcpy(ctx->d_embed_mats, packed.data(), packed.size(), cudaMemcpyHostToDevice);
  if (err == cudaSuccess) err = upload_plan(pl, H);
  if (err != cudaSuccess) {
    if (pl.d_vecs) cudaFree(pl.d_vecs);
    if (ctx->d_embed_mats) { cudaFree(ctx->d_embed_mats); ctx->d_embed_mats = nullptr; }
    return cuda_fail(err);
  }
  pl.wmats = ctx->d_embed_mats;
  ctx->embed_plan = std::move(pl);
  ctx->embed_layers = L;
  ctx->embed_dim = D;
  ctx->embed_eps = eps;
  return GNN_OK;
}

int gnn_embed(gnn_ctx* ctx, const float* node_feats, int64_t n_nodes, float* embedding, gnn_stream_t stream) {
  if (!count_ok(n_nodes) || !ctx || ctx->embed_layers == 0) return GNN_ERR_INVALID_ARG;
  if (n_nodes == 0) return GNN_OK;
  if (!node_feats || !embedding) return GNN_ERR_INVALID_ARG;
  TileParams p{};
  p.n_rows = (int)n_nodes;
  p.n_nodes = (int)n_nodes;
  p.n_layers = ctx->embed_layers;
  p.n_feat = p.n_in = ctx->cfg.n_node_feat;
  p.eps = ctx->embed_eps;
  p.x = node_feats;
  p.x_stride = ctx->cfg.n_node_feat;
  p.emb = embedding;
  p.emb_dim = ctx->embed_dim;
  p.err = ctx->d_err;
  cudaStream_t st = (cudaStream_t)stream;
  const bool bf = ctx->cfg.precision == GNN_PRECISION_BF16;
  if (ctx->cfg.hidden == 128) {
    if (bf) launch_tile<TileKind::Embed, 128, true>(ctx, ctx->embed_plan, p, st);
    else launch_tile<TileKind::Embed, 128, false>(ctx, ctx->embed_plan, p, st);
  } else {
    if (bf) launch_tile<TileKind::Embed, 64, true>(ctx, ctx->embed_plan, p, st);
    else launch_tile<TileKind::Embed, 64, false>(ctx, ctx->embed_plan, p, st);
  }
  const cudaError_t err = cudaGetLastError();
  return err == cudaSuccess ? GNN_OK : cuda_fail(err);
}

int gnn_build_graph(gnn_ctx* ctx, const float* embedding, int emb_dim, const float* node_feats, int64_t n_nodes,
                    float radius, int64_t max_edges, int32_t* edge_index, int32_t* n_edges, gnn_stream_t stream) {
  if (!count_ok(n_nodes) || !count_ok(max_edges) || !ctx || emb_dim < 1 || emb_dim > kMaxEmbedDim ||
      !(radius > 0.f) || !n_edges)
    return GNN_ERR_INVALID_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  if (n_nodes == 0) {
    const cudaError_t err = cudaMemsetAsync(n_edges, 0, sizeof(int32_t), st);
    return err == cudaSuccess ? GNN_OK : cuda_fail(err);
  }
  if (!embedding || !node_feats || (max_edges > 0 && !edge_index)) return GNN_ERR_INVALID_ARG;
  const int N = (int)n_nodes, tb = 256;
  // grid over 4 embedding coordinates when there are at least 4 (on the full event's 8-dimensional
  // embedding, when the writing pass still searched again: 9.0 ms against 14.8 ms with 3), else over 3
  const int K = emb_dim >= 4 ? 4 : 3;
  const int grid = frnn_grid(radius, K);
  int n_cells = 1;
  for (int k = 0; k < K; ++k) n_cells *= grid;
  const int chunks = (emb_dim + 3) / 4;                   // float4 chunks per sorted embedding
  // partner chains kept by the counting pass: one first chunk per hit, pool chunks after them (a hit
  // whose chain cannot grow is searched again by the writing pass)
  const int64_t pool64 = ctx->graph_pool >= 0 ? ctx->graph_pool : (int64_t)N;
  int pool = (int)(pool64 < (int64_t)INT_MAX - N ? pool64 : (int64_t)INT_MAX - N);
  // scratch: emb_s [N, 4 * chunks] (first, 16-byte aligned), partner chunks, r_s, keys/vals (two
  // buffers each), per-hit counts, per-block sums, radix histograms, cell starts, the pool counter
  const int nb = (int)blocks_for(N, tb);
  // B fragments of the pair filter: 16 bytes x 32 lanes per eight hits and set of eight coordinates
  const int sets = (chunks + 1) / 2;
  const size_t frag_ints = ((size_t)N + 7) / 8 * 128 * (size_t)sets;
  const size_t fixed = 4 * (size_t)chunks * N + frag_ints + (size_t)N * kFrnnChunk + 6 * (size_t)N + (size_t)nb +
                       radix_hist_ints(N) + (size_t)n_cells + 2;
  // Where memory does not hold the default pool, the build goes on without one: the same edges, found twice
  // for hits with more than 15 partners.  A scratch made so (aux_tight) is kept for calls that it can serve.
  if (ctx->aux_tight && ctx->graph_pool < 0 && fixed <= ctx->aux_ints)
    pool = (int)std::min<size_t>(pool, (ctx->aux_ints - fixed) / kFrnnChunk);
  const size_t need = fixed + (size_t)pool * kFrnnChunk;
  if (need > ctx->aux_ints) {
    if (ctx->aux) { cudaStreamSynchronize(st); cudaFree(ctx->aux); ctx->aux = nullptr; ctx->aux_ints = 0; }
    ctx->aux_tight = false;
    size_t ints = need;
    cudaError_t err = dev_alloc((void**)&ctx->aux, ints * sizeof(int));
    if (err == cudaErrorMemoryAllocation && ctx->graph_pool < 0) {
      (void)cudaGetLastError();
      ctx->aux_tight = true;
      pool = 0;
      ints = fixed;
      err = dev_alloc((void**)&ctx->aux, ints * sizeof(int));
    }
    if (err != cudaSuccess) return cuda_fail(err);
    ctx->aux_ints = ints;
  }
  const size_t chain_ints = ((size_t)N + (size_t)pool) * kFrnnChunk;
  float4* emb_s = (float4*)ctx->aux;
  uint4* frag = (uint4*)(ctx->aux + 4 * (size_t)chunks * N);
  int* chains = (int*)frag + frag_ints;
  float* r_s = (float*)(chains + chain_ints);
  int* keys_a = (int*)(r_s + N);
  int* keys_b = keys_a + N;
  int* vals_a = keys_b + N;
  int* vals_b = vals_a + N;
  int* counts = vals_b + N;
  int* cells = counts;                                    // the hits' cells, until they are sorted
  int* block_sums = counts + N;
  int* hist = block_sums + nb;
  int* cell_start = hist + radix_hist_ints(N);
  int* next_chunk = cell_start + n_cells + 1;
  cudaError_t le = cudaSuccess;                           // first launch error
  auto chk = [&](cudaError_t e) { if (le == cudaSuccess) le = e; };
  if (K == 4) chk(launch_pdl(frnn_cell_kernel<4>, nb, tb, 0, st, embedding, N, emb_dim, grid, cells, next_chunk));
  else chk(launch_pdl(frnn_cell_kernel<3>, nb, tb, 0, st, embedding, N, emb_dim, grid, cells, next_chunk));
  int* const skeys[2] = {keys_a, keys_b};
  int* const svals[2] = {vals_a, vals_b};
  const int sorted = launch_radix_sort(RadixKeys{cells}, N, n_cells - 1, skeys, svals, hist, st, &le);
  if (le != cudaSuccess) return cuda_fail(le);
  const int *kin = skeys[sorted], *vin = svals[sorted];
  const float r2 = radius * radius;
  const int xs = ctx->cfg.n_node_feat;
  const int sb = compact_blocks(N), scan_tiles = compact_tiles(N);
  const int pb = (int)blocks_for(N, kFrnnBlockQueries);
  const int fb = (int)blocks_for(blocks_for(N, 8) * (int64_t)32, tb);
  const int cb = (int)blocks_for((int64_t)N * kFrnnCopyLanes, tb);
  const int sc = (int)blocks_for((int64_t)n_cells + 1, tb);
  switch (chunks * 8 + K) {
#define GNN_FRNN_CASE(CH, KK)                                                                                    \
  case CH * 8 + KK:                                                                                              \
    chk(launch_pdl(frnn_layout_kernel<CH>, fb + sc, tb, 0, st, embedding, node_feats, xs, N, emb_dim, vin, kin, n_cells,\
                   fb, (float2*)emb_s, r_s, frag, cell_start));                                                        \
    if (KK == 3 && N >= kFrnnSingleHits)                                                                               \
      chk(launch_pdl(frnn_single_kernel, blocks_for(N, kFrnnSingleThreads), kFrnnSingleThreads, 0, st, emb_s, N, r2,   \
                     grid, kin, cell_start, counts, chains, next_chunk, pool));                                        \
    else                                                                                                               \
      chk(launch_pdl(frnn_pairs_kernel<CH, KK>, pb, kFrnnPairsThreads, 0, st, emb_s, frag, r_s, N, r2, grid, kin, vin, \
                     cell_start, 0, counts, nullptr, 0, nullptr, chains, next_chunk, pool, ctx->d_err));               \
    chk(launch_pdl(scan_reduce_kernel, sb, kScanBlock, 0, st, counts, N, scan_tiles, block_sums));                     \
    chk(launch_pdl(scan_apply_kernel, sb, kScanBlock, 0, st, counts, N, scan_tiles, block_sums, n_edges));             \
    chk(launch_pdl(frnn_pairs_kernel<CH, KK>, pb, kFrnnPairsThreads, 0, st, emb_s, frag, r_s, N, r2, grid, kin, vin,   \
                   cell_start, 1, counts, n_edges, (int)max_edges, edge_index, chains, next_chunk, pool, ctx->d_err)); \
    chk(launch_pdl(frnn_copy_kernel, cb, tb, 0, st, r_s, N, vin, counts, n_edges, (int)max_edges, chains, edge_index));\
    break;
    GNN_FRNN_CASE(1, 3)
    GNN_FRNN_CASE(2, 3)
    GNN_FRNN_CASE(3, 3)
    GNN_FRNN_CASE(4, 3)
    GNN_FRNN_CASE(1, 4)
    GNN_FRNN_CASE(2, 4)
    GNN_FRNN_CASE(3, 4)
    GNN_FRNN_CASE(4, 4)
#undef GNN_FRNN_CASE
  }
  if (le != cudaSuccess) return cuda_fail(le);
  const cudaError_t err = cudaGetLastError();
  return err == cudaSuccess ? GNN_OK : cuda_fail(err);
}

int gnn_track_labels(gnn_ctx* ctx, const float* edge_scores, const int32_t* edge_index, int64_t n_nodes,
                     int64_t n_edges, float threshold, int32_t* labels, gnn_stream_t stream) {
  if (!count_ok(n_nodes) || !count_ok(n_edges) || !ctx) return GNN_ERR_INVALID_ARG;
  if (n_nodes == 0) return n_edges == 0 ? GNN_OK : GNN_ERR_INVALID_ARG;
  if (!labels || (n_edges > 0 && (!edge_scores || !edge_index))) return GNN_ERR_INVALID_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  const int N = (int)n_nodes, E = (int)n_edges, tb = 256;
  cudaError_t le = launch_pdl(cc_init_kernel, blocks_for(N, tb), tb, 0, st, labels, N);
  if (le == cudaSuccess && E > 0)
    le = launch_pdl(cc_union_kernel, blocks_for(E, tb), tb, 0, st, edge_scores, edge_index, N, E, threshold, labels, ctx->d_err);
  if (le == cudaSuccess) le = launch_pdl(cc_flatten_kernel, blocks_for(N, tb), tb, 0, st, labels, N, ctx->d_err);
  if (le != cudaSuccess) return cuda_fail(le);
  const cudaError_t err = cudaGetLastError();
  return err == cudaSuccess ? GNN_OK : cuda_fail(err);
}

#ifdef GNN_TRACE
int gnn_trace_read(gnn_ctx* ctx, unsigned long long* host) {
  cudaDeviceSynchronize();
  return cudaMemcpy(host, ctx->trace, 3 * kTraceEvents * 8, cudaMemcpyDeviceToHost) == cudaSuccess ? 0 : -4;
}
#endif

int gnn_debug_fail_allocs(int n) {
  if (n < 0) return GNN_ERR_INVALID_ARG;
  g_fail_allocs.store(n);
  return GNN_OK;
}

int gnn_debug_graph_pool(gnn_ctx* ctx, int64_t chunks) {
  if (!ctx) return GNN_ERR_INVALID_ARG;
  ctx->graph_pool = chunks < 0 ? -1 : chunks;
  return GNN_OK;
}

int gnn_debug_wait_timeout(gnn_ctx* ctx, int64_t limit_ns, gnn_stream_t stream) {
  if (!ctx || limit_ns <= 0 || limit_ns > (int64_t)kWaitLimitNs) return GNN_ERR_INVALID_ARG;
  wait_timeout_kernel<<<1, 32, 0, (cudaStream_t)stream>>>((uint64_t)limit_ns, ctx->d_err);
  const cudaError_t err = cudaGetLastError();
  return err == cudaSuccess ? GNN_OK : cuda_fail(err);
}

int gnn_profile_enable(gnn_ctx* ctx, int on) {
  if (!ctx) return GNN_ERR_INVALID_ARG;
  ctx->prof_on = on != 0;
  return GNN_OK;
}

int gnn_profile_read(gnn_ctx* ctx, double* ms, int64_t* launches, int n_groups) {
  if (!ctx || n_groups < 0) return GNN_ERR_INVALID_ARG;
  double acc[kProfGroups] = {0};
  int64_t cnt[kProfGroups] = {0};
  for (size_t i = 0; i < ctx->prof_used; ++i) {
    gnn_ctx::ProfRec& r = ctx->prof[i];
    if (cudaEventSynchronize(r.b) != cudaSuccess) return cuda_fail(cudaGetLastError());
    float t = 0.f;
    if (cudaEventElapsedTime(&t, r.a, r.b) != cudaSuccess) return cuda_fail(cudaGetLastError());
    acc[r.group] += t;
    cnt[r.group] += r.launches;
  }
  ctx->prof_used = 0;
  for (int g = 0; g < n_groups && g < kProfGroups; ++g) {
    if (ms) ms[g] = acc[g];
    if (launches) launches[g] = cnt[g];
  }
  return kProfGroups;
}

int gnn_status(gnn_ctx* ctx, gnn_stream_t stream) {
  if (!ctx) return GNN_ERR_INVALID_ARG;
  cudaError_t err = cudaStreamSynchronize((cudaStream_t)stream);
  if (err != cudaSuccess) return cuda_fail(err);
  uint32_t word = 0;
  err = cudaMemcpy(&word, ctx->d_err, 4, cudaMemcpyDeviceToHost);
  if (err == cudaSuccess) err = cudaMemset(ctx->d_err, 0, 4);
  if (err != cudaSuccess) return cuda_fail(err);
  if (word & DEV_ERR_TIMEOUT) return GNN_ERR_DEVICE_TIMEOUT;
  if (word & DEV_ERR_CAPACITY) return GNN_ERR_CAPACITY;
  if (word & DEV_ERR_INDEX_RANGE) return GNN_ERR_INDEX_RANGE;
  return GNN_OK;
}

void gnn_destroy(gnn_ctx* ctx) {
  if (!ctx) return;
  cudaDeviceSynchronize();
  free_workspace(ctx);
  if (ctx->d_mats) cudaFree(ctx->d_mats);
  for (int i = 0; i < 7; ++i)
    if (ctx->plan[i].d_vecs) cudaFree(ctx->plan[i].d_vecs);
  if (ctx->filter_plan.d_vecs) cudaFree(ctx->filter_plan.d_vecs);
  if (ctx->d_filter_mats) cudaFree(ctx->d_filter_mats);
  if (ctx->embed_plan.d_vecs) cudaFree(ctx->embed_plan.d_vecs);
  if (ctx->d_embed_mats) cudaFree(ctx->d_embed_mats);
  if (ctx->aux) cudaFree(ctx->aux);
  if (ctx->d_err) cudaFree(ctx->d_err);
  if (ctx->stage) cudaFree(ctx->stage);
#ifdef GNN_TRACE
  if (ctx->trace) cudaFree(ctx->trace);
#endif
  for (auto& r : ctx->prof) { cudaEventDestroy(r.a); cudaEventDestroy(r.b); }
  delete ctx;
}

int gnn_debug_copy(gnn_ctx* ctx, int which, void* dst, size_t bytes, gnn_stream_t stream) {
  if (!ctx || !dst || !ctx->ws) return GNN_ERR_INVALID_ARG;
  const int64_t N = ctx->last_nodes, E = ctx->last_edges, H = ctx->cfg.hidden;
  const void* src = nullptr;
  size_t need = 0;
  switch (which) {
    case 0: src = ctx->rowptr; need = 4 * (size_t)(N + 1); break;
    case 1: src = ctx->perm; need = 4 * (size_t)E; break;
    case 2: src = ctx->src_sorted; need = 4 * (size_t)E; break;
    case 3: src = ctx->h; need = state_bytes(ctx) * (size_t)((N + kTileRows - 1) / kTileRows * kTileRows * H); break;
    case 4: src = ctx->e; need = state_bytes(ctx) * (size_t)((E + kTileRows - 1) / kTileRows * kTileRows * H); break;
    default: return GNN_ERR_INVALID_ARG;
  }
  if (bytes < need) return GNN_ERR_INVALID_ARG;
  const cudaError_t err = cudaMemcpyAsync(dst, src, need, cudaMemcpyDeviceToDevice, (cudaStream_t)stream);
  return err == cudaSuccess ? GNN_OK : cuda_fail(err);
}

}  // extern "C"

// ---------------------------------------------------------------------------
// Allocation-free CSR build: the radix-sort scratch lives in one file-scope
// device array instead of context workspace.  Layout (int32 words):
// keys_a | keys_b | vals_a | vals_b (GNN_CSR_NOALLOC_MAX_EDGES each) | per-tile
// digit counts and digit totals.  Host code must not use the
// array's name as a device address: every call asks cudaGetSymbolAddress for
// it, with the caller's device current.  The address is not cached, because it
// belongs to the current context's copy of the module: it changes after
// cudaDeviceReset and differs under another context on the same device.
static_assert(4ull * GNN_CSR_NOALLOC_MAX_EDGES +
                      ((GNN_CSR_NOALLOC_MAX_EDGES + kRadixTile - 1) / kRadixTile + 1) * (unsigned long long)kRadixMaxBins <=
                  GNN_CSR_NOALLOC_SCRATCH_BYTES / 4,
              "count area too small");
static __device__ __align__(256) unsigned char g_csr_noalloc_scratch[GNN_CSR_NOALLOC_SCRATCH_BYTES];

extern "C" int gnn_csr_build_noalloc(const int32_t* edge_index, int64_t n_nodes, int64_t n_edges,
                                     int32_t* rowptr, int32_t* perm, int32_t* src_sorted, gnn_stream_t stream) {
  if (!count_ok(n_nodes) || n_edges < 0 || n_edges > GNN_CSR_NOALLOC_MAX_EDGES || !rowptr)
    return GNN_ERR_INVALID_ARG;
  if (n_edges > 0 && (!edge_index || !perm || !src_sorted)) return GNN_ERR_INVALID_ARG;
  void* sp = nullptr;                             // device address of the scratch array (current context)
  cudaError_t ce = cudaGetSymbolAddress(&sp, g_csr_noalloc_scratch);
  if (ce != cudaSuccess) return cuda_fail(ce);
  unsigned char* scratch = static_cast<unsigned char*>(sp);
  cudaStream_t st = (cudaStream_t)stream;
  const int N = (int)n_nodes, E = (int)n_edges;
  const int tb = 256;
  if (E == 0) {                                   // every row pointer is 0
    csr_rowptr_kernel<<<blocks_for((int64_t)N + 1, tb), tb, 0, st>>>(nullptr, 0, N, rowptr);
    ce = cudaGetLastError();
    return ce == cudaSuccess ? GNN_OK : cuda_fail(ce);
  }
  int* words = reinterpret_cast<int*>(scratch);
  int* const keys[2] = {words, words + GNN_CSR_NOALLOC_MAX_EDGES};
  int* const vals[2] = {words + 2 * GNN_CSR_NOALLOC_MAX_EDGES, words + 3 * GNN_CSR_NOALLOC_MAX_EDGES};
  int* hist = words + 4 * GNN_CSR_NOALLOC_MAX_EDGES;
  ce = launch_csr(edge_index, N, E, keys, vals, hist, perm, src_sorted, nullptr, rowptr, nullptr, nullptr, st);
  if (ce != cudaSuccess) return cuda_fail(ce);
  ce = cudaGetLastError();
  return ce == cudaSuccess ? GNN_OK : cuda_fail(ce);
}
