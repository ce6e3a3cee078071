"""The MMA-issuing warp of the tile kernels (csrc/mlp_tiles.cuh), run on the CPU from its own source against
a model of what it talks to: mbarriers, copies and commits that arrive late and in any order, and worker
groups that publish their next operand when a job's result is there.  For every shape of its schedule
(kernel kind, hidden width, precision, layers, tiles per block): the jobs all run, no job writes a
tensor-memory region that another still uses, and when the warp leaves nothing is on its way to the
block's shared memory."""
import ctypes

import pytest

from tests import host_cuda

MAIN = r"""
#include <climits>
#include <cstdint>
#include <cstdio>
#include <map>
#include <random>
#include <type_traits>
#include <vector>
#define __device__
#define __host__
#define __forceinline__ inline
#define GNN_TRACE_AT(a, b)
namespace gnn {
constexpr uint32_t idesc_bf16_f32(uint32_t, uint32_t) { return 0; }
constexpr uint64_t kWaitLimitNs = 2000000000ull;
enum : uint32_t { DEV_ERR_TIMEOUT = 2u };
@TYPES@

struct Bar { int need = 1, arrived = 0, phases = 0; long tx = 0; };
struct Late { uint64_t* bar; long bytes; int job; };      // a copy (bytes > 0) or a commit after `job`
static std::map<uint64_t*, Bar> bars_;
static std::vector<Late> late;
static std::mt19937 rng;
static uint64_t now;
static int issued, complete, faults;                      // jobs issued; MMAs complete up to job
static std::map<int, std::pair<int, int>> regions;        // job -> regions of A and D
static void settle(Bar& b) { if (b.arrived == b.need && b.tx == 0) { b.arrived = 0; ++b.phases; } }
static void arrive(uint64_t* bar, long tx = 0) {
  Bar& b = bars_[bar];
  b.tx += tx;
  if (++b.arrived > b.need) ++faults;
  settle(b);
}
static bool land(uint64_t* bar) {                         // one thing on its way to bar arrives
  std::vector<int> on;
  for (int i = 0; i < (int)late.size(); ++i) if (late[i].bar == bar) on.push_back(i);
  if (on.empty()) return false;
  const int i = on[rng() % on.size()];
  const Late l = late[i];
  late.erase(late.begin() + i);
  if (l.bytes) { Bar& b = bars_[bar]; b.tx -= l.bytes; settle(b); }
  else { if (l.job > complete) complete = l.job; arrive(bar); }
  return true;
}
static bool passed(uint64_t* bar, uint32_t parity) { return (uint32_t)(bars_[bar].phases & 1) != parity; }

// the worker groups
static uint64_t *a_full_, *d_full_;
static int groups, jobs, my_tiles, seen[3], sent[3];      // results seen, operands published, per group
static int total_of(int g) { return (my_tiles - g + groups - 1) / groups * jobs; }
static void publish(int g) { for (int w = 0; w < 8; ++w) arrive(&a_full_[g]); ++sent[g]; }
static void work() {
  for (int g = 0; g < groups; ++g) {
    if (rng() & 1) land(&d_full_[g]);
    if (bars_[&d_full_[g]].phases > seen[g]) {
      ++seen[g];
      if (sent[g] < total_of(g)) publish(g);
    }
  }
}

static bool warp_all(bool x) { return x; }
static bool elect_one() { return true; }
static void __syncwarp() {}
static uint64_t global_timer_ns() { return now += 100000; }
static void atomicOr(uint32_t* p, uint32_t v) { *p |= v; }
static bool mbar_test_wait(uint64_t* bar, uint32_t parity) { work(); if (rng() & 1) land(bar); return passed(bar, parity); }
static bool bounded_wait(uint64_t* bar, uint32_t parity, volatile int*, uint32_t* err) {
  while (!passed(bar, parity)) { work(); if (!land(bar)) { *err |= DEV_ERR_TIMEOUT; return false; } }
  return true;
}
static void drain_wait(uint64_t* bar, uint32_t parity) { while (!passed(bar, parity) && land(bar)) {} }
static void mbar_arrive(uint64_t* bar) { arrive(bar); }
static void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) { arrive(bar, bytes); }
static void bulk_g2s(void*, const void*, uint32_t bytes, uint64_t* bar) { late.push_back({bar, (long)bytes, 0}); }
static void mma_commit(uint64_t* bar) { late.push_back({bar, 0, issued}); }
static void tc_fence_after() {}
static uint32_t smem_u32(const void*) { return 0; }
static uint64_t sdesc_kmajor_sw128(uint32_t) { return 0; }
static uint64_t sdesc_kmajor_plain(uint32_t) { return 0; }
static void mma_bf16_ss(uint32_t, uint64_t, uint64_t, uint32_t, uint32_t) {}
static int width;
static void mma_bf16_ts(uint32_t d, uint32_t a, uint64_t, uint32_t, uint32_t) { regions[issued + 1] = {(int)a / width, (int)d / width}; }

template <TileKind KIND, int H, bool BF>
int issuer(TileParams p, unsigned seed) {
  using G = TileGeom<H, BF>;
  constexpr int NG = TileRoles<KIND>::NG, STAGES = tile_max_stages<KIND, H, BF>(), NSPARE = G::NREG - NG;
  static uint64_t words[15 + 2 * 8];
  uint64_t *a_full = words, *d_full = words + 3, *spare_free = words + 6, *c_full = words + 14, *w_full = words + 15,
           *w_empty = words + 15 + STAGES;
  volatile int abort_word = 0, d_region[3] = {0, 0, 0};
  volatile int* abort_flag = &abort_word;
  static uint8_t ring[1], consts[1];
  const uint32_t tmem_base = 0;
  const int lane = 0, n_my = p.n_tiles, n_rounds = (n_my + NG - 1) / NG;
  const bool resident = p.n_jobs <= STAGES;
  bars_.clear(); late.clear(); regions.clear();
  rng.seed(seed);
  issued = complete = faults = 0;
  groups = NG; jobs = p.n_jobs; my_tiles = n_my; width = H; a_full_ = a_full; d_full_ = d_full;
  for (int g = 0; g < NG; ++g) { bars_[&a_full[g]].need = 8; bars_[&d_full[g]].need = NG == 3 ? 2 : 1; seen[g] = sent[g] = 0; }
  for (int s = 0; s < STAGES; ++s) bars_[&w_empty[s]].need = NG;
  mbar_arrive_expect_tx(c_full, 16);
  bulk_g2s(consts, nullptr, 16, c_full);
  if (resident) {
    mbar_arrive_expect_tx(w_full, (uint32_t)p.n_jobs);
    for (int j = 0; j < p.n_jobs; ++j) bulk_g2s(ring, nullptr, 1, w_full);
  }
  for (int g = 0; g < NG && g < n_my; ++g) publish(g);
@ISSUER@
  int want = 0;
  for (int g = 0; g < NG && g < n_my; ++g) want += total_of(g);
  if (*p.err || abort_word || issued != want) return -1;
  return faults ? -2 : (int)late.size();
}

template <TileKind K>
static int run(int H, int bf, const TileParams& p, unsigned seed) {
  if (H == 128) return bf ? issuer<K, 128, true>(p, seed) : issuer<K, 128, false>(p, seed);
  return bf ? issuer<K, 64, true>(p, seed) : issuer<K, 64, false>(p, seed);
}
}  // namespace gnn
using namespace gnn;
// Returns what is still on its way when the warp has left (-1: not all jobs ran, -2: a region or barrier misused).
extern "C" int leave(int kind, int H, int bf, int L, int tiles, unsigned seed) {
  uint32_t err = 0;
  TileParams p{};
  const bool node = kind == 0 || kind == 3;
  p.n_tiles = tiles;
  p.n_jobs = kind == 0 ? L + 2 : kind == 3 ? L + 3 : L;
  p.n_in = 2;
  p.err = &err;
  if (kind == 3) p.job_acc[1] = 1;
  for (int j = 0, a = 0; j < kMaxJobs; ++j) {             // as the launch sets them
    if (j > 0 && !(p.job_acc[j] || (node && j == p.n_jobs - 1))) a ^= 1;
    p.job_areg[j] = a;
  }
  switch (kind) {
    case 0: return run<TileKind::NodeEncoder>(H, bf, p, seed);
    case 1: return run<TileKind::EdgeEncoder>(H, bf, p, seed);
    case 2: return run<TileKind::EdgeUpdate>(H, bf, p, seed);
    case 3: return run<TileKind::NodeUpdate>(H, bf, p, seed);
    case 4: return run<TileKind::Classifier>(H, bf, p, seed);
    case 5: return run<TileKind::Filter>(H, bf, p, seed);
    default: return run<TileKind::Embed>(H, bf, p, seed);
  }
}
"""
# where the schedule has issued a job: its D region is nobody's A or D, and no MMA in flight reads it
JOB = r"""
          ++issued;
          {
            const std::pair<int, int> now_ = regions[issued];
            for (int o = complete + 1; o < issued; ++o)
              if (regions[o].first == now_.second) ++faults;
            if constexpr (NG == 3)
              for (int o = 0; o < NG; ++o) if (o != g && (int)reg_g[o] == now_.second) ++faults;
          }
          mma_commit(&d_full[g]);"""


@pytest.fixture(scope="module")
def leave(tmp_path_factory):
    text = host_cuda.source("mlp_tiles.cuh")
    types = host_cuda.between(text, "enum class TileKind", "__device__ __forceinline__ float2 f2(")
    warp = host_cuda.between(text, "    // The groups advance independently", "  } else {\n    // Worker groups")
    warp = host_cuda.replace(warp, "          mma_commit(&d_full[g]);", JOB)
    warp = warp.replace("#pragma unroll", "")
    lib = host_cuda.compile_host(tmp_path_factory.mktemp("host"), MAIN.replace("@TYPES@", types).replace("@ISSUER@", warp))
    return lib.leave


@pytest.mark.parametrize("bf", [0, 1])
@pytest.mark.parametrize("H", [64, 128])
@pytest.mark.parametrize("kind", range(7))
def test_nothing_is_in_flight_when_the_issuer_leaves(leave, kind, H, bf):
    for L in (2, 3, 4):
        for tiles in (1, 2, 3, 4, 5, 7, 12, 25):
            for seed in range(4):
                left = leave(kind, H, bf, L, tiles, ctypes.c_uint(seed))
                assert left >= 0, f"L {L}, {tiles} tiles, seed {seed}: code {left}"
                assert left == 0, f"L {L}, {tiles} tiles, seed {seed}: {left} arrivals on their way"
