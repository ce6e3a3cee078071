"""The pair search's kernels (csrc/frnn.cuh), run on the CPU from their own source: no data race in a
warp's shared memory, and the edge list of the oracle for chains of several chunks, used-up pools, and
pairs at the radius for every set of operands and row level."""
import ctypes
import re

import numpy as np
import pytest

from oracle import gnn_oracle as O
from tests import host_cuda
from tests.test_gpu_pair_filter import near_the_radius, pairs_at_the_radius

MAIN = r"""
#include "ptx.cuh"
#include "frnn.cuh"
using namespace gnn;
template <int CH, int K>
static void build(const float* emb, const float* x, int n, int dim, float radius, int pool, int cap, int32_t* out,
                  int* n_edges, uint32_t* err, bool single) {
  const int grid = frnn_grid(radius, K);
  int n_cells = 1;
  for (int k = 0; k < K; ++k) n_cells *= grid;
  std::vector<int> cells(n), ids(n), keys(n), starts(n_cells + 1), counts(n), chains((size_t)(n + pool) * kFrnnChunk, -99);
  std::vector<float4> emb_s((size_t)n * CH);
  std::vector<float> r_s(n);
  std::vector<uint4> frag((size_t)(n + 7) / 8 * 32 * ((CH + 1) / 2));
  int next = -1;
  const int nb = (n + 255) / 256;
  host::launch(nb, 256, [&] { frnn_cell_kernel<K>(emb, n, dim, grid, cells.data(), &next); });
  for (int i = 0; i < n; ++i) ids[i] = i;
  std::stable_sort(ids.begin(), ids.end(), [&](int a, int b) { return cells[a] < cells[b]; });
  for (int i = 0; i < n; ++i) keys[i] = cells[ids[i]];
  const int fb = ((n + 7) / 8 * 32 + 255) / 256;
  host::launch(fb, 256, [&] {
    frnn_layout_kernel<CH>(emb, x, 1, n, dim, ids.data(), keys.data(), n_cells, fb, (float2*)emb_s.data(), r_s.data(),
                           frag.data(), starts.data());
  });
  for (int j = 0; j <= n_cells; ++j) starts[j] = std::lower_bound(keys.begin(), keys.end(), j) - keys.begin();
  auto pairs = [&](int write) {
    host::launch((n + kFrnnBlockQueries - 1) / kFrnnBlockQueries, kFrnnPairsThreads, [&] {
      frnn_pairs_kernel<CH, K>(emb_s.data(), frag.data(), r_s.data(), n, radius * radius, grid, keys.data(), ids.data(),
                               starts.data(), write, counts.data(), n_edges, cap, out, chains.data(), &next, pool, err);
    });
  };
  if (K == 3 && single)
    host::launch((n + kFrnnSingleThreads - 1) / kFrnnSingleThreads, kFrnnSingleThreads, [&] {
      frnn_single_kernel(emb_s.data(), n, radius * radius, grid, keys.data(), starts.data(), counts.data(), chains.data(),
                         &next, pool);
    });
  else
    pairs(0);
  int sum = 0;
  for (int& c : counts) { const int k = c; c = sum; sum += k; }
  *n_edges = sum;
  pairs(1);
  host::launch((4 * n + 255) / 256, 256, [&] {
    frnn_copy_kernel(r_s.data(), n, ids.data(), counts.data(), n_edges, cap, chains.data(), out);
  });
}
extern "C" int build_graph(const float* emb, const float* x, int n, int dim, float radius, int pool, int cap,
                           int32_t* out, int* n_edges, int single) {
  uint32_t err = 0;
  host::races = host::mmas = host::matches = host::tests = 0;
  if (dim < 4) build<1, 3>(emb, x, n, dim, radius, pool, cap, out, n_edges, &err, single);
  else if (dim <= 8) build<2, 4>(emb, x, n, dim, radius, pool, cap, out, n_edges, &err, single);
  else if (dim <= 12) build<3, 4>(emb, x, n, dim, radius, pool, cap, out, n_edges, &err, single);
  else build<4, 4>(emb, x, n, dim, radius, pool, cap, out, n_edges, &err, single);
  return err ? -1 : host::races;
}
extern "C" int mmas() { return host::mmas; }
extern "C" int matches() { return host::matches; }
extern "C" int tests() { return host::tests; }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    text = host_cuda.source("frnn.cuh")
    shared = host_cuda.between(text, "  struct Warp {", "  };")
    checked = re.sub(r"\b(int|unsigned char) (?=\w+\[)", r"host::Cell<\1> ", shared)
    assert checked.count("host::Cell") == 5
    text = host_cuda.replace(text.replace(shared, checked), "      hit = s < r2;", "      hit = s < r2; ++host::tests;")
    return host_cuda.compile_host(tmp_path_factory.mktemp("host"), MAIN, [("frnn.cuh", text)])


def build(lib, emb, r, radius, pool=None, single=False):
    n, dim = emb.shape
    pool = n if pool is None else pool
    cap = n * n
    out = np.full(2 * cap, -1, np.int32)
    m = ctypes.c_int(0)
    p = lambda a: a.ctypes.data_as(ctypes.c_void_p)  # noqa: E731
    races = lib.build_graph(p(emb), p(r), n, dim, ctypes.c_float(radius), pool, cap, p(out), ctypes.byref(m), int(single))
    return out[:2 * m.value].reshape(2, -1), races


def ordered(ei):
    e = ei.T.astype(np.int64)
    return e[np.lexsort((e[:, 1], e[:, 0]))]


@pytest.mark.parametrize("pool", [None, 0, 7])
def test_chains_of_several_chunks(lib, pool):
    """Clumps of up to 60 hits within the radius of each other: a batch of 32 pairs holds several partners of
    one query, whose chain begins new chunks in the middle of it."""
    rng = np.random.default_rng(3)
    centres = rng.standard_normal((4, 8))
    emb = np.repeat(centres / np.linalg.norm(centres, axis=1, keepdims=True), [60, 33, 16, 1], axis=0)
    emb = (emb + 0.001 * rng.standard_normal(emb.shape)).astype(np.float32)[rng.permutation(110)]
    r = rng.random(110).astype(np.float32)
    ei, races = build(lib, emb, r, 0.1, pool)
    np.testing.assert_array_equal(ordered(ei), O.radius_graph(emb, r, 0.1))
    np.testing.assert_array_equal(ei, build(lib, emb, r, 0.1)[0])     # the pool changes nothing
    assert races == 0, f"{races} unordered accesses to shared memory"


@pytest.mark.parametrize("dim", [4, 12])
def test_sparse_hits_share_runs(lib, dim):
    """Parallel lines of hits, one every other cell of a row: a row's own 63 runs would take a batch of four blocks
    for a few candidates each; a coarser level takes half of the blocks."""
    rng = np.random.default_rng(0)
    line = np.stack(np.meshgrid(*[np.arange(5)] * 3, indexing="ij"), -1).reshape(-1, 3) * (2 / 64) + 0.01
    emb = np.zeros((line.shape[0], 20, dim))
    emb[:, :, :3] = line[:, None]
    emb[:, :, 3] = (np.arange(20) * 2 - 20) * (2 / 64) + 0.01
    emb = (emb.reshape(-1, dim) + 1e-4 * rng.random((2500, 1))).astype(np.float32)
    r = rng.random(2500).astype(np.float32)
    ei, _ = build(lib, emb, r, 0.02)
    np.testing.assert_array_equal(ordered(ei), O.radius_graph(emb, r, 0.02))
    warps, mma = (2500 + 15) // 16, 2 if dim <= 8 else 4
    blocks = lib.mmas() / warps / mma                # of eight candidates, per sixteen hits
    assert blocks <= 120, f"{blocks:.0f} blocks (one row of cells at a time: 178)"


def test_pairs_below_the_filters_resolution(lib):
    """Hits 0.002 apart, searched at half of that: the filter lets all of them through (it is right to about 0.01 on
    unit vectors), the exact test none, and no lists are gone through for them."""
    emb = np.zeros((200, 8), np.float32)
    emb[:, 0] = 0.6
    emb[:, 4] = 0.4 + 0.002 * (np.arange(200) % 20)
    emb[:, 5] = 0.4 + 0.002 * (np.arange(200) // 20)
    ei, races = build(lib, emb, np.zeros(200, np.float32), 0.001)
    assert ei.shape[1] == 0 and races == 0
    assert lib.matches() == 0


def test_infinite_and_nan_hits_are_no_candidates(lib):
    """A hit with an infinite or NaN coordinate is within no radius of any: no exact test for it.  Long hits
    whose squares overflow are still tested."""
    rng = np.random.default_rng(1)
    emb = rng.standard_normal((120, 8)).astype(np.float32)
    emb[::3, 2] = np.nan
    emb[1::6, 7] = np.inf
    emb[2::12] = np.float32(1e20)
    emb[5] = -np.inf
    r = rng.random(120).astype(np.float32)
    ei, _ = build(lib, emb, r, 3.0)
    with np.errstate(invalid="ignore", over="ignore"):
        np.testing.assert_array_equal(ordered(ei), O.radius_graph(emb, r, 3.0))
    ei, _ = build(lib, np.full((200, 8), np.nan, np.float32), np.zeros(200, np.float32), 0.2)
    assert ei.shape[1] == 0 and lib.tests() == 0


@pytest.mark.parametrize("dim", [1, 2, 3])
def test_single_hits_and_filter_agree(lib, dim):
    """The counting pass by single hits gives the lists of the filter's, with room for the chains and without."""
    rng = np.random.default_rng(dim)
    emb = rng.uniform(-1, 1, (300, dim)).astype(np.float32)
    emb[:120] = emb[0] + 0.02 * rng.standard_normal((120, dim)).astype(np.float32)     # runs and chains of several parts
    r = rng.random(300).astype(np.float32)
    want, _ = build(lib, emb, r, 0.05)
    np.testing.assert_array_equal(ordered(want), O.radius_graph(emb, r, 0.05))
    for pool in (None, 0, 40):
        np.testing.assert_array_equal(build(lib, emb, r, 0.05, pool, single=True)[0], want)


@pytest.mark.parametrize("dim", [3, 8, 12, 16])
@pytest.mark.parametrize("scale", [1e-3, 1.0, 37.0])
def test_pairs_at_the_radius(lib, dim, scale):
    """Pairs whose distance is the radius to a millionth, with every error of the tensor core against them."""
    emb, radius = pairs_at_the_radius(dim, scale, 30, 9)
    r = np.random.default_rng(0).random(len(emb)).astype(np.float32)
    want = O.radius_graph(emb, r, radius)
    inside, outside = near_the_radius(emb, radius)
    assert inside > 60 and outside > 60
    np.testing.assert_array_equal(ordered(build(lib, emb, r, float(radius))[0]), want)
