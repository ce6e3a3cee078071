"""The exclusive scan of graph building's counts (csrc/compact.cuh), run on the CPU from its own source: the
offsets and the total where a block takes one run of 1,024 entries and where it takes several, totals past
32 bits, and a number of block sums to add up that does not outgrow the entries."""
import ctypes

import numpy as np
import pytest

from tests import host_cuda

MAIN = r"""
#include "ptx.cuh"
#include "compact.cuh"
using namespace gnn;
extern "C" long long blocks(long long n) { return compact_blocks(n); }
extern "C" long long tiles(long long n) { return compact_tiles(n); }
extern "C" int scan(int* v, int n, int per, int blocks) {
  std::vector<int> sums(blocks);
  int total = -1;
  host::launch(blocks, kScanBlock, [&] { scan_reduce_kernel(v, n, per, sums.data()); });
  host::launch(blocks, kScanBlock, [&] { scan_apply_kernel(v, n, per, sums.data(), &total); });
  return total;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    lib = host_cuda.compile_host(tmp_path_factory.mktemp("host"), MAIN, [("compact.cuh", host_cuda.source("compact.cuh"))])
    for f in (lib.blocks, lib.tiles):
        f.argtypes, f.restype = [ctypes.c_longlong], ctypes.c_longlong
    return lib


@pytest.mark.parametrize("n", [1, 1024, 2048 * 1024, 2048 * 1024 + 1, 10 ** 8, 2147475455])
def test_block_sums_stay_few(lib, n):
    """Every block adds up the block sums: no more of those additions than entries, once they are many."""
    b = lib.blocks(n)
    assert b * lib.tiles(n) * 1024 >= n and (b - 1) * lib.tiles(n) * 1024 < n
    assert b * b <= max(n, 2048 ** 2)


@pytest.mark.parametrize("n,per", [(1, 1), (1023, 1), (1025, 1), (5000, 1), (1, 2), (2048, 2), (2049, 2), (5000, 3), (9000, 4)])
def test_offsets(lib, n, per):
    v = np.random.default_rng(n).integers(0, 50, n).astype(np.int32)
    got = v.copy()
    total = lib.scan(got.ctypes.data_as(ctypes.c_void_p), n, per, (n + 1024 * per - 1) // (1024 * per))
    assert total == v.sum()
    np.testing.assert_array_equal(got, np.cumsum(v) - v)


@pytest.mark.parametrize("per", [1, 2])
def test_total_saturates(lib, per):
    v = np.full(3000, 2 ** 20, np.int32)
    assert lib.scan(v.ctypes.data_as(ctypes.c_void_p), 3000, per, 3 if per == 1 else 2) == 2 ** 31 - 1
