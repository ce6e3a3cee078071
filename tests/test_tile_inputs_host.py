"""The tile kernels' loads of endpoints and inputs ahead of their tile (csrc/mlp_tiles.cuh), run on the CPU
from their own source with overflow checks: at the largest count that a call accepts, tiles up to two
rounds past the last are asked for, and give no row."""
import subprocess
import sys

import pytest

from tests import host_cuda

MAIN = r"""
#include <climits>
#include <cstddef>
#include <cstdint>
#include <type_traits>
struct float2 { float x, y; };
static float2 make_float2(float x, float y) { return {x, y}; }
static constexpr int kTileRows = 128;
enum class TileKind { NodeEncoder, EdgeEncoder, EdgeUpdate, NodeUpdate, Classifier, Filter, Embed };
struct Params { int n_rows, n_tiles, n_nodes, n_feat, n_in, x_stride; const float* x; const int *src_sorted, *dst_sorted; const int32_t* ei_in; };

template <TileKind KIND>
static int past_the_end(int rows, int ahead) {
  static const float x[16] = {0};
  Params p{};                                             // null index arrays: no row may be read
  p.n_rows = rows;
  p.n_tiles = (int)(((long long)rows + kTileRows - 1) / kTileRows);
  p.n_nodes = 1;
  p.n_feat = p.x_stride = 2;
  p.n_in = 2;
  p.x = x;
  const int lane = 31, trow = 119;
  float2 x_in[8];
  int ends[2][2], valid_next = 0;
@LOADS@
  load_ends(p.n_tiles - 1 + ahead);
  load_inputs(p.n_tiles - 1 + ahead);
  return valid_next;
}
extern "C" int run(int rows, int ahead) {
  return past_the_end<TileKind::Filter>(rows, ahead) + past_the_end<TileKind::EdgeEncoder>(rows, ahead) +
         past_the_end<TileKind::NodeEncoder>(rows, ahead);
}
"""
MAX_COUNT = 2147475455                               # GNN_MAX_COUNT


@pytest.mark.parametrize("rows", [1, 128, MAX_COUNT - 117000, MAX_COUNT])
def test_rows_past_the_end(tmp_path, rows):
    text = host_cuda.source("mlp_tiles.cuh")
    loads = host_cuda.between(text, "    auto tile_row = ", "    // Inputs -> A operand of the first job")
    host_cuda.compile_host(tmp_path, MAIN.replace("@LOADS@", loads.replace("#pragma unroll", "")),
                           flags=["-fsanitize=signed-integer-overflow", "-fsanitize-undefined-trap-on-error"])
    for ahead in (1, 3 * 152, 6 * 152):                   # a block's next tile, and the one after it
        call = f"import ctypes; assert ctypes.CDLL({str(tmp_path / 'host.so')!r}).run({rows}, {ahead}) == 0"
        assert subprocess.run([sys.executable, "-c", call]).returncode == 0, f"{rows} rows, {ahead} tiles ahead"
