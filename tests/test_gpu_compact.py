"""The filter's compaction where its split changes: edge counts around a warp, a tile of 1,024 edges and
the 2,048 tiles above which a block takes two, at thresholds that keep all, half and none of the edges;
the kept list bit-exact against applyFiltering of the same scores."""
import numpy as np
import pytest

from oracle import gnn_oracle as O
from paper_2402_09633_gb300 import synthetic as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("e", [1, 31, 33, 255, 257, 1023, 1024, 1025, 5000, 2048 * 1024, 2048 * 1024 + 1, 2100003])
def test_compact_sizes(e):
    import torch
    from paper_2402_09633_gb300 import InteractionNetwork
    cfg = S.ModelConfig(3, 2, 64, 1, 2)
    net = InteractionNetwork(cfg, S.pack_blob(cfg, S.init_weights(cfg, 0)))
    net.load_filter(S.pack_filter_blob(cfg, S.init_filter_weights(cfg, 1)))
    rng = np.random.default_rng(e)
    x = rng.standard_normal((500, 3)).astype(np.float32)
    ei = rng.integers(0, 500, size=(2, e)).astype(np.int32)
    dx, dei = torch.from_numpy(x).cuda(), torch.from_numpy(ei).cuda()
    median = float(net.filter_edges(dx, dei, 2.0)[0].median())
    for thr in (-1.0, median, 2.0):
        sc, kept, ids = (t.cpu().numpy() for t in net.filter_edges(dx, dei, thr))
        want_kept, want_ids = O.apply_filtering(sc, ei, thr)
        np.testing.assert_array_equal(ids, want_ids)
        np.testing.assert_array_equal(kept, want_kept)
    assert net.status() == 0
    net.close()
