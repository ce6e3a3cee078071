"""The pair search of graph building where its tensor-core filter can go wrong (through the C ABI).

CPU: the filter value, evaluated with the kernel's bf16 splits, never excludes a pair within the radius
(unit vectors, and vectors of any scale).  GPU: edge sets bit-exact against the oracle for hit counts
around a warp's sixteen queries and a block of eight candidates, every embedding width, coincident hits,
hits outside the unit sphere, and infinities and NaN (which are never within a radius)."""
import numpy as np
import pytest

from oracle import gnn_oracle as O
from paper_2402_09633_gb300 import synthetic as S


def _bf16(a):
    return O.round_bf16(np.asarray(a, np.float32).astype(np.float64)).astype(np.float32)


def _parts(v):
    out = []
    for _ in range(3):
        q = _bf16(v)
        out.append(q)
        v = (v - q).astype(np.float32)
    return out


@pytest.mark.parametrize("dim,scale", [(8, 1.0), (16, 1.0), (3, 1.0), (8, 1e-3), (8, 37.0)])
def test_filter_excludes_no_pair(dim, scale):
    rng = np.random.default_rng(dim)
    n = 20000
    a = rng.standard_normal((n, dim))
    a /= np.linalg.norm(a, axis=1, keepdims=True)
    a = (a * scale).astype(np.float32)
    radius = np.float32(0.08 * scale)
    step = rng.standard_normal((n, dim))
    step /= np.linalg.norm(step, axis=1, keepdims=True)
    # distances from zero to a little beyond the radius, half of them within 1e-6 of it
    d = np.where(rng.random(n) < 0.5, rng.random(n) * 1.01, 1.0 + 1e-6 * rng.standard_normal(n))
    b = (a + step * (d * radius)[:, None]).astype(np.float32)
    r2 = np.float32(radius * radius)
    within = O.sq_dist_f32(a, b) < r2
    assert 0 < within.sum() < n
    c = np.float32(1.0 / 16384.0)
    ah, bh = _bf16(-2 * a), _bf16(b)
    al, bl = _bf16(-2 * a - ah), _bf16(b - bh)
    na = ((a * a).sum(1) * (1 - c) - (r2 * np.float32(1 + 1 / 4096) + np.float32(1e-35))).astype(np.float32)
    nb = ((b * b).sum(1) * (1 - c)).astype(np.float32)
    f = (ah.astype(np.float64) * bh + ah.astype(np.float64) * bl + al.astype(np.float64) * bh).sum(1)
    f += sum(p.astype(np.float64) for p in _parts(na)) + sum(p.astype(np.float64) for p in _parts(nb))
    # the accumulation inside the tensor core: 33 terms, each off by at most 2^-22 of the largest
    slip = 33 * 2.0 ** -22 * 2 * np.maximum((a * a).sum(1), (b * b).sum(1))
    assert np.all(f[within] + slip[within] < 0)


def _edges(emb, r_col, radius, room):
    import torch
    from paper_2402_09633_gb300 import InteractionNetwork
    cfg = S.ModelConfig(3, 2, 64, 0, 2)
    net = InteractionNetwork(cfg, S.pack_blob(cfg, S.init_weights(cfg, 0)))
    x = np.zeros((emb.shape[0], 3), np.float32)
    x[:, 0] = r_col
    ei, n = net.build_graph(torch.from_numpy(emb).cuda(), torch.from_numpy(x).cuda(), float(radius), room)
    out = ei.cpu().numpy().T.astype(np.int64)
    net.close()
    return out[np.lexsort((out[:, 1], out[:, 0]))] if n else out.reshape(0, 2)


def _unit(rng, n, dim):
    e = rng.standard_normal((n, dim))
    return (e / np.linalg.norm(e, axis=1, keepdims=True)).astype(np.float32)


def pairs_at_the_radius(dim, scale, anchors, partners):
    """Hits of length about `scale`, `partners` of them at a distance within 1e-6 of the radius from each anchor, on
    either side; the radius."""
    rng = np.random.default_rng(dim)
    a = rng.standard_normal((anchors, dim))
    a /= np.linalg.norm(a, axis=1, keepdims=True)
    a = (a * scale).astype(np.float32)
    radius = np.float32(0.08 * scale)
    step = rng.standard_normal((anchors, partners, dim))
    step /= np.linalg.norm(step, axis=2, keepdims=True)
    b = a[:, None] + step * (radius * (1 + 1e-6 * rng.standard_normal((anchors, partners, 1))))
    emb = np.concatenate([a, b.reshape(-1, dim).astype(np.float32)])
    return np.ascontiguousarray(emb[rng.permutation(len(emb))]), radius


def near_the_radius(emb, radius):
    """How many pairs within the radius, and how many outside it, lie within 3e-6 of it."""
    i, j = np.triu_indices(len(emb), 1)
    d = np.sqrt(O.sq_dist_f32(emb[i], emb[j]).astype(np.float64))
    near = np.abs(d / radius - 1) < 3e-6
    inside = near & (O.sq_dist_f32(emb[i], emb[j]) < np.float32(radius * radius))
    return inside.sum(), near.sum() - inside.sum()


@pytest.mark.gpu
@pytest.mark.parametrize("dim", [3, 8, 16])
@pytest.mark.parametrize("scale", [1e-3, 1.0, 37.0])
def test_pairs_at_the_radius(dim, scale):
    """The filter's margin on the GPU: thousands of pairs whose distance is the radius to a millionth."""
    emb, radius = pairs_at_the_radius(dim, scale, 300, 12)
    r = np.random.default_rng(0).random(len(emb)).astype(np.float32)
    want = O.radius_graph(emb, r, radius)
    inside, outside = near_the_radius(emb, radius)
    assert inside > 1000 and outside > 1000
    np.testing.assert_array_equal(_edges(emb, r, radius, 20 * len(emb)), want)


@pytest.mark.gpu
@pytest.mark.parametrize("n", [1, 2, 7, 8, 9, 15, 16, 17, 63, 64, 65, 700])
@pytest.mark.parametrize("dim,radius", [(8, 0.9), (2, 0.05), (5, 0.3)])
def test_hit_counts(n, dim, radius):
    rng = np.random.default_rng(n + dim)
    emb, r = _unit(rng, n, dim), rng.random(n).astype(np.float32)
    np.testing.assert_array_equal(_edges(emb, r, radius, n * n), O.radius_graph(emb, r, radius))


@pytest.mark.gpu
@pytest.mark.parametrize("dim", range(1, 17))
def test_widths(dim):
    rng = np.random.default_rng(dim)
    emb, r = _unit(rng, 400, dim), rng.integers(0, 5, 400).astype(np.float32)
    emb[10:40] = emb[0]                              # coincident hits: one query sees a full run of them
    radius = 0.4 if dim > 2 else 0.02
    np.testing.assert_array_equal(_edges(emb, r, radius, 160000), O.radius_graph(emb, r, radius))


@pytest.mark.gpu
@pytest.mark.parametrize("dim", [3, 8, 12])
def test_values_off_the_sphere(dim):
    rng = np.random.default_rng(dim)
    emb = (rng.standard_normal((500, dim)) * 40).astype(np.float32)
    emb[:200] = emb[0] + 0.2 * rng.standard_normal((200, dim)).astype(np.float32)
    emb[200:203] = np.float32(1e20)                  # squares overflow; three coincident hits
    emb[203, 0], emb[204, 1], emb[205, 2] = np.inf, -np.inf, np.nan
    emb[206:208] = np.inf
    r = rng.random(500).astype(np.float32)
    with np.errstate(invalid="ignore", over="ignore"):
        want = O.radius_graph(emb, r, 1.0)
    assert want.shape[0] > 100
    np.testing.assert_array_equal(_edges(emb, r, 1.0, 250000), want)


@pytest.mark.gpu
@pytest.mark.parametrize("dim,radius", [(1, 2e-5), (2, 0.006), (3, 0.04)])
@pytest.mark.parametrize("n", [65535, 65536, 70001])
def test_single_hits_in_few_dimensions(n, dim, radius):
    """Both sides of the hit count from which up to three dimensions are searched by single hits; byte for byte the
    same with chunks for few and for none of the hits with more than 15 partners."""
    import ctypes
    import torch
    from paper_2402_09633_gb300 import InteractionNetwork
    kd = pytest.importorskip("scipy.spatial")
    rng = np.random.default_rng(n + dim)
    emb = rng.uniform(-1, 1, (n, dim)).astype(np.float32)
    emb[:200] = emb[0] + np.float32(radius / 5) * rng.standard_normal((200, dim)).astype(np.float32)
    emb[200] = np.nan
    x = np.zeros((n, 3), np.float32)
    x[:, 0] = rng.random(n)
    cfg = S.ModelConfig(3, 2, 64, 0, 2)
    net = InteractionNetwork(cfg, S.pack_blob(cfg, S.init_weights(cfg, 0)))
    net.lib.gnn_debug_graph_pool.argtypes = [ctypes.c_void_p, ctypes.c_int64]
    lists = []
    for pool in (-1, 0, 100):
        net.lib.gnn_debug_graph_pool(net.handle, pool)
        lists.append(net.build_graph(torch.from_numpy(emb).cuda(), torch.from_numpy(x).cuda(), radius, 20 * n)[0].cpu().numpy())
    net.close()
    assert all(a.tobytes() == lists[0].tobytes() for a in lists)
    ok = np.delete(np.arange(n), 200)
    cand = kd.cKDTree(emb[ok].astype(np.float64)).query_pairs(radius * 1.001, output_type="ndarray")
    want = O.radius_graph(emb, x[:, 0], radius, np.sort(ok[cand], 1))
    got = lists[0].T.astype(np.int64)
    np.testing.assert_array_equal(got[np.lexsort((got[:, 1], got[:, 0]))], want)


@pytest.mark.gpu
def test_more_hits_than_one_scan_tile_per_block():
    """Above 2,048 x 1,024 hits a block of the counts' scan takes two tiles: a lattice of isolated hits, 200,000
    of which have one partner."""
    rng = np.random.default_rng(1)
    n, m = 2_000_003, 200_000
    at = rng.permutation(40 ** 4)[:n]
    emb = np.stack([at // 40 ** k % 40 for k in range(4)], 1) * (1.8 / 39) - 0.9
    owner = rng.permutation(n)[:m]
    emb = np.concatenate([emb, emb[owner] + [0, 0, 0, 0.01]]).astype(np.float32)
    r = rng.random(n + m).astype(np.float32)
    pair = np.stack([owner, n + np.arange(m)], 1)
    first = (r[pair[:, 0]] < r[pair[:, 1]]) | ((r[pair[:, 0]] == r[pair[:, 1]]) & (pair[:, 0] < pair[:, 1]))
    pair = np.where(first[:, None], pair, pair[:, ::-1])
    np.testing.assert_array_equal(_edges(emb, r, 0.02, 1 << 20), pair[np.lexsort((pair[:, 1], pair[:, 0]))])
