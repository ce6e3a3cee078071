"""Serving-style use of the C ABI (the paper's throughput levers: several model instances on one
GPU, Section 3.2): a gnn_infer call captured once into a CUDA graph and replayed, and several
contexts scoring different events concurrently on their own streams."""
import numpy as np
import pytest

from paper_2402_09633_gb300 import synthetic as S
from tests.gpu_util import check_parity

pytestmark = pytest.mark.gpu


def _event(seed, n=3000, e=10007):
    return S.generate_event(S.EventSpec(n, 9, "powerlaw", 0.02, n_edges=e), seed)


def test_cuda_graph_capture_and_replay():
    """After gnn_reserve, gnn_infer only enqueues kernels: it can be captured into a CUDA graph,
    and replaying the graph on new inputs (same sizes) gives the eager result bit for bit."""
    import torch
    from paper_2402_09633_gb300 import InteractionNetwork
    cfg = S.ModelConfig(12, 2, 128, 3, 3)
    W = S.init_weights(cfg, 5)
    net = InteractionNetwork(cfg, S.pack_blob(cfg, W))
    x0, e0 = _event(0)
    x1, e1 = _event(1)
    assert x0.shape == x1.shape and e0.shape == e1.shape
    net.reserve(x0.shape[0], e0.shape[1])
    xs = torch.from_numpy(x0).cuda()
    es = torch.from_numpy(e0).cuda()
    out = torch.empty(e0.shape[1], dtype=torch.float32, device="cuda")
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        net.infer(xs, es, out, stream=stream)                 # warm-up outside capture
    stream.synchronize()
    eager0 = out.cpu().numpy().copy()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream):
        net.infer(xs, es, out, stream=stream)
    for x, e, want in ((x1, e1, None), (x0, e0, eager0)):
        xs.copy_(torch.from_numpy(x)); es.copy_(torch.from_numpy(e))
        g.replay()
        torch.cuda.synchronize()
        got = out.cpu().numpy()
        if want is not None:
            assert got.tobytes() == want.tobytes()
        else:
            eager = net.infer(torch.from_numpy(x).cuda(), torch.from_numpy(e).cuda()).cpu().numpy()
            assert got.tobytes() == eager.tobytes()
            check_parity(got, W, x, e, cfg.n_iters)
    assert net.status() == 0
    net.close()


def test_capture_of_the_steps_around_the_network():
    """The embedding, graph building, filter and track labels only enqueue kernels once their scratch is there: each
    captured into a CUDA graph gives the eager outputs on new inputs of the same sizes, byte for byte."""
    import ctypes
    import torch
    from paper_2402_09633_gb300 import InteractionNetwork
    cfg = S.ModelConfig(12, 2, 64, 1, 2)
    net = InteractionNetwork(cfg, S.pack_blob(cfg, S.init_weights(cfg, 5)))
    net.load_embedding(S.pack_embed_blob(cfg, S.init_embed_weights(cfg, 8, 2)))
    net.load_filter(S.pack_filter_blob(cfg, S.init_filter_weights(cfg, 3)))
    n, m, room = 3000, 10007, 60000
    xs, es = torch.zeros(n, 12, device="cuda"), torch.zeros(2, m, dtype=torch.int32, device="cuda")
    emb = torch.zeros(n, 8, device="cuda")
    score = torch.zeros(m, device="cuda")

    def ints(*size):
        return torch.zeros(*size, dtype=torch.int32, device="cuda")
    edges, n_edges, kept, kept_id, n_kept, labels = ints(2 * room), ints(1), ints(2 * m), ints(m), ints(1), ints(n)
    outs = {"embed": [emb], "graph": [n_edges, edges], "filter": [score, n_kept, kept, kept_id], "labels": [labels]}
    p = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    stream = torch.cuda.Stream()
    st = ctypes.c_void_p(stream.cuda_stream)
    calls = {
        "embed": lambda: net.lib.gnn_embed(net.handle, p(xs), n, p(emb), st),
        "graph": lambda: net.lib.gnn_build_graph(net.handle, p(emb), 8, p(xs), n, 0.3, room, p(edges), p(n_edges), st),
        "filter": lambda: net.lib.gnn_filter_edges(net.handle, p(xs), p(es), n, m, 0.5, p(score), p(kept), p(kept_id),
                                                   p(n_kept), st),
        "labels": lambda: net.lib.gnn_track_labels(net.handle, p(score), p(es), n, m, 0.5, p(labels), st)}

    def inputs(seed):
        x, e = _event(seed)
        assert x.shape == (n, 12) and e.shape == (2, m)
        xs.copy_(torch.from_numpy(x)); es.copy_(torch.from_numpy(e))

    def clear():
        for t in (t for o in outs.values() for t in o):
            t.zero_()
        torch.cuda.synchronize()

    def read():
        torch.cuda.synchronize()
        return {k: [t.cpu().numpy().tobytes() for t in o] for k, o in outs.items()}
    inputs(0)
    graphs = {}
    for k, call in calls.items():
        assert call() == 0                                     # eager first: the scratch is made here
        stream.synchronize()
        graphs[k] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graphs[k], stream=stream):
            assert call() == 0
    for seed in (1, 0):
        inputs(seed)
        clear()
        for call in calls.values():
            assert call() == 0
        want = read()
        assert 0 < int(n_edges.item()) <= room and 0 < int(n_kept.item()) < m
        clear()
        for g in graphs.values():
            g.replay()
            torch.cuda.synchronize()
        assert read() == want
    assert net.status() == 0
    net.close()


def test_concurrent_contexts_on_separate_streams():
    """Several contexts (model instances) score different events on their own streams at the same
    time; each result equals its event scored alone."""
    import torch
    from paper_2402_09633_gb300 import InteractionNetwork
    cfg = S.ModelConfig(12, 2, 128, 2, 3)
    W = S.init_weights(cfg, 6)
    events = [_event(k, n=2000 + 500 * k, e=7000 + 1000 * k) for k in range(3)]
    nets = [InteractionNetwork(cfg, S.pack_blob(cfg, W)) for _ in events]
    streams = [torch.cuda.Stream() for _ in events]
    inputs = [(torch.from_numpy(x).cuda(), torch.from_numpy(e).cuda()) for x, e in events]
    outs = []
    torch.cuda.synchronize()
    for net, st, (xs, es) in zip(nets, streams, inputs):
        with torch.cuda.stream(st):
            outs.append(net.infer(xs, es, stream=st))
    for net, st in zip(nets, streams):
        assert net.status(stream=st) == 0
    ref = InteractionNetwork(cfg, S.pack_blob(cfg, W))
    for (x, e), (xs, es), o in zip(events, inputs, outs):
        alone = ref.infer(xs, es).cpu().numpy()
        assert o.cpu().numpy().tobytes() == alone.tobytes()
        check_parity(alone, W, x, e, cfg.n_iters)
    ref.close()
    for net in nets:
        net.close()
