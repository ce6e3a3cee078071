"""The CSR sort where its digits change: node counts on both sides of one, two and three passes, edge
counts around a tile of 4,096 and a warp's 512 elements, bit-exact against a stable host sort (through
gnn_csr_build_noalloc, which shares the sort with gnn_infer)."""
import ctypes

import numpy as np
import pytest

from oracle import gnn_oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 3, 255, 2047, 2048, 70000, (1 << 22) - 1, 1 << 22, (1 << 24) + 5])
@pytest.mark.parametrize("e", [1, 31, 511, 513, 4095, 4096, 4097, 50001])
def test_csr_digits(n, e):
    import torch
    from paper_2402_09633_gb300 import binding
    lib = binding.load_library()
    vp, i64 = ctypes.c_void_p, ctypes.c_int64
    lib.gnn_csr_build_noalloc.argtypes = [vp, i64, i64, vp, vp, vp, vp]
    lib.gnn_csr_build_noalloc.restype = ctypes.c_int
    rng = np.random.default_rng(n + e)
    ei = rng.integers(0, n, size=(2, e)).astype(np.int32)
    ei[1, : e // 3] = n - 1                              # one long segment at the end of the key range
    dev = torch.from_numpy(ei).cuda()
    rowptr = torch.full((n + 1,), -7, dtype=torch.int32, device="cuda")
    perm = torch.full((e,), -7, dtype=torch.int32, device="cuda")
    src = torch.full((e,), -7, dtype=torch.int32, device="cuda")
    p = lambda t: vp(t.data_ptr())  # noqa: E731
    rc = lib.gnn_csr_build_noalloc(p(dev), n, e, p(rowptr), p(perm), p(src), vp(torch.cuda.current_stream().cuda_stream))
    torch.cuda.synchronize()
    assert rc == 0
    want_rowptr, want_src, want_perm = O.csr_by_destination(ei[0], ei[1], n)
    np.testing.assert_array_equal(perm.cpu().numpy(), want_perm)
    np.testing.assert_array_equal(src.cpu().numpy(), want_src)
    np.testing.assert_array_equal(rowptr.cpu().numpy(), want_rowptr)
