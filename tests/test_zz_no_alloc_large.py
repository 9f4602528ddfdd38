"""knn_search_noalloc where its scratch is nearly full (candidate buffers of fewer
entries), and with more work items than CTAs (items from a queue): the same as
knn_search, and as the oracle on some of the rows."""
import ctypes

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n_ref,n_q,k", [(200_000, 1000, 10), (150_000, 2000, 10), (190_000, 100, 50),
                                         (100_000, 1000, 200), (6000, 20_000, 10), (9000, 24_000, 100)])
def test_large_problems_match_knn_search(n_ref, n_q, k):
    from paper_1112_0059_gb300 import build, lnbnn
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    build.build()
    lib = lnbnn.load_library()
    P = ctypes.c_void_p
    lib.knn_search_noalloc.argtypes = [P, ctypes.c_int64, P, ctypes.c_int64, ctypes.c_int32, P, P, P]
    lib.knn_search_noalloc.restype = ctypes.c_int
    rng = np.random.default_rng(n_ref + k)
    ref = rng.integers(0, 256, size=(n_ref, 128), dtype=np.uint8)
    q = rng.integers(0, 256, size=(n_q, 128), dtype=np.uint8)
    rd, qd = torch.from_numpy(ref).cuda(), torch.from_numpy(q).cuda()
    idx = torch.empty((n_q, k), dtype=torch.int32, device="cuda")
    dist = torch.empty_like(idx)
    code = lib.knn_search_noalloc(P(rd.data_ptr()), n_ref, P(qd.data_ptr()), n_q, k, P(idx.data_ptr()),
                                  P(dist.data_ptr()), P(torch.cuda.current_stream().cuda_stream))
    assert code == 0, lnbnn.STATUS.get(code)
    with lnbnn.Index(rd, torch.zeros(n_ref, dtype=torch.int32, device="cuda"), 1) as ix:
        want_idx, want_dist = ix.knn_search(qd, k)
        ix.sync()
    assert torch.equal(idx, want_idx) and torch.equal(dist, want_dist)
    rows = rng.choice(n_q, size=50, replace=False)
    wd, wi = oracle.knn(ref, q[rows], k)
    assert np.array_equal(dist.cpu().numpy()[rows], wd) and np.array_equal(idx.cpu().numpy()[rows], wi)
