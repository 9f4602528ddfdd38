"""What a workspace admits: every call of the size it was made for, whatever the
schedule was when it was made and is when it is used, and calls of other shapes
that fit it, with the oracle's results."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def lnbnn():
    from paper_1112_0059_gb300 import build, lnbnn
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    build.build()
    lnbnn.load_library()
    return lnbnn


def _case(seed, N, M):
    rng = np.random.default_rng(seed)
    ref = rng.integers(0, 256, size=(N, 128)).astype(np.uint8)
    q = rng.integers(0, 256, size=(M, 128)).astype(np.uint8)
    return ref, q, torch.from_numpy(ref).cuda(), torch.from_numpy(q).cuda()


def _check(ix, ws, ref, q, qd, k, rows):
    idx, dist = ix.knn_search(qd, k, workspace=ws)
    ix.sync()
    wd, wi = oracle.knn(ref, q[rows], k)
    assert np.array_equal(dist.cpu().numpy()[rows], wd) and np.array_equal(idx.cpu().numpy()[rows], wi)


@pytest.mark.parametrize("made,used", [(dict(query_tiles=2), dict(automatic=True)),
                                       (dict(automatic=True), dict(query_tiles=2)),
                                       (dict(query_tiles=2, persistent=1), dict(query_tiles=1, persistent=0))])
def test_made_and_used_under_different_schedules(lnbnn, made, used):
    M, k = 20_000, 10  # more query tiles than SMs
    ref, q, rd, qd = _case(1, 5000, M)
    rows = np.random.default_rng(2).choice(M, size=300, replace=False)
    with lnbnn.Index(rd, torch.zeros(len(ref), dtype=torch.int32, device="cuda"), 1) as ix:
        ix.set_schedule(**made)
        with ix.workspace(M, k) as ws:
            ix.set_schedule(**used)
            _check(ix, ws, ref, q, qd, k + 1, rows)  # lists of max_k + 1, as a classify call keeps
            _check(ix, ws, ref, q[:999], qd[:999].contiguous(), k, np.arange(0, 999, 3))


@pytest.mark.parametrize("N,made,m,k", [(7000, (100, 10), 300, 2),    # smaller candidate buffers for more CTAs
                                        (60_000, (100, 10), 250, 5),
                                        (600, (128, 200), 700, 10),   # fewer buffers than CTAs: items from a queue
                                        (5000, (1000, 10), 100, 100),  # longer lists of fewer queries
                                        (60_000, (3000, 12), 8, 255),
                                        (60_000, (3000, 2), 40, 63)])  # takes fewer splits
def test_other_shapes_that_fit(lnbnn, N, made, m, k):
    ref, q, rd, qd = _case(3, N, m)
    with lnbnn.Index(rd, torch.zeros(N, dtype=torch.int32, device="cuda"), 1) as ix, ix.workspace(*made) as ws:
        _check(ix, ws, ref, q, qd, k, np.arange(m))
