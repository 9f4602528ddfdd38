"""The lists of the k nearest at their edges: every list length class, references
at tile edges (too few tiles for a warm-up, the 32-column and the wide one),
heavy ties, and references in order of falling distance, where every column is
a candidate and the candidate buffers fill at every step."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SCHEDULES = (dict(automatic=True), dict(splits=1, query_tiles=1), dict(splits=3, bound_per_tile=0, persistent=0),
             dict(splits=1, query_tiles=2, persistent=1))


@pytest.fixture(scope="module")
def lnbnn():
    from paper_1112_0059_gb300 import build, lnbnn
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    build.build()
    lnbnn.load_library()
    return lnbnn


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def check(lnbnn, ref, q, k1, shortlist=None):
    want = oracle.knn_coarse(ref, q, k1, shortlist) if shortlist else oracle.knn(ref, q, k1)
    with lnbnn.Index(dev(ref), dev(np.zeros(len(ref), np.int32)), 1) as ix:
        if shortlist:
            ix.prepare_fp8()
        for sch in SCHEDULES:
            ix.set_schedule(**sch)
            i, d = ix.knn_search(dev(q), k1, shortlist=shortlist)
            ix.sync()
            assert np.array_equal(d.cpu().numpy(), want[0]) and np.array_equal(i.cpu().numpy(), want[1]), (len(ref), sch)


@pytest.mark.parametrize("k1", [1, 16, 17, 32, 33, 64, 65, 128, 129, 255])
def test_lists_at_tile_edges(lnbnn, k1):
    rng = np.random.default_rng(k1)
    for n, hi in ((256, 3), (257, 256), (1279, 4), (6 * 256 + 1, 256), (40_001, 6)):
        if n < k1:
            continue
        ref = rng.integers(0, hi, size=(n, 128)).astype(np.uint8)
        q = rng.integers(0, hi, size=(130, 128)).astype(np.uint8)
        q[:2], ref[n // 2] = ref[0], ref[0]
        check(lnbnn, ref, q, k1)


@pytest.mark.parametrize("k1,shortlist", [(11, None), (50, None), (200, None), (11, 24), (11, 64), (11, 128)])
def test_falling_distances(lnbnn, k1, shortlist):
    rng = np.random.default_rng(3)
    q0 = rng.integers(0, 256, size=128)
    ref = rng.integers(0, 256, size=(9000, 128)).astype(np.uint8)
    ref = ref[np.argsort(-((ref.astype(np.int64) - q0) ** 2).sum(1), kind="stable")]
    q = np.clip(q0 + rng.integers(-3, 4, size=(140, 128)), 0, 255).astype(np.uint8)
    check(lnbnn, ref, q, k1, shortlist)
