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


@pytest.mark.parametrize("k1,shortlist", [(1, None), (6, None), (7, None), (32, None), (11, 32), (31, 32)])
def test_rows_of_many_lists(lnbnn, k1, shortlist):
    """One list of a row, a lane's worth of lists and one more, the most there
    can be, and keys that all come from one list or are spread over all."""
    rng = np.random.default_rng(k1)
    near = rng.integers(0, 256, size=128)
    ref = rng.integers(0, 256, size=(320 * 256, 128)).astype(np.uint8)
    at = np.concatenate([np.arange(70_000, 70_040), np.arange(100, 81_000, 2_000)])
    ref[at] = np.clip(near + rng.integers(-2, 3, size=(len(at), 128)), 0, 255)
    q = rng.integers(0, 256, size=(9, 128)).astype(np.uint8)
    q[:4] = ref[at[:4]]
    labels = (np.arange(len(ref)) % 11).astype(np.int32)
    off = np.array([0, 1, 1, 9])
    want = oracle.knn_coarse(ref, q, k1, shortlist) if shortlist else oracle.knn(ref, q, k1)
    with lnbnn.Index(dev(ref), dev(labels), 11) as ix:
        if shortlist:
            ix.prepare_fp8()
        for splits in (1, 2, 32, 33, 160, 161, 304):
            ix.set_schedule(splits=splits)
            i, d = ix.knn_search(dev(q), k1, shortlist=shortlist)
            t, c = ix.lnbnn_classify(dev(q), dev(off), k1 - 1, shortlist=shortlist) if k1 > 1 else (None, None)
            ix.sync()
            assert np.array_equal(d.cpu().numpy(), want[0]) and np.array_equal(i.cpu().numpy(), want[1]), splits
            if t is not None:
                total = np.zeros((3, 11), np.int64)
                for r in range(9):
                    seen = set()
                    for s in range(k1 - 1):
                        lab = labels[want[1][r, s]]
                        if lab not in seen:
                            seen.add(lab)
                            total[0 if r == 0 else 2, lab] += int(want[0][r, s]) - int(want[0][r, k1 - 1])
                assert np.array_equal(t.cpu().numpy(), total) and np.array_equal(c.cpu().numpy(), total.argmin(1)), splits
