"""Launches of up to 96 query rows, which are spread over the four TMEM lane quarters:
every row count at the edges of that, every scan and list kind, against the oracle."""
import numpy as np
import pytest

import oracle
import oracle.logodds

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def lnbnn():
    from paper_1112_0059_gb300 import build, lnbnn
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    build.build()
    lnbnn.load_library()
    return lnbnn


@pytest.mark.parametrize("width,weight", [(128, None), (130, 10)])
def test_row_counts(lnbnn, width, weight):
    N, C = 9000, 5
    rng = np.random.default_rng(width)
    ref = rng.integers(0, 256, (N, width)).astype(np.uint8)
    ref[70:75] = ref[3]
    labels = (np.arange(N) % C).astype(np.int32)
    q = rng.integers(0, 256, (130, width)).astype(np.uint8)
    q[0] = ref[3]
    wd, wi = oracle.knn(ref, q, 129, location_weight=weight)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    with lnbnn.Index(dev(ref), dev(labels), C, location_weight=weight) as ix:
        if weight is None:
            ix.prepare_fp8()
        for m in (1, 2, 3, 4, 5, 7, 8, 9, 17, 31, 32, 33, 63, 64, 65, 93, 94, 95, 96, 97, 127, 128, 129):
            qd = dev(q[:m])
            off = np.array([0, m // 3, m], np.int64)
            for schedule in (dict(automatic=True), dict(query_tiles=2), dict(splits=3)):
                ix.set_schedule(**schedule)
                for k in (1, 10, 24, 32, 50, 129):
                    i, d = ix.knn_search(qd, k)
                    ix.sync()
                    assert np.array_equal(d.cpu().numpy(), wd[:m, :k]) and np.array_equal(i.cpu().numpy(), wi[:m, :k]), (m, k)
                if weight is None:
                    for s in (16, 48, 100):
                        i, d = ix.knn_search(qd, 9, shortlist=s)
                        ix.sync()
                        cd, ci = oracle.knn_coarse(ref, q[:m], 9, s)
                        assert np.array_equal(d.cpu().numpy(), cd) and np.array_equal(i.cpu().numpy(), ci), (m, s)
                t, c = ix.lnbnn_classify(qd, dev(off), 10)
                nt, nc = ix.nbnn_classify(qd, dev(off))
                lt, lc, ln = ix.nbnn_logodds_classify(qd, dev(off), 1e-5)
                ix.sync()
                wt = oracle.local_nbnn(ref, labels, C, q[:m], off, 10, location_weight=weight)
                wn = oracle.nbnn(ref, labels, C, q[:m], off, location_weight=weight)
                assert np.array_equal(t.cpu().numpy(), wt[0]) and np.array_equal(c.cpu().numpy(), wt[1]), m
                assert np.array_equal(nt.cpu().numpy(), wn[0]) and np.array_equal(nc.cpu().numpy(), wn[1]), m
                assert np.array_equal(ln.cpu().numpy(), np.diff(off) * C)
            ix.set_schedule(automatic=True)
