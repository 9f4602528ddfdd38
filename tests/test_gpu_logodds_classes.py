"""The log-odds rule with more classes than a block keeps a table for: totals within
float64 rounding of the oracle's, alone and in the batch, and no step in the time
where the form changes."""
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


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("C,positive_only", [(1024, True), (1025, True), (4096, False), (8192, True), (8193, False)])
def test_many_classes_and_chunks(lnbnn, C, positive_only):
    """An increment is a difference of terms of at most beta D + log C; up to 203 of
    them add up, in chunks."""
    rng = np.random.default_rng(C)
    beta, sizes = 1e-3, [203, 0, 3, 15, 16, 1]
    ref = rng.integers(0, 7, size=(C + 300, 128)).astype(np.uint8)
    labels = rng.integers(0, C, size=len(ref)).astype(np.int32)
    labels[:C] = np.arange(C)
    q = rng.integers(0, 7, size=(sum(sizes), 128)).astype(np.uint8)
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    with lnbnn.Index(dev(ref), dev(labels), C) as ix, ix.workspace(len(q), 1) as ws:
        t, c, n = ix.nbnn_logodds_classify(dev(q), dev(off), beta, positive_only=positive_only, workspace=ws)
        alone = ix.nbnn_logodds_classify(dev(q[:203]), dev(off[:2]), beta, positive_only=positive_only)
        ix.sync()
        assert torch.equal(alone[0][0], t[0]) and torch.equal(alone[1][0], c[0]) and torch.equal(alone[2][0], n[0])
    # the increments with every class's others as the row's sum without it, in long doubles
    # (the exponents span 4.6 at most, so the difference keeps their precision)
    D = oracle.class_min(ref, labels, C, q).astype(np.longdouble)
    x = -beta * (D - D.min(axis=1, keepdims=True))
    e = np.exp(x)
    inc = x - np.log(e.sum(axis=1, keepdims=True) - e) + np.log(np.longdouble(C - 1))
    tol_inc = oracle.logodds.decision_tolerance(D.astype(np.float64), beta)
    ot, _, on, near = oracle.logodds.sum_increments(inc.astype(np.float64), off, positive_only, tol_inc)
    tol = 203 * 8 * np.finfo(np.float64).eps * (beta * 128 * 6 ** 2 + np.log(C)) * 16
    assert np.abs(t.cpu().numpy() - ot).max() <= tol + tol_inc * near.max()
    assert np.all(np.abs(n.cpu().numpy() - on) <= near)


def test_time_of_one_class_more(lnbnn):
    """4,097 classes take about as long as 4,096, and 8,192 about twice that."""
    ms = {}
    for C in (4096, 4097, 8192):
        rng = np.random.default_rng(C)
        ref = dev(rng.integers(0, 256, size=(2 * C, 128)).astype(np.uint8))
        q = dev(rng.integers(0, 256, size=(1000, 128)).astype(np.uint8))
        off = dev(np.array([0, 1000], np.int64))
        with lnbnn.Index(ref, dev((np.arange(2 * C) // 2).astype(np.int32)), C) as ix:
            times = []
            for _ in range(4):
                a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
                a.record()
                ix.nbnn_logodds_classify(q, off, 1e-5)
                b.record()
                torch.cuda.synchronize()
                times.append(a.elapsed_time(b))
            ms[C] = min(times)
    assert ms[4097] < 3 * ms[4096] and ms[8192] < 6 * ms[4096], ms
