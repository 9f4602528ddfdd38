"""The per-image sums at their edges: images around the row chunks and blocks
of the score, NBNN and log-odds kernels, neighbour counts around a warp's
lanes, class counts around the shared-memory tables."""
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


SIZES = [7, 8, 9, 0, 15, 16, 17, 1, 31, 33, 0, 128, 129]


def case(seed, C, n, sizes=SIZES):
    rng = np.random.default_rng(seed)
    ref = rng.integers(0, 7, size=(n, 128)).astype(np.uint8)
    labels = rng.integers(0, C, size=n).astype(np.int32)
    labels[:C] = np.arange(C)
    q = rng.integers(0, 7, size=(sum(sizes), 128)).astype(np.uint8)
    return ref, labels, q, np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)


@pytest.mark.parametrize("k,C", [(1, 9), (31, 9), (32, 9), (33, 9), (64, 9), (65, 9), (128, 9), (129, 9), (255, 9),
                                 (10, 8192), (10, 8193)])
def test_local_and_nbnn_sums(lnbnn, k, C):
    ref, labels, q, off = case(k, C, C + 700)
    with lnbnn.Index(dev(ref), dev(labels), C) as ix:
        t, c = ix.lnbnn_classify(dev(q), dev(off), k)
        nt, nc = ix.nbnn_classify(dev(q), dev(off))
        ix.sync()
    for got, want in (((t, c), oracle.local_nbnn(ref, labels, C, q, off, k)), ((nt, nc), oracle.nbnn(ref, labels, C, q, off))):
        assert np.array_equal(got[0].cpu().numpy(), want[0]) and np.array_equal(got[1].cpu().numpy(), want[1])


@pytest.mark.parametrize("C", [2, 33, 1024, 1025, 4097])
def test_logodds_class_counts(lnbnn, C):
    """Totals within float64 rounding of the oracle's (an increment is a
    difference of terms of at most beta D + log C, and up to 33 of them add up),
    the same alone and in the batch."""
    beta, sizes = 1e-3, SIZES[:10] if C < 100 else [7, 0, 8, 1, 17]
    ref, labels, q, off = case(C, C, C + 300, sizes)
    with lnbnn.Index(dev(ref), dev(labels), C) as ix:
        lt, lc, ln = ix.nbnn_logodds_classify(dev(q), dev(off), beta)
        a, b = int(off[-2]), int(off[-1])
        alone = ix.nbnn_logodds_classify(dev(q[a:b]), dev(np.array([0, b - a])), beta)
        ix.sync()
        assert torch.equal(alone[0][0], lt[-1]) and torch.equal(alone[1][0], lc[-1]) and torch.equal(alone[2][0], ln[-1])
    ot = oracle.logodds.nbnn_logodds(ref, labels, C, q, off, beta, False)[0]
    dmax = 128 * 6 ** 2
    tol = 33 * 8 * np.finfo(np.float64).eps * (beta * dmax + np.log(C)) * 16
    assert np.abs(lt.cpu().numpy() - ot).max() <= tol
    assert np.array_equal(ln.cpu().numpy(), np.diff(off) * C)


@pytest.mark.parametrize("n_img", [1, 255, 4095, 4096, 9000])
def test_totals_cleared_and_offsets_checked(lnbnn, n_img):
    """Whatever the totals held before a call, and an image whose offset is out
    of order in any part of the check."""
    C = 7
    sizes = [1] * 40 + [0] * (n_img - 40) if n_img > 1 else [40]
    ref, labels, q, off = case(n_img, C, 400, sizes)
    want = oracle.local_nbnn(ref, labels, C, q, off, 3)[0]
    with lnbnn.Index(dev(ref), dev(labels), C) as ix:
        buf = torch.full((n_img * C + 1,), -5, dtype=torch.int64, device="cuda")
        cls = torch.empty(n_img, dtype=torch.int32, device="cuda")
        t = buf[1:].view(n_img, C)  # 8-byte aligned only
        for qq, oo in ((q, off), (q[:0], off * 0)):
            t.fill_(-5)
            ix.lnbnn_classify(dev(qq), dev(oo), 3, out=(t, cls))
            ix.sync()
            assert np.array_equal(t.cpu().numpy(), want if len(qq) else want * 0) and int(buf[0]) == -5
        bad = off.copy()
        bad[n_img - 1 if n_img > 1 else 1] = 41
        ix.lnbnn_classify(dev(q), dev(bad), 3)
        with pytest.raises(lnbnn.LnbnnError):
            ix.sync()
