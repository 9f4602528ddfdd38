"""Images of a few rows among larger ones: the rows of a block then belong to many
images, with and without a table of the classes in shared memory."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("C,k", [(9, 10), (9, 50), (8193, 10)])
@pytest.mark.parametrize("sizes", [[1] * 3000, [2, 0, 1] * 400 + [40, 8, 7, 300] + [1, 0, 0, 5] * 300, [0] * 50 + [1500]])
def test_tiny_images(C, k, sizes):
    from paper_1112_0059_gb300 import build, lnbnn
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    build.build()
    if C > 1000:
        sizes = sizes[:100] + sizes[-100:]
    rng = np.random.default_rng(len(sizes))
    ref = rng.integers(0, 7, size=(C + 500, 128)).astype(np.uint8)
    labels = rng.integers(0, C, size=len(ref)).astype(np.int32)
    labels[:C] = np.arange(C)
    q = rng.integers(0, 7, size=(sum(sizes), 128)).astype(np.uint8)
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    with lnbnn.Index(dev(ref), dev(labels), C) as ix:
        t, c = ix.lnbnn_classify(dev(q), dev(off), k)
        nt, nc = ix.nbnn_classify(dev(q), dev(off))
        ix.sync()
        for got, want in (((t, c), oracle.local_nbnn(ref, labels, C, q, off, k)),
                          ((nt, nc), oracle.nbnn(ref, labels, C, q, off))):
            assert np.array_equal(got[0].cpu().numpy(), want[0]) and np.array_equal(got[1].cpu().numpy(), want[1])
        bad = off.copy()
        bad[len(off) // 2] += 1 + off[-1]
        ix.lnbnn_classify(dev(q), dev(bad), k)
        with pytest.raises(lnbnn.LnbnnError):
            ix.sync()
