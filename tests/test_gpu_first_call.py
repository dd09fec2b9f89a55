"""The first call of a context on a stream that does not wait for the default stream: the context's tables are there."""
import pytest
import torch

from paper_2405_01834_gb300 import inputs, mdx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lq,n", [((2, 2, 2, 2), 3), ((6, 6, 6, 6), 1)])
def test_first_rys_call_on_a_non_blocking_stream(lq, n):
    """The node table is uploaded inside the call: the launch that follows on the caller's stream (or, of several
    classes, on an internal one) reads all of it. A fresh context each time."""
    b, q = inputs.class_sweep(lq, n_bra=n, n_ket=n, seed=41)
    db = mdx.DeviceBasis(b)
    eng = mdx.Engine(0)
    want = eng.eri4(db, q)[0]
    eng.sync()
    eng.close()
    for _ in range(10):
        eng = mdx.Engine(0)
        with torch.cuda.stream(torch.cuda.Stream()):
            v, _ = eng.eri4(db, q)
            eng.sync()
            assert torch.equal(v, want)
        eng.close()
