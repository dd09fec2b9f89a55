"""Launches too small to fill the GPU: lanes that share a quartet's primitive pairs in the register kernel."""
import pytest

import oracle
from oracle import parity
from paper_2405_01834_gb300 import inputs, mdx

pytestmark = pytest.mark.gpu


# register classes (R, [p|cd] and the shellset in registers) and shared-memory ones; contraction degrees that leave
# partial rounds of primitives for every lane count
@pytest.mark.parametrize("lq,K", [((0, 0, 0, 0), (5, 7, 3, 11)), ((1, 0, 1, 0), (3, 6, 1, 5)), ((0, 1, 2, 0), (1, 1, 6, 3)),
                                  ((1, 1, 1, 1), (3, 3, 3, 3)), ((2, 1, 1, 0), (1, 3, 3, 6)), ((3, 0, 0, 2), (2, 1, 6, 1)),
                                  ((4, 0, 1, 0), (1, 7, 1, 1)), ((1, 2, 1, 1), (5, 1, 1, 2))])
def test_lanes_sharing_a_quartet(lq, K):
    b, q = inputs.class_sweep(lq, n_bra=151, n_ket=163, seed=77, K=K)
    eng, db = mdx.Engine(0), mdx.DeviceBasis(b)
    assert eng.plan_info(*lq, K[0] * K[1], K[2] * K[3]).register_kernel == 1
    sizes = (1, 5, 33, 1000, 4000)         # from 32 lanes per quartet down
    ref, roff = oracle.eri4(b, q[: sizes[-1]])
    for n in sizes:
        part, off = eng.eri4(db, q[:n])
        parity.check(part.cpu().numpy(), ref[: roff[n]], roff[: n + 1], "%s K=%s n=%d" % (lq, K, n),
                     parity.Eri4Evaluator(b, q[:n]))
    eng.sync()
    eng.close()
