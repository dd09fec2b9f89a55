"""Launches too small to fill the GPU: lanes that share a quartet's primitive pairs in the register kernel, and
per-class launches spread over several streams (also inside a stream capture)."""
import numpy as np
import pytest
import torch

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


# team-kernel classes (total angular momentum 7 and more, several column groups in the last): teams that share a
# quartet's primitive pairs, summed inside a cluster (store) or digested one by one (exchange)
@pytest.mark.parametrize("lq,K", [((2, 2, 2, 1), (3, 3, 3, 3)), ((3, 2, 2, 0), (1, 2, 1, 5)), ((2, 2, 2, 2), (2, 1, 2, 3)),
                                  ((3, 3, 3, 3), (1, 2, 2, 1)), ((4, 1, 1, 1), (1, 7, 3, 1))])
def test_teams_sharing_a_quartet(lq, K):
    b, q = inputs.class_sweep(lq, n_bra=5, n_ket=7, seed=78, K=K)
    eng, db = mdx.Engine(0), mdx.DeviceBasis(b)
    assert eng.plan_info(*lq, K[0] * K[1], K[2] * K[3]).register_kernel == 0
    ref, roff = oracle.eri4(b, q)
    for n in (1, 3, len(q)):
        v, off = eng.eri4(db, q[:n])
        parity.check(v.cpu().numpy(), ref[: roff[n]], roff[: n + 1], "%s K=%s n=%d" % (lq, K, n),
                     parity.Eri4Evaluator(b, q[:n]))
    eng.sync()
    eng.close()


def test_multi_class_batch_in_a_capture():
    """A captured multi-class run replays to the same bits; a run of another batch on another stream while the
    capture holds the context's streams keeps its own results."""
    b = inputs.small_molecule(n_atoms=3)
    q = inputs.unique_quartets(b.n_shells)
    eng, db = mdx.Engine(0), mdx.DeviceBasis(b)
    b1, b2 = eng.batch_eri4(db, q), eng.batch_eri4(db, q[::3])
    o1, o2 = (torch.zeros(x.total, dtype=torch.float64, device="cuda") for x in (b1, b2))
    b1.run(o1)
    b2.run(o2)
    torch.cuda.synchronize()
    want1, want2 = o1.clone(), o2.clone()
    o1.zero_()
    o2.zero_()
    torch.cuda.synchronize()
    side, g = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, capture_error_mode="relaxed"):
        b1.run(o1)
        with torch.cuda.stream(side):
            b2.run(o2)
        b1.run(o1)
    torch.cuda.synchronize()
    assert torch.equal(o2, want2) and not o1.any()
    for _ in range(2):
        o1.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(o1, want1)
    eng.sync()
    b1.close()
    b2.close()
    eng.close()
