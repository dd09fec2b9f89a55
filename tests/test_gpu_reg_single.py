"""Uncontracted shellsets of the one-warp register kernel (columns [p|cd] formed one at a time) against the oracle, with
quartet counts around the warp and shells that share centres."""
import numpy as np
import pytest
import torch

import oracle
from oracle import parity
from paper_2405_01834_gb300 import inputs, mdx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lq", [(1, 1, 1, 1), (2, 0, 1, 1), (1, 1, 0, 2), (2, 0, 2, 0), (0, 2, 2, 0), (0, 0, 2, 2), (1, 0, 2, 1),
                                (0, 1, 0, 4), (0, 0, 5, 0), (1, 0, 0, 3)])
def test_uncontracted_shellsets(lq):
    b, q = inputs.class_sweep(lq, n_bra=11, n_ket=6, seed=80)
    b.center[1] = b.center[0]           # a one-centre bra, a one-centre ket, and a quartet on one centre
    b.center[23] = b.center[22]
    b.center[24:26] = b.center[2:4] = b.center[2]
    eng, db = mdx.Engine(0), mdx.DeviceBasis(b)
    assert eng.plan_info(*lq).register_kernel == 1
    ref, roff = oracle.eri4(b, q)
    for n in (1, 31, 33, 66):
        v, off = eng.eri4(db, q[:n])
        parity.check(v.cpu().numpy()[: roff[n]], ref[: roff[n]], roff[: n + 1], "%s n=%d" % (lq, n),
                     parity.Eri4Evaluator(b, q[:n]))
    eng.close()
