"""Contracted [ds) kets whose second shell's exponents are next to nothing: the pair distance that the sums of scaled R
tables recover from (Q - C) / s stays finite in its square."""
import numpy as np
import pytest
import torch

import oracle
from oracle import parity
from paper_2405_01834_gb300 import inputs, mdx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lq", [(0, 0, 2, 0), (1, 1, 2, 0)])
@pytest.mark.parametrize("z", [1e-130, 1e-170, 1e-280])
def test_tiny_second_exponents(lq, z):
    n = 180   # one lane per quartet, so that every lane runs all the ket primitives
    b, q = inputs.class_sweep(lq, n_bra=n, n_ket=n, seed=83, K=(1, 1, 1, 3))
    for s in range(2 * n + 1, 4 * n, 2):
        o = b.prim_off[s]
        b.exps[o: o + 3] *= z
    eng, db = mdx.Engine(0), mdx.DeviceBasis(b)
    v, off = eng.eri4(db, q)
    eng.sync()
    sel = np.arange(0, len(q), 307)
    ref, roff = oracle.eri4(b, q[sel])
    v, off = v.cpu().numpy(), np.asarray(off.cpu())
    got = np.concatenate([v[off[i]: off[i + 1]] for i in sel])
    parity.check(got, ref, roff, "%s exponents x %g" % (lq, z), parity.Eri4Evaluator(b, q[sel]))
    eng.close()
