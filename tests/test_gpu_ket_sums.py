"""Register-kernel classes whose contracted kets [ps), [ds), [pp) are summed as scaled R tables, against the oracle: every
layout of the tables (registers, shared memory, two groups), the fewest ket primitives that take it, ket shells that
share a centre, and ket exponents far apart on either shell."""
import numpy as np
import pytest
import torch

import oracle
from oracle import parity
from paper_2405_01834_gb300 import inputs, mdx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lq,K", [((0, 0, 1, 0), (1, 2, 3, 6)), ((1, 0, 1, 1), (1, 1, 3, 1)), ((0, 1, 2, 0), (1, 2, 1, 6)),
                                  ((2, 1, 1, 0), (1, 1, 2, 2)), ((1, 1, 2, 0), (1, 1, 3, 2)), ((2, 0, 1, 1), (1, 1, 1, 3)),
                                  ((4, 0, 1, 0), (1, 1, 3, 1)), ((2, 3, 1, 0), (1, 1, 3, 1)), ((0, 5, 1, 0), (1, 1, 2, 3))])
def test_contracted_kets(lq, K):
    n = 180   # 32,400 quartets: one lane each, so that every lane runs all the ket primitives
    b, q = inputs.class_sweep(lq, n_bra=n, n_ket=n, seed=79, K=K)
    for k in range(0, n, 3):            # a third of the kets: both shells on one centre
        b.center[2 * n + 2 * k + 1] = b.center[2 * n + 2 * k]
    for k in range(1, n, 6):            # exponents ten orders apart, the small one on the first or the second shell
        s = 2 * n + 2 * k + (k // 6) % 2
        o = b.prim_off[s]
        b.exps[o: o + b.nprim[s]] *= 1e-10
    for k in range(2, n, 6):            # negative exponents on the second shell, within those of the first
        i, j = (b.exps[b.prim_off[s]: b.prim_off[s] + b.nprim[s]] for s in (2 * n + 2 * k, 2 * n + 2 * k + 1))
        j[:] = -0.01 * i.min()
    eng, db = mdx.Engine(0), mdx.DeviceBasis(b)
    assert eng.plan_info(*lq, K[0] * K[1], K[2] * K[3]).register_kernel == 1
    v, off = eng.eri4(db, q)
    torch.cuda.synchronize()
    sel = np.arange(0, len(q), 101)
    ref, roff = oracle.eri4(b, q[sel])
    v, off = v.cpu().numpy(), np.asarray(off.cpu())
    got = np.concatenate([v[off[i]: off[i + 1]] for i in sel])
    parity.check(got, ref, roff, "%s K=%s" % (lq, K), parity.Eri4Evaluator(b, q[sel]))
    eng.close()
