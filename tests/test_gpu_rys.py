"""The Rys-quadrature kernel (shellsets of uncontracted classes without a register kernel) against the oracle: tables in
shared memory in one chunk or several, tables in global memory, odd and even total angular momentum, one-centre bras,
and the ends of the node table (T = 0, T around 100, T far above)."""
import numpy as np
import pytest
import torch

import oracle
from oracle import parity
from paper_2405_01834_gb300 import inputs, mdx

pytestmark = pytest.mark.gpu

CLASSES4 = [((6, 1, 0, 0), 9), ((2, 2, 2, 1), 9), ((2, 2, 2, 2), 9), ((0, 3, 1, 4), 7), ((3, 3, 3, 3), 5),
            ((4, 2, 5, 0), 5), ((4, 4, 4, 4), 3), ((6, 6, 3, 3), 2), ((5, 5, 5, 5), 2), ((6, 5, 4, 6), 2), ((6, 6, 6, 6), 2)]
CLASSES3 = [((6, 1, 0), 9), ((3, 2, 2), 7), ((4, 4, 3), 5), ((6, 6, 6), 2)]


def _is_rys(eng, lq, batch, one=False):
    """The batch's class count differs from the step programs' exactly when the Rys kernel runs."""
    return batch.exec_fma != batch.n * eng.plan_info(*lq, one_centre=one).exec_fma


@pytest.mark.parametrize("lq,n", CLASSES4)
def test_rys_4center(lq, n):
    b, q = inputs.class_sweep(lq, n_bra=n, n_ket=n, seed=91)
    eng, db = mdx.Engine(0), mdx.DeviceBasis(b)
    B = eng.batch_eri4(db, q)
    assert _is_rys(eng, lq, B)
    out = torch.full((B.total,), float("nan"), dtype=torch.float64, device="cuda")
    B.run(out)
    B.run(out)
    eng.sync()
    ref, off = oracle.eri4(b, q)
    parity.check(out.cpu().numpy(), ref, off, "rys %s" % (lq,), parity.Eri4Evaluator(b, q))
    B.close()
    eng.close()


@pytest.mark.parametrize("lt,n", CLASSES3)
def test_rys_3center(lt, n):
    aux, orb, t = inputs.class_sweep3(lt, n_aux=n, n_ket=n, seed=92)
    eng = mdx.Engine(0)
    B = eng.batch_eri3(mdx.DeviceBasis(aux), mdx.DeviceBasis(orb), t)
    assert _is_rys(eng, (lt[0], 0, lt[1], lt[2]), B, True)
    out = torch.full((B.total,), float("nan"), dtype=torch.float64, device="cuda")
    B.run(out)
    eng.sync()
    ref, off = oracle.eri3(aux, orb, t)
    parity.check(out.cpu().numpy(), ref, off, "rys3 %s" % (lt,), parity.Eri3Evaluator(aux, orb, t))
    B.close()
    eng.close()


@pytest.mark.parametrize("lq", [(2, 2, 2, 2), (3, 3, 3, 2), (5, 4, 4, 5)])
def test_rys_node_table_ends(lq):
    """zeta_p = zeta_q = 2 (rho = 1), so T is the squared distance of the two pairs: 0, on both sides of an interval's
    end and of 100, and large; through the one-shot call, whose arrays are context workspace."""
    bb = inputs.BasisBuilder()
    quartets = []
    for R in (0.0, 1e-6, np.sqrt(1.0 - 1e-12), 1.0, 3.3, np.sqrt(99.999), 10.0, np.sqrt(100.001), 40.0):
        s = len(bb.l)
        for l, z in zip(lq, (0.0, 0.0, R, R)):
            bb.add_shell(l, [0.3, -0.2, z], [1.0], [float(inputs.primitive_norm(l, np.array([1.0]))[0])])
        quartets.append([s, s + 1, s + 2, s + 3])
    b, q = bb.build(), np.array(quartets, dtype=np.int32)
    eng = mdx.Engine(0)
    v, off = eng.eri4(mdx.DeviceBasis(b), q)
    eng.sync()
    ref, roff = oracle.eri4(b, q)
    assert np.array_equal(off.cpu().numpy(), roff)
    parity.check(v.cpu().numpy(), ref, roff, "rys T ends %s" % (lq,), parity.Eri4Evaluator(b, q))
    eng.close()
