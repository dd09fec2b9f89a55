"""The work model of the batched exchange: that of mdx_exchange_screen, whose class order the paper's figures use."""
import pytest
import torch

import numpy as np

from paper_2405_01834_gb300 import inputs, mdx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tau", [0.0, 1e-9])
def test_model_flops_are_those_of_the_screening(tau):
    eng = mdx.Engine(0)
    mols = [inputs.molecule(seed=90 + i, n_atoms=1 + i % 2) for i in range(3)]
    mols.append(inputs.small_molecule(seed=80, n_atoms=3, shells=(2, 0, 1), K=2))
    bases = [mdx.DeviceBasis(b) for b in mols]
    Ds = [torch.from_numpy(inputs.density(b.nao, 5 + i)) for i, b in enumerate(mols)]
    xb = eng.xbatch(bases, Ds, tau=tau)
    n, flops = 0, 0.0
    for b, db, D in zip(mols, bases, Ds):
        p = np.array([(i, j) for i in range(b.n_shells) for j in range(i + 1)], dtype=np.int32)
        _, m, f = eng.exchange_screen(db, p, eng.schwarz(db, p), D, tau, list_quartets=False)
        n += m
        flops += f
    assert xb.n_quartets == n
    assert xb.model_flops == pytest.approx(flops, rel=1e-12)
    assert sum(xb.launch_info(i)[2] for i in range(xb.n_class_launches)) == pytest.approx(flops, rel=1e-12)
    eng.sync()
    xb.close()
    eng.close()
