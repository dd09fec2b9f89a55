"""mdx_set_class_shape: a team size or a shared-memory budget means the team kernel, neither the engine's own choice."""
import pytest
import torch

from paper_2405_01834_gb300 import inputs, mdx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lq", [(2, 2, 2, 2), (3, 3, 3, 3)])
def test_a_given_shape_runs_teams(lq):
    b, q = inputs.class_sweep(lq, n_bra=3, n_ket=3, seed=57)
    db = mdx.DeviceBasis(b)
    want = None
    for shape, kernel in (({}, "k_rys"), ({"smem_budget": 64 * 1024}, "k_quartets"), ({"team_threads": 128}, "k_quartets"),
                          ({"variant": 1}, "k_quartets"), ({}, "k_rys")):
        eng = mdx.Engine(0)
        eng.set_class_shape(*lq, **shape)
        B = eng.batch_eri4(db, q)
        assert [c["kernel"] for c in B.classes()] == [kernel], shape
        if kernel == "k_quartets":   # the shape asked for is the one that runs
            assert B.exec_fma == B.n * eng.plan_info(*lq).exec_fma
        out = torch.empty(B.total, dtype=torch.float64, device="cuda")
        B.run(out)
        eng.sync()
        want = out.clone() if want is None else want
        assert float((out - want).abs().max()) <= 1e-12 * float(want.abs().max())
        B.close()
        eng.close()
