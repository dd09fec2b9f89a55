"""The shares of small launches (lanes and teams per quartet) depend on the call alone."""
import pytest
import torch

from paper_2405_01834_gb300 import inputs, mdx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("atoms,every", [(2, 1), (4, 2), (6, 1)])
def test_bits_do_not_depend_on_another_capture(atoms, every):
    """A multi-class run gives the same bits while another capture holds the context's streams and all its launches go
    to the caller's stream."""
    b = inputs.small_molecule(n_atoms=atoms)
    q = inputs.unique_quartets(b.n_shells)[::every]
    eng, db = mdx.Engine(0), mdx.DeviceBasis(b)
    b1, b2 = eng.batch_eri4(db, q[::7]), eng.batch_eri4(db, q)
    o1, o2 = (torch.zeros(x.total, dtype=torch.float64, device="cuda") for x in (b1, b2))
    b1.run(o1)
    b2.run(o2)
    torch.cuda.synchronize()
    want = o2.clone()
    o2.zero_()
    torch.cuda.synchronize()
    side, g = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, capture_error_mode="relaxed"):
        b1.run(o1)
        with torch.cuda.stream(side):
            b2.run(o2)
    torch.cuda.synchronize()
    assert torch.equal(o2, want)
    eng.sync()
    b1.close()
    b2.close()
    eng.close()
