"""The autotuner times the launch that runs: its trials share quartets between lanes and teams as the run of the whole
class does."""
import pytest
import torch

from paper_2405_01834_gb300 import inputs, mdx

pytestmark = pytest.mark.gpu


# the register kernel is the last shape that a register class tries, so its trial's integrals are what is left in the
# output; few trial quartets of a class that fills the GPU (one lane each), and of one that does not
@pytest.mark.parametrize("lq,K,n,trial", [((0, 0, 0, 0), (5, 7, 3, 11), 200, 3), ((1, 0, 1, 0), (3, 6, 1, 5), 200, 40),
                                          ((1, 1, 1, 1), (3, 3, 3, 3), 40, 2)])
def test_trials_share_quartets_as_the_run_does(lq, K, n, trial):
    b, q = inputs.class_sweep(lq, n_bra=n, n_ket=n, seed=85, K=K)
    eng = mdx.Engine(0)
    B = eng.batch_eri4(mdx.DeviceBasis(b), q)
    out = torch.zeros(B.total, dtype=torch.float64, device="cuda")
    B.run(out)
    torch.cuda.synchronize()
    m = trial * (B.total // len(q))
    want = out[:m].clone()
    out.zero_()
    torch.cuda.synchronize()
    B.autotune(out, max_trial=trial)
    torch.cuda.synchronize()
    assert torch.equal(out[:m], want) and not out[m:].any()
    B.close()
    eng.close()
