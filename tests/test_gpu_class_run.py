"""What a prepared batch says it runs, and the operations it counts for it."""
import pytest

from paper_2405_01834_gb300 import inputs, mdx

pytestmark = pytest.mark.gpu


def nherm(n):
    return (n + 1) * (n + 2) * (n + 3) // 6


def _batch(eng, lq, K, n):
    b, q = inputs.class_sweep(lq, n_bra=n, n_ket=n, seed=51, K=K)
    return eng.batch_eri4(mdx.DeviceBasis(b), q)


@pytest.fixture(scope="module")
def eng():
    e = mdx.Engine(0)
    yield e
    e.close()


def one(B):
    (c,) = B.classes()
    assert B.exec_fma == pytest.approx(c["n"] * c["exec_fma"], rel=1e-12) and c["n"] == B.n
    return c


@pytest.mark.parametrize("lq", [(2, 2, 2, 2), (3, 3, 3, 3), (6, 6, 6, 6)])
def test_rys_operations(eng, lq):
    """Two instructions per integral and node, a product and a multiply-add: three operations, 1.5 multiply-adds."""
    c = one(_batch(eng, lq, (1, 1, 1, 1), 2))
    n_out = 1
    for l in lq:
        n_out *= inputs.ncart(l)
    nodes = sum(lq) // 2 + 1
    assert c["kernel"] == "k_rys" and c["lanes"] == c["teams"] == 1
    assert c["fp64_instr"] - c["exec_fma"] == pytest.approx(0.5 * nodes * n_out, rel=1e-9)
    assert 1.5 * nodes * n_out < c["exec_fma"] < 2.5 * nodes * n_out


@pytest.mark.parametrize("lq,K,per_prim,per_bra", [
    # sums of R tables: orders 0 .. L_b and 1 .. L_b + 1 for [ps), six terms of [p|cd] per Hermite index
    ((3, 0, 1, 0), (1, 2, 3, 6), nherm(3) + nherm(4) - 1, 6 * nherm(3)),
    ((1, 1, 1, 0), (3, 1, 1, 6), nherm(2) + nherm(3) - 1, 6 * nherm(2))])
def test_ket_sums_operations(eng, lq, K, per_prim, per_bra):
    """A launch that fills the GPU sums R tables in place of the ket transform (two products per component and Hermite
    index); a small one shares the primitives between lanes and transforms each."""
    Kb, Kk = K[0] * K[1], K[2] * K[3]
    plan = eng.plan_info(*lq, Kb, Kk).exec_fma
    ket = 6 * nherm(lq[0] + lq[1])
    c = one(_batch(eng, lq, K, 180))
    assert c["kernel"] == "k_reg" and c["lanes"] == 1
    assert c["exec_fma"] == pytest.approx(plan + Kb * (Kk * (per_prim - ket) + per_bra), rel=1e-12)
    assert c["fp64_instr"] == c["exec_fma"]
    c = one(_batch(eng, lq, K, 3))
    assert c["lanes"] > Kk // 3
    assert c["exec_fma"] == plan


def test_kernels_of_a_mixed_batch(eng):
    """One class of each kernel, in one batch."""
    bb = inputs.BasisBuilder()
    for l, K in ((0, 1), (1, 1), (2, 1), (2, 3), (0, 3)):
        for x in range(2):
            bb.add_shell(l, [0.3 * l, 0.7 * x, 0.1 * K], [1.0 + k for k in range(K)], [1.0] * K)
    q = [[0, 1, 0, 1], [2, 3, 2, 3], [4, 5, 4, 5], [6, 7, 6, 7], [8, 9, 8, 9]]
    B = eng.batch_eri4(mdx.DeviceBasis(bb.build()), q)
    got = {(c["l"], c["K"]): c for c in B.classes()}
    assert len(got) == 5
    assert got[(1, 1, 1, 1), (1, 1)]["kernel"] == "k_reg_single"
    assert got[(2, 2, 2, 2), (1, 1)]["kernel"] == "k_rys"
    assert got[(2, 2, 2, 2), (9, 9)]["kernel"] == "k_quartets" and got[(2, 2, 2, 2), (9, 9)]["teams"] > 1
    assert got[(0, 0, 0, 0), (9, 9)]["kernel"] == "k_reg" and got[(0, 0, 0, 0), (9, 9)]["lanes"] > 1
    assert B.exec_fma == pytest.approx(sum(c["exec_fma"] for c in B.classes()), rel=1e-12)
    B.close()
