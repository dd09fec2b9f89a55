"""Runs of prepared batches that overlap on the GPU: the Rys classes whose axis tables live in global memory."""
import pytest
import torch

from paper_2405_01834_gb300 import inputs, mdx

pytestmark = pytest.mark.gpu


def _batches(eng):
    """One batch over two such classes, more quartets than the GPU holds blocks in the first, and one of another
    class: their areas have different sizes."""
    b1, q1 = inputs.class_sweep((6, 6, 6, 6), n_bra=16, n_ket=12, seed=31)
    b2, q2 = inputs.class_sweep((5, 5, 5, 5), n_bra=20, n_ket=11, seed=32)
    return [eng.batch_eri4(mdx.DeviceBasis(b), q) for b, q in ((b2, q2), (b1, q1))]


def _out(B):
    return torch.full((B.total,), float("nan"), dtype=torch.float64, device="cuda")


def test_runs_on_several_streams():
    """Each batch on three streams at once, into its own output every time: the bits of a run by itself."""
    eng = mdx.Engine(0)
    Bs = _batches(eng)
    want = []
    for B in Bs:
        o = _out(B)
        B.run(o)
        torch.cuda.synchronize()
        want.append(o)
    streams = [torch.cuda.Stream() for _ in range(3)]
    outs = [[_out(B) for _ in streams] for B in Bs]
    torch.cuda.synchronize()
    for i, s in enumerate(streams):
        with torch.cuda.stream(s):
            for j in range(len(Bs)):
                k = (i + j) % len(Bs)
                Bs[k].run(outs[k][i])
    torch.cuda.synchronize()
    for w, os in zip(want, outs):
        for o in os:
            assert torch.equal(o, w)
    eng.sync()
    for B in Bs:
        B.close()
    eng.close()


def test_captured_runs_replayed_side_by_side():
    eng = mdx.Engine(0)
    B = _batches(eng)[1]
    want = _out(B)
    B.run(want)
    outs, graphs = [_out(B) for _ in range(3)], [torch.cuda.CUDAGraph() for _ in range(3)]
    streams = [torch.cuda.Stream() for _ in range(3)]
    torch.cuda.synchronize()
    for g, o, s in zip(graphs, outs, streams):
        with torch.cuda.stream(s):
            with torch.cuda.graph(g, stream=s):
                B.run(o)
    torch.cuda.synchronize()
    for _ in range(2):
        for g, s in zip(graphs, streams):
            with torch.cuda.stream(s):
                g.replay()
    torch.cuda.synchronize()
    for o in outs:
        assert torch.equal(o, want)
    eng.sync()
    B.close()
    eng.close()


def test_areas_are_shared_and_given_back():
    """The batches of an engine share one set of areas (152 x 749 KB for [ii|ii]), whichever of them is closed, and the
    engine gives it back."""
    eng = mdx.Engine(0)
    b, q = inputs.class_sweep((6, 6, 6, 6), n_bra=1, n_ket=1, seed=31)
    db = mdx.DeviceBasis(b)
    free = lambda: torch.cuda.mem_get_info()[0]  # noqa: E731
    area = 152 * 749112
    torch.cuda.synchronize()
    before = free()
    first = eng.batch_eri4(db, q)
    used = before - free()
    assert used >= area
    more = [eng.batch_eri4(db, q) for _ in range(8)]
    assert before - free() < used + area // 2
    first.close()
    o = _out(more[0])
    more[0].run(o)
    eng.sync()
    assert torch.isfinite(o).all()
    for x in more:
        x.close()
    B = eng.batch_eri4(db, q)
    assert before - free() < used + area // 2
    B.close()
    eng.close()
    assert before - free() < area // 2
