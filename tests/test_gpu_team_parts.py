"""Teams that share a quartet's primitive pairs where its shellset is digested or contracted, not stored: exchange and
gradient of a few contracted shells of high angular momentum, against the oracle."""
import ctypes
import os
import subprocess

import numpy as np
import pytest
import torch

import oracle
from paper_2405_01834_gb300 import inputs, mdx

pytestmark = pytest.mark.gpu

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2405_01834_gb300", "csrc")
SHIM = """
#include "mdx_internal.h"
extern "C" int parts(int la, int lb, int lc, int ld, int Kb, int Kk, long long nq, int concurrent) {
  mdx::Plan p;
  std::string err;
  if (!mdx::build_plan(mdx::ClassKey{la, lb, lc, ld, Kb, Kk, 0, 0}, mdx::PlanConfig{}, p, err) || p.d.reg) return -1;
  int nb = 0, nk = 0;
  mdx::team_parts(p.d, nq, concurrent, false, &nb, &nk);
  return nb * nk;
}
"""
STREAMS = 8   # launches of a call that can run side by side


@pytest.fixture(scope="module")
def parts(tmp_path_factory):
    d = tmp_path_factory.mktemp("parts")
    (d / "shim.cpp").write_text(SHIM)
    so = str(d / "shim.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(d / "shim.cpp")] +
                   [os.path.join(CSRC, f) for f in ("plan.cpp", "boys_table.cpp", "solid.cpp")] + ["-o", so], check=True)
    lib = ctypes.CDLL(so)
    lib.parts.argtypes = [ctypes.c_int] * 6 + [ctypes.c_longlong, ctypes.c_int]
    return lib.parts


# one class of shells, so that the class and the number of quartets of each launch are known: n (n + 1) / 2 pairs
CASES = [(2, 3, 2), (2, 5, 1), (3, 2, 2), (4, 2, 1)]   # l, K, atoms


def _inputs(l, K, atoms):
    b = inputs.small_molecule(seed=91, n_atoms=atoms, shells=(l,), K=K)
    pairs = np.array([(i, j) for i in range(b.n_shells) for j in range(i + 1)], dtype=np.int32)
    return b, pairs, inputs.density(b.nao, 15, occ_fraction=0.4)


@pytest.mark.parametrize("l,K,atoms", CASES)
def test_exchange(parts, l, K, atoms):
    b, pairs, D = _inputs(l, K, atoms)
    nq = len(pairs) * (len(pairs) + 1) // 2
    assert parts(l, l, l, l, K * K, K * K, nq, 1) > 1
    eng, db = mdx.Engine(0), mdx.DeviceBasis(b)
    got = eng.exchange(db, pairs, eng.schwarz(db, pairs), torch.from_numpy(D), 0.0).cpu().numpy()
    assert eng.last_quartet_count() == nq
    ref = oracle.exchange(b, D)
    np.testing.assert_allclose(got, ref, rtol=0, atol=1e-12 * np.max(np.abs(ref)))
    eng.close()


@pytest.mark.parametrize("l,K,atoms", [c for c in CASES if c[2] > 1])
def test_gradient(parts, l, K, atoms):
    b, pairs, D = _inputs(l, K, atoms)
    nq = len(pairs) * (len(pairs) + 1) // 2
    assert parts(l + 1, l, l, l, K * K, K * K, nq, STREAMS) > 1
    eng, db = mdx.Engine(0), mdx.DeviceBasis(b)
    g, e = eng.exchange_grad(db, pairs, eng.schwarz(db, pairs), torch.from_numpy(D), tau=0.0, n_atoms=b.n_atoms)
    ref, eref = -oracle.exchange_grad(b, D), -oracle.exchange_energy(b, D)
    np.testing.assert_allclose(g.cpu().numpy(), ref, rtol=0, atol=1e-11 * max(np.max(np.abs(ref)), 1e-3))
    assert abs(float(e) - eref) <= 1e-11 * abs(eref)
    eng.close()
