"""Pairs whose shells share a centre: the Hermite expansion has no terms of the wrong parity, however large the
coordinates. Shells far from the origin and 6 to 10 bohr from each other, where such a term would show the charge
instead of a multipole."""
import numpy as np
import pytest
import torch

import oracle
from paper_2405_01834_gb300 import inputs, mdx

pytestmark = pytest.mark.gpu
# Relative to the shellset's largest integral. The integrals are sums of some dozens of terms without cancellation
# (about 60 roundings of 1.1e-16 if all had one sign); an ulp of P - A (1.4e-14 at these coordinates) times twice an
# exponent and the distance would be 1e-13 and more.
TOL = 1e-14


def _check(got, ref, off):
    for i in range(len(off) - 1):
        r = ref[off[i]: off[i + 1]]
        e = np.abs(got[off[i]: off[i + 1]] - r).max() / np.abs(r).max()
        assert e < TOL, (i, e)


@pytest.mark.parametrize("la,lc,ld", [(3, 2, 2), (5, 2, 2), (5, 3, 2), (1, 3, 2), (1, 2, 2), (1, 1, 0), (3, 1, 1)])
def test_one_centre_bra(la, lc, ld):
    rng = np.random.default_rng(5)
    aux, orb, t = inputs.BasisBuilder(), inputs.BasisBuilder(), []
    for i in range(40):
        C = rng.uniform(60.0, 120.0, 3)
        u = rng.normal(size=3)
        A = C + u / np.linalg.norm(u) * rng.uniform(6.0, 10.0)
        aux.add_shell(la, A, [rng.uniform(2.0, 6.0)], [1.0])
        for l in (lc, ld):
            orb.add_shell(l, C, [rng.uniform(1.0, 3.0)], [1.0])
        t.append((i, 2 * i, 2 * i + 1))
    aux, orb, t = aux.build(), orb.build(), np.array(t, dtype=np.int32)
    eng = mdx.Engine(0)
    v, _ = eng.eri3(mdx.DeviceBasis(aux), mdx.DeviceBasis(orb), t)
    eng.sync()
    ref, off = oracle.eri3(aux, orb, t, precision=1)
    _check(v.cpu().numpy(), ref, off)
    eng.close()


@pytest.mark.parametrize("lq,K", [((0, 0, 1, 0), (1, 1, 3, 3)), ((1, 1, 1, 0), (2, 1, 3, 6)), ((2, 1, 1, 0), (3, 3, 3, 3))])
def test_concentric_contracted_kets(lq, K):
    rng = np.random.default_rng(6)
    n = 170   # one lane per quartet: the register kernel sums the kets
    bb = inputs.BasisBuilder()
    C = rng.uniform(60.0, 64.0, 3)
    u = rng.normal(size=3)
    A = C + u / np.linalg.norm(u) * 9.0
    for _ in range(n):
        for l, k in zip(lq[:2], K[:2]):
            bb.add_shell(l, A, rng.uniform(1.0, 3.0, k), [1.0] * k)
    for _ in range(n):
        for l, k in zip(lq[2:], K[2:]):
            bb.add_shell(l, C, rng.uniform(1.0, 3.0, k), [1.0] * k)
    b = bb.build()
    q = np.array([(2 * i, 2 * i + 1, 2 * n + 2 * j, 2 * n + 2 * j + 1) for j in range(n) for i in range(n)], dtype=np.int32)
    eng = mdx.Engine(0)
    v, off = eng.eri4(mdx.DeviceBasis(b), q)
    eng.sync()
    sel = np.arange(0, len(q), 97)
    ref, roff = oracle.eri4(b, q[sel], precision=1)
    v, off = v.cpu().numpy(), off.cpu().numpy()
    _check(np.concatenate([v[off[i]: off[i + 1]] for i in sel]), ref, roff)
    eng.close()
