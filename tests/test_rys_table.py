"""The library's Rys nodes and weights (host-built table) against the moments they must reproduce:
sum_r w_r x_r^k = F_k(T) for k <= 2n - 1, with the oracle's long-double Boys function."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import oracle

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2405_01834_gb300", "csrc")
SHIM = """
#include "mdx_internal.h"
extern "C" {
long long rys_size() { return (long long)mdx::rys_table().size(); }
const double* rys_data() { return mdx::rys_table().data(); }
long long rys_first(int n) { return mdx::rys_offset(n); }
int rys_terms() { return mdx::kRysTerms; }
int rys_intervals() { return mdx::kRysIntervals; }
int rys_max() { return mdx::kRysMax; }
}
"""


@pytest.fixture(scope="module")
def table(tmp_path_factory):
    d = tmp_path_factory.mktemp("rys")
    (d / "shim.cpp").write_text(SHIM)
    so = str(d / "shim.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(d / "shim.cpp"),
                    os.path.join(CSRC, "rys_table.cpp"), "-o", so, "-lpthread"], check=True)
    lib = ctypes.CDLL(so)
    lib.rys_size.restype = lib.rys_first.restype = ctypes.c_longlong
    lib.rys_data.restype = ctypes.POINTER(ctypes.c_double)
    tab = np.ctypeslib.as_array(lib.rys_data(), (lib.rys_size(),)).copy()
    return tab, lib


def _rule(table, n, T):
    """Nodes and weights the way the kernel forms them."""
    tab, lib = table
    C, I, o = lib.rys_terms(), lib.rys_intervals(), lib.rys_first(n)
    if T < I:
        i = int(T)
        c = tab[o + i * C * 2 * n: o + (i + 1) * C * 2 * n].reshape(C, 2 * n)
        f = c[-1].copy()
        for k in range(C - 2, -1, -1):
            f = f * (T - (i + 0.5)) + c[k]
        return f[:n], f[n:]
    c = tab[o + I * C * 2 * n: o + I * C * 2 * n + 2 * n]
    return c[:n] / T, c[n:] / np.sqrt(T)


@pytest.mark.parametrize("n", range(1, 14))
def test_rys_moments(table, n):
    assert n <= table[1].rys_max()
    rng = np.random.default_rng(n)
    Ts = np.concatenate([[0.0, 1e-10, 0.5, 1.0 - 1e-15, 1.0, 37.0, 99.0, 100.0 - 1e-13], rng.uniform(0.0, 100.0, 60),
                         [100.0, 133.7, 1e4]])
    for T in Ts:
        x, w = _rule(table, n, float(T))
        assert (x > 0).all() and (x < 1).all() and (w > 0).all() and (np.diff(x) > 0).all()
        F = oracle.boys(2 * n - 1, float(T), precision=1)
        for k in range(2 * n):
            # node and weight to one rounding of their value and of the Horner steps (2 ulp), k + 1 factors in
            # a sum of positive terms, and its own rounding
            assert abs((w * x ** k).sum() / F[k] - 1.0) <= (2 * k + 6) * 2.3e-16, (n, T, k)
