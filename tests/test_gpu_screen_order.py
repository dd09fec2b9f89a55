"""The list of mdx_exchange_screen: groups of one class pair, of the shells in index order, the higher class as bra."""
import numpy as np
import pytest
import torch

from paper_2405_01834_gb300 import inputs, mdx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shells", [(0, 1, 2), (2, 0, 1)])
def test_kept_list_is_grouped_by_class_pair(shells):
    b = inputs.small_molecule(seed=87, n_atoms=3, shells=shells, K=2)
    pairs = np.array([(j, i) if (i + j) % 2 else (i, j) for i in range(b.n_shells) for j in range(i + 1)], dtype=np.int32)
    eng, db = mdx.Engine(0), mdx.DeviceBasis(b)
    D = torch.from_numpy(inputs.density(b.nao, 7))
    kept, n, _ = eng.exchange_screen(db, pairs, eng.schwarz(db, pairs), D, 1e-10)
    eng.sync()
    cls = [(int(b.l[max(p)]), int(b.l[min(p)]), int(b.nprim[p[0]] * b.nprim[p[1]])) for p in pairs]
    rows = [(cls[x], cls[y]) for x, y in kept.cpu().numpy()]
    assert n == len(rows) > 0
    assert all(x >= y for x, y in rows)
    assert rows == sorted(rows)   # one contiguous group per class pair
    eng.close()
