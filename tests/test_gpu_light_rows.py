"""Light rows ordered by buckets of their columns: columns spread out, close together, and both in turn."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2608_09713_b200 import binding
    return binding


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("spread", [0.0, 0.5, 1.0])  # share of the rows whose columns go anywhere
@pytest.mark.parametrize("items", [40, 100, 180, 400])  # products of a row: all classes of light rows
def test_columns_spread_and_close(B, items, spread, mode):
    rng = np.random.default_rng(items)
    m, d = 3000, 12
    n = max(int(m * d * d / items), 64)
    rows = []
    for i in range(m):
        if rng.random() < spread:
            r = rng.choice(n, d, replace=False)
        else:  # the columns of a row and its neighbours: the products' columns stand together
            r = (i * n // m + rng.choice(4 * d, d, replace=False)) % n
        rows.append(np.unique(r).astype(np.int32))
    rp = np.concatenate(([0], np.cumsum([r.size for r in rows]))).astype(np.int64)
    ci, v = np.concatenate(rows), rng.standard_normal(rp[-1])
    got = [t.cpu().numpy() for t in B.tril_syrk(m, n, *(torch.from_numpy(t).cuda() for t in (rp, ci, v)), mode=mode)[:3]]
    ref = oracle.syrk(m, n, rp, ci, v, mode)
    assert np.array_equal(got[0], ref.rowptr) and np.array_equal(got[1], ref.colidx)
    assert np.all(np.abs(got[2] - ref.vals) <= 1e-13 * ref.absvals)  # a few hundred terms at most, a rounding of 1.1e-16 each
