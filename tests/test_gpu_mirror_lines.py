"""The mirror on both sides of the lines between its sorts, and rows copied by pieces of entries."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2608_09713_b200 import binding
    return binding


def _check(B, m, rowptr, colidx, dtype, seed):
    vals = np.random.default_rng(seed).standard_normal(colidx.size)
    vals = vals.astype(np.float32) if dtype == torch.float32 else vals
    got = [t.cpu().numpy() for t in B.spsyrk_mirror(m, *(torch.from_numpy(t).cuda() for t in (rowptr, colidx, vals)))]
    ref = oracle.mirror(m, rowptr, colidx, vals.astype(np.float64))
    assert np.array_equal(got[0], ref[0]) and np.array_equal(got[1], ref[1]) and np.array_equal(got[2].astype(np.float64), ref[2])


def _csr(m, rows, cols):
    code = np.unique(rows.astype(np.int64) * m + cols)
    rowptr = np.searchsorted(code // m, np.arange(m + 1)).astype(np.int64)
    return rowptr, (code % m).astype(np.int32)


@pytest.mark.parametrize("kind", ["random", "one column", "few"])
@pytest.mark.parametrize("m", [65536, 65537, 262_144, 262_145])
def test_double_precision_by_rows(B, m, kind):
    rng = np.random.default_rng(m)
    if kind == "few":
        rows = rng.integers(0, m, 500)
    elif kind == "one column":  # most rows store column 7, and every 512th column is crowded
        rows = np.concatenate((np.arange(7, m), rng.integers(0, m, 3 * m)))
    else:
        rows = rng.integers(0, m, 6 * m)
    cols = (rng.random(rows.size) * (rows + 1)).astype(np.int64)
    if kind == "one column":
        cols[:m - 7] = 7
        cols[m - 7:] = cols[m - 7:] // 512 * 512
    _check(B, m, *_csr(m, rows, cols), torch.float64, 3)


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("m", [1000, 2111])
def test_long_rows_and_gaps(B, m, dtype):
    """More than 256 entries per row on average: rows of every length, empty ones singly, in dozens and by the hundred."""
    rng = np.random.default_rng(m)
    full = [np.arange(i + 1) if rng.random() < 0.7 else np.sort(rng.choice(i + 1, rng.integers(0, min(i + 1, 40)), replace=False)) for i in range(m)]
    for lo, hi in ((5, 6), (m // 2, m // 2 + 31), (m // 2 + 40, m // 2 + 73), (m - 400, m - 250)):
        full[lo:hi] = [np.zeros(0, dtype=np.int64)] * (hi - lo)
    rowptr = np.concatenate(([0], np.cumsum([r.size for r in full]))).astype(np.int64)
    assert m != 2111 or rowptr[-1] // m >= 256
    _check(B, m, rowptr, np.concatenate(full).astype(np.int32), dtype, 4)
