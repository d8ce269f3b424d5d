"""The kernels of the heavy rows (rank, direct with and without parts, packed counters of dense binary rows) at the
sizes where they can go wrong, against the CPU oracle: structure and int32 values exact, fp64 within 1e-12 and fp32 within
1e-5 of the sum of absolute partial products (the bars of the parity tests)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2608_09713_b200 import workloads as W
from test_gpu_parity import B, dev, run_and_compare  # noqa: F401  (B is the fixture)

pytestmark = pytest.mark.gpu


def matrix(m, n, rows_cols, dtype, seed=3, ones=False):
    """CSR from a list of (row, columns) pairs plus one nonzero in every other row."""
    cols = {i: np.unique(c) for i, c in rows_cols}
    for i in range(m):
        cols.setdefault(i, np.array([(i * 7919) % n]))
    rowptr = np.zeros(m + 1, dtype=np.int64)
    np.cumsum([cols[i].size for i in range(m)], out=rowptr[1:])
    colidx = np.concatenate([cols[i] for i in range(m)]).astype(np.int32)
    rng = np.random.default_rng(seed)
    vals = np.ones(colidx.size) if ones else rng.integers(1, 9, colidx.size) if dtype == np.int32 else rng.uniform(-1, 1, colidx.size)
    return W.CSR(m, n, rowptr, colidx, vals.astype(dtype))


@pytest.mark.parametrize("dtype", [np.float64, np.float32, np.int32])
@pytest.mark.parametrize("m", [8191, 8193, 20000])
def test_long_rows_in_parts(B, m, dtype):
    """Rows of 300 and of 600 nonzeros (one and two batches of lists) over columns of hundreds of entries: several chunks of
    8192 columns, cut into parts (20000 rows) or not."""
    rng = np.random.default_rng(m)
    n = 700
    pairs = [(i, rng.choice(n, 40, replace=False)) for i in range(0, m, 2)]
    pairs += [(m - 1, rng.choice(n, 600, replace=False)), (m - 2, rng.choice(n, 300, replace=False)), (m // 2, rng.choice(n, 513, replace=False))]
    run_and_compare(B, matrix(m, n, pairs, dtype), 0)


@pytest.mark.parametrize("dtype", [np.float64, np.int32])
def test_sparse_rows_by_entries_and_range(B, dtype):
    """Rank kernels: last rows with 33 to 5000 nonzeros of nearly private columns, entries on both sides of the slot
    counts; ranges on both sides of the narrower bitmaps (65536, 131072 columns) and beyond one chunk (262144)."""
    m, n = 270000, 400000
    rng = np.random.default_rng(5)
    pairs = []
    for i in (65535, 65536, 131071, 131072, 262143, 262144, m - 1):
        pairs.append((i, rng.choice(n, 700, replace=False)))
    for i, d in ((200000, 33), (200001, 4000), (200002, 20000)):
        pairs.append((i, rng.choice(n, d, replace=False)))
    a = matrix(m, n, pairs, dtype)
    rows = np.array([i for i, _ in pairs])
    c_rowptr, c_colidx, c_vals, plan = B.tril_syrk(a.m, a.n, *dev(a))
    cols = oracle.transpose(a.m, a.n, a.rowptr, a.colidx, a.vals)
    rp = c_rowptr.cpu().numpy()
    for i in rows:
        ref = oracle.syrk(a.m, a.n, a.rowptr, a.colidx, a.vals, oracle.TRIL, int(i), int(i) + 1, cols=cols)
        s, e = int(rp[i]), int(rp[i + 1])
        assert np.array_equal(c_colidx[s:e].cpu().numpy(), ref.colidx), i
        got = c_vals[s:e].cpu().numpy()
        if dtype == np.int32:
            assert np.array_equal(got, oracle.to_int32(ref.vals))
        else:
            assert np.all(np.abs(got - ref.vals) <= 1e-12 * ref.absvals)


@pytest.mark.parametrize("dtype", [np.int32, np.float32, np.float64])
@pytest.mark.parametrize("deg", [255, 256])
def test_dense_binary_rows(B, dtype, deg):
    """Every row stores column 0: all rows are dense.  At most 255 nonzeros take the packed counters, more do not; the
    output may start anywhere (rows begin at i (i + 1) / 2, and the arrays here one element past an aligned address)."""
    m, n = 1003, 4000
    rng = np.random.default_rng(deg)
    pairs = [(i, np.concatenate([[0], 1 + rng.choice(n - 1, deg - 1, replace=False, p=None)])) for i in range(m)]
    a = matrix(m, n, pairs, dtype, ones=True)
    (rp, ci, cv), ref, plan = run_and_compare(B, a, 0)
    shift_ci = torch.full((ci.numel() + 1,), -1, dtype=torch.int32, device="cuda")[1:]
    shift_cv = torch.zeros(cv.numel() + 1, dtype=cv.dtype, device="cuda")[1:]
    B.spsyrk_numeric(plan, rp, shift_ci, shift_cv)
    assert torch.equal(shift_ci, ci) and torch.equal(shift_cv, cv)
    if dtype == np.int32:
        jac = torch.full((cv.numel() + 1,), -1.0, dtype=torch.float32, device="cuda")
        for out in (jac[1:], jac[:-1]):
            B.spsyrk_plan_set_jaccard(plan, out)
            B.spsyrk_numeric(plan, rp, ci, cv)
            exp = oracle.jaccard(0, m, a.rowptr, ref.rowptr, ref.colidx, oracle.to_int32(ref.vals))
            assert np.array_equal(out.cpu().numpy(), exp.astype(np.float32))
