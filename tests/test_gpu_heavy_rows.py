"""The kernels of the heavy rows (rank with and without parts, direct, packed counters of dense binary rows) at the
sizes where they can go wrong, against the CPU oracle: structure and int32 values exact, fp64 within 1e-12 and fp32 within
1e-5 of the sum of absolute partial products (the bars of the parity tests)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2608_09713_b200 import workloads as W
from test_gpu_parity import B, check_values, dev, run_and_compare  # noqa: F401  (B is the fixture)

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
def test_long_rows_of_several_blocks(B, m, dtype):
    """Rows of 300 and of 600 nonzeros (one and two batches of lists) over columns of hundreds of entries: one to three blocks
    of 8192 columns, no more entries than the slots hold."""
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


def cut_matrix(dtype):
    """60000 rows of six nonzeros; rows of 200 and 600 nonzeros have about 40000 and 59000 entries: two parts of the rank
    kernel with doubles (24576 slots), one or two with int32 (51200), in the lower triangle near the end and in the
    upper parts of the full output near the beginning."""
    m, n = 60000, 1200
    rng = np.random.default_rng(11)
    cols = rng.integers(0, n, (m, 6))
    pairs = [(i, cols[i]) for i in range(m)]
    long = {50: 600, 51: 200, 30000: 600, 40000: 600, 40001: 200, m - 3: 200, m - 2: 600, m - 1: 600}
    return matrix(m, n, [(i, rng.choice(n, long[i], replace=False) if i in long else c) for i, c in pairs], dtype), sorted(long)


@pytest.mark.parametrize("dtype", [np.float64, np.float32, np.int32])
@pytest.mark.parametrize("mode", [0, 1])
def test_long_rows_in_parts(B, dtype, mode):
    a, long = cut_matrix(dtype)
    (rp, ci, cv), ref, plan = run_and_compare(B, a, mode)
    counts = (rp[1:] - rp[:-1])[torch.tensor(long, device="cuda")]
    assert int((counts > 51200).sum()) >= 2  # more than any route's slots
    ranges = [0, 50, 51, 30000, 40000, 40001, 40002, a.m - 2, a.m - 1, a.m]
    c2, v2 = torch.full_like(ci, -1), torch.zeros_like(cv)
    order = [3, 0, 8, 1, 5, 2, 7, 4, 6]
    for b in order:
        B.spsyrk_numeric_rows(plan, ranges[b], ranges[b + 1], rp, c2, v2)
        written = c2 >= 0
        s0, e0 = int(rp[ranges[b]]), int(rp[ranges[b + 1]])
        assert bool(written[s0:e0].all()) and int(written.sum()) == sum(int(rp[ranges[x + 1]] - rp[ranges[x]]) for x in order[: order.index(b) + 1])
    assert torch.equal(c2, ci)
    check_values(v2.cpu().numpy(), ref, a.vals.dtype)
    if mode == 0:
        B.spsyrk_plan_lend_map(plan, None)
        rp1, ci1, cv1 = B.onepass_syrk(plan)
        assert torch.equal(rp1, rp) and torch.equal(ci1, ci)
        check_values(cv1.cpu().numpy(), ref, a.vals.dtype)


@pytest.mark.parametrize("dtype", [np.float64, np.float32, np.int32])
def test_long_dense_binary_rows(B, dtype):
    """Dense rows of a binary matrix with more than 255 nonzeros over a range of several chunks of the direct kernel."""
    m, n = 26000, 3000
    rng = np.random.default_rng(12)
    pairs = [(i, np.concatenate([[0], rng.integers(1, n, 2)])) for i in range(m)]
    for i in (11000, 13000, m - 2, m - 1):
        pairs[i] = (i, np.concatenate([[0], 1 + rng.choice(n - 1, 299, replace=False)]))
    a = matrix(m, n, pairs, dtype, ones=True)
    rows = np.array([0, 5000, 11000, 13000, m - 3, m - 2, m - 1])
    c_rowptr, c_colidx, c_vals, plan = B.tril_syrk(a.m, a.n, *dev(a))
    assert torch.equal(c_rowptr, torch.arange(m + 1, device="cuda") * torch.arange(1, m + 2, device="cuda") // 2)
    cols = oracle.transpose(a.m, a.n, a.rowptr, a.colidx, a.vals)
    for i in rows:
        ref = oracle.syrk(a.m, a.n, a.rowptr, a.colidx, a.vals, oracle.TRIL, int(i), int(i) + 1, cols=cols)
        s, e = int(c_rowptr[i]), int(c_rowptr[i + 1])
        assert np.array_equal(c_colidx[s:e].cpu().numpy(), ref.colidx)
        assert np.array_equal(c_vals[s:e].cpu().numpy().astype(np.float64), ref.vals)


def test_row_ranges_launch_what_they_hold(B):
    """A row range without heavy rows launches no kernel of theirs, a range with one such row one."""
    m, n = 5000, 4000
    rng = np.random.default_rng(13)
    pairs = [(i, rng.choice(n, 40 + i % 300, replace=False)) for i in range(2000, m, 2)]
    a = matrix(m, n, pairs, np.float64)
    rp, ci, cv, plan = B.tril_syrk(a.m, a.n, *dev(a))
    heavy = [i for i in range(m) if a.rowptr[i + 1] - a.rowptr[i] > 32]
    light_kernels = 5  # one per class of light rows, at most

    def launches(r0, r1):
        before = B.spsyrk_launch_count()
        B.spsyrk_numeric_rows(plan, r0, r1, rp, ci, cv)
        return B.spsyrk_launch_count() - before

    assert launches(0, heavy[0]) <= 1 + light_kernels
    assert launches(heavy[7], heavy[7] + 1) == 2
    assert launches(heavy[-1] - 1, heavy[-1]) <= 2
