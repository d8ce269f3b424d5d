"""Rows that the plan treats apart: long ones (left to a warp or the whole CTA) and dense ones (their counts are settled without
a counting kernel)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2608_09713_b200 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2608_09713_b200 import binding
    return binding


def _matrix(lengths, n, seed, full_column=False, empty=()):
    rng = np.random.default_rng(seed)
    rows = []
    for i, d in enumerate(lengths):
        r = np.sort(rng.choice(n, d, replace=False))
        if full_column and i not in empty and (r.size == 0 or r[0] != 0):
            r = np.concatenate(([0], r))
        rows.append(r.astype(np.int32))
    rp = np.concatenate(([0], np.cumsum([r.size for r in rows]))).astype(np.int64)
    return W.CSR(len(rows), n, rp, np.concatenate(rows), rng.standard_normal(rp[-1]))


def _check(a, ref, out):
    rp, ci, cv = (t.cpu().numpy() for t in out)
    assert np.array_equal(rp, ref.rowptr) and np.array_equal(ci, ref.colidx)
    assert np.all(np.abs(cv - ref.vals) <= 1e-12 * ref.absvals)


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("average", [2, 7, 14, 30])  # 4, 8, 16 and 32 lanes per row
def test_long_rows_among_short_ones(B, average, mode):
    g = 4 if average <= 4 else 8 if average <= 8 else 16 if average <= 16 else 32
    edges = [8 * g - 1, 8 * g, 8 * g + 1, 1023, 1024, 1025, 4000]
    crowd = [8 * g + 5] * 300  # long rows only: a CTA's whole tile of them
    short = (sum(edges) + sum(crowd)) * 2 // average
    lengths = [average // 2] * (short // 2) + edges + [average // 2] * (short // 2) + crowd
    a = _matrix(lengths, 60_000, average)
    d = (torch.from_numpy(a.rowptr).cuda(), torch.from_numpy(a.colidx).cuda(), torch.from_numpy(a.vals).cuda())
    rp, ci, cv, plan = B.tril_syrk(a.m, a.n, *d, mode=mode)
    ref = oracle.syrk(a.m, a.n, a.rowptr, a.colidx, a.vals, mode)
    _check(a, ref, (rp, ci, cv))
    assert B.spsyrk_plan_stats(plan)[0] == int(ref.work.sum())
    assert np.array_equal(B.spsyrk_plan_buffers(plan)[3].cpu().numpy(), oracle.syrk(a.m, a.n, a.rowptr, a.colidx, a.vals, 0, counts_only=True).work) or mode


@pytest.mark.parametrize("rows", [500, 9000])  # 9000: rows beyond a block of 8192 columns
@pytest.mark.parametrize("empty", [(), (3, 100)], ids=["all dense", "not all"])
def test_dense_rows(B, rows, empty):
    a = _matrix([40 if i not in empty else 0 for i in range(rows)], 300, 5, full_column=True, empty=empty)
    d = (torch.from_numpy(a.rowptr).cuda(), torch.from_numpy(a.colidx).cuda(), torch.from_numpy(a.vals).cuda())
    whole = oracle.syrk(a.m, a.n, a.rowptr, a.colidx, a.vals, 0) if rows == 500 else None
    plan = B.spsyrk_plan(a.m, a.n, *d)
    for r0, r1 in ((0, rows), (rows - 150, rows - 20), (0, 5)):  # the same plan for several ranges
        B.spsyrk_plan_set_rows(plan, r0, r1)
        ref = oracle.syrk(a.m, a.n, a.rowptr, a.colidx, a.vals, 0, r0, r1) if (r0, r1) != (0, rows) or whole is None else whole
        for _ in range(2):  # the counting pass again on the same binning
            rp = torch.empty(r1 - r0 + 1, dtype=torch.int64, device="cuda")
            nnz = B.spsyrk_symbolic(plan, rp)
            ci, cv = torch.empty(nnz, dtype=torch.int32, device="cuda"), torch.empty(nnz, dtype=torch.float64, device="cuda")
            B.spsyrk_numeric(plan, rp, ci, cv)
            _check(a, ref, (rp, ci, cv))
    B.spsyrk_plan_set_block(plan, rows - 100, rows, 50, rows - 60)  # a narrowed range of columns
    ref = oracle.syrk(a.m, a.n, a.rowptr, a.colidx, a.vals, 0, rows - 100, rows)
    rp = torch.empty(101, dtype=torch.int64, device="cuda")
    nnz = B.spsyrk_symbolic(plan, rp)
    ci, cv = torch.empty(nnz, dtype=torch.int32, device="cuda"), torch.empty(nnz, dtype=torch.float64, device="cuda")
    B.spsyrk_numeric(plan, rp, ci, cv)
    keep = (ref.colidx >= 50) & (ref.colidx < rows - 60)
    row_of = np.repeat(np.arange(100), np.diff(ref.rowptr))[keep]
    assert np.array_equal(rp.cpu().numpy(), np.concatenate(([0], np.cumsum(np.bincount(row_of, minlength=100)))))
    assert np.array_equal(ci.cpu().numpy(), ref.colidx[keep])
    assert np.all(np.abs(cv.cpu().numpy() - ref.vals[keep]) <= 1e-12 * ref.absvals[keep])
