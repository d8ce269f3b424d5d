"""Rows of binary matrices that are full in part: counted and computed through the masks of the heaviest columns."""
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


def _sets(m, n, d, seed):
    """Sets of about d of n columns, the low ones in most sets but none in all; some sets empty, some of more than 255 columns."""
    rng = np.random.default_rng(seed)
    rows = []
    for i in range(m):
        k = 0 if i % 97 == 5 else min(n, 300) if i % 101 == 7 else d
        r = np.unique((n * rng.random(k) ** 3).astype(np.int32))
        rows.append(r[r != i % 40])
    rp = np.concatenate(([0], np.cumsum([r.size for r in rows]))).astype(np.int64)
    return rp, np.concatenate(rows).astype(np.int32)


def _run(B, plan, rows, dtype, jaccard):
    rp = torch.empty(rows + 1, dtype=torch.int64, device="cuda")
    nnz = B.spsyrk_symbolic(plan, rp)
    ci, cv = torch.empty(nnz, dtype=torch.int32, device="cuda"), torch.empty(nnz, dtype=dtype, device="cuda")
    jac = torch.empty(nnz, dtype=torch.float32, device="cuda") if jaccard else None
    if jaccard:
        B.spsyrk_plan_set_jaccard(plan, jac)
    B.spsyrk_numeric(plan, rp, ci, cv)
    return tuple(t.cpu().numpy() if t is not None else None for t in (rp, ci, cv, jac))


@pytest.mark.parametrize("dtype", [torch.int32, torch.float32, torch.float64])
@pytest.mark.parametrize("m,n,d", [(300, 400, 30), (1500, 900, 24), (2051, 3000, 40), (4099, 500, 12), (9001, 40_000, 14)])
def test_partly_full_rows(B, m, n, d, dtype):
    rp, ci = _sets(m, n, d, m)
    npdt = {torch.int32: np.int32, torch.float32: np.float32, torch.float64: np.float64}[dtype]
    dev = (torch.from_numpy(rp).cuda(), torch.from_numpy(ci).cuda(), torch.ones(ci.size, dtype=dtype, device="cuda"))
    ref = oracle.syrk(m, n, rp, ci, np.ones(ci.size, dtype=npdt), oracle.TRIL)
    jaccard = dtype == torch.int32
    plan = B.spsyrk_plan(m, n, *dev)
    got = _run(B, plan, m, dtype, jaccard)
    assert np.array_equal(got[0], ref.rowptr) and np.array_equal(got[1], ref.colidx)
    assert np.array_equal(got[2].astype(np.float64), ref.vals)  # whole numbers
    if jaccard:
        exp = oracle.jaccard(0, m, rp, ref.rowptr, ref.colidx, oracle.to_int32(ref.vals))
        assert np.array_equal(got[3], exp.astype(np.float32)) or np.all(np.abs(got[3] - exp) <= 1e-7 * exp)
        return
    # the same plan for a range of rows, then for a block whose columns are a part of the triangle (no masks there)
    r0, r1, s0, s1 = m // 3, m - 7, m // 5, m // 2
    B.spsyrk_plan_set_rows(plan, r0, r1)
    got = _run(B, plan, r1 - r0, dtype, False)
    part = slice(ref.rowptr[r0], ref.rowptr[r1])
    assert np.array_equal(got[0], ref.rowptr[r0:r1 + 1] - ref.rowptr[r0])
    assert np.array_equal(got[1], ref.colidx[part]) and np.array_equal(got[2].astype(np.float64), ref.vals[part])
    B.spsyrk_plan_set_block(plan, r0, r1, s0, s1)
    got = _run(B, plan, r1 - r0, dtype, False)
    keep = (ref.colidx[part] >= s0) & (ref.colidx[part] < s1)
    assert np.array_equal(got[1], ref.colidx[part][keep]) and np.array_equal(got[2].astype(np.float64), ref.vals[part][keep])


@pytest.mark.parametrize("m,n,d", [(1500, 900, 24), (4099, 500, 12)])
def test_partly_full_rows_both_triangles(B, m, n, d):
    rp, ci = _sets(m, n, d, m)
    dev = (torch.from_numpy(rp).cuda(), torch.from_numpy(ci).cuda(), torch.ones(ci.size, dtype=torch.float64, device="cuda"))
    ref = oracle.syrk(m, n, rp, ci, np.ones(ci.size), oracle.FULL)
    got = [t.cpu().numpy() for t in B.tril_syrk(m, n, *dev, mode=B.FULL)[:3]]
    assert np.array_equal(got[0], ref.rowptr) and np.array_equal(got[1], ref.colidx) and np.array_equal(got[2], ref.vals)


@pytest.mark.parametrize("share", [0.2, 0.4])
def test_a_few_heavy_columns(B, share):
    """Ten columns of 400 are heavier than the rest: with 0.2 their products are fewer than the rows to look at, which are counted
    without masks then, with 0.4 more."""
    m, n = 3000, 400
    rng = np.random.default_rng(3)
    keep = rng.random((m, n)) < np.where(np.arange(n) % 40 == 7, share, 0.125)
    rp = np.concatenate(([0], np.cumsum(keep.sum(1)))).astype(np.int64)
    ci = np.nonzero(keep)[1].astype(np.int32)
    dev = (torch.from_numpy(rp).cuda(), torch.from_numpy(ci).cuda(), torch.ones(ci.size, dtype=torch.int32, device="cuda"))
    ref = oracle.syrk(m, n, rp, ci, np.ones(ci.size, dtype=np.int32), oracle.TRIL)
    got = _run(B, B.spsyrk_plan(m, n, *dev), m, torch.int32, False)
    assert np.array_equal(got[0], ref.rowptr) and np.array_equal(got[1], ref.colidx) and np.array_equal(got[2].astype(np.float64), ref.vals)
