"""Calls outside the common sequence: matrices that fail their checks in a workspace with old contents, one plan on
several streams and threads, row ranges, similarities of values other than one; against the CPU oracle or against the
same product computed the common way."""
import threading

import numpy as np
import pytest
import torch

import oracle
from paper_2608_09713_b200 import workloads as W
from test_gpu_parity import B, dev, run_and_compare  # noqa: F401  (B is the fixture)

pytestmark = pytest.mark.gpu


def random_csr(m, n, per_row, dtype, seed, ones=False):
    """CSR with 1 to 2 * per_row - 1 entries per row, uniform columns."""
    rng = np.random.default_rng(seed)
    rows = [np.unique(rng.integers(0, n, rng.integers(1, 2 * per_row))) for _ in range(m)]
    rowptr = np.zeros(m + 1, dtype=np.int64)
    np.cumsum([r.size for r in rows], out=rowptr[1:])
    vals = np.ones(rowptr[-1]) if ones else rng.integers(1, 9, rowptr[-1]) if dtype == np.int32 else rng.uniform(-1, 1, rowptr[-1])
    return W.CSR(m, n, rowptr, np.concatenate(rows).astype(np.int32), vals.astype(dtype))


# ------------------------------------------------------------------ streams and torch's allocator
@pytest.mark.parametrize("call", ["product", "one pass", "mirror"])
def test_memory_of_the_binding_while_another_stream_uses_it(B, call):
    """A call on another stream than the current one leaves its workspace in use when it returns, and the plan is dropped: new tensors
    of the current stream must not get that memory yet."""
    a = random_csr(30_000, 30_000, 12, np.float64, 5)
    d = dev(a)
    c = B.tril_syrk(a.m, a.n, *d)[:3]

    def run(stream):
        if call == "product":
            return B.tril_syrk(a.m, a.n, *d, stream=stream)[:3]
        if call == "mirror":
            return B.spsyrk_mirror(a.m, *c, stream=stream)
        return B.onepass_syrk(B.spsyrk_plan(a.m, a.n, *d, stream=stream), stream)

    expected = run(None)
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    for _ in range(5):
        got = run(side)
        others = [torch.full((1 << k,), 0x5a, dtype=torch.uint8, device="cuda") for k in range(12, 29)]
        torch.cuda.synchronize()
        assert all(torch.equal(x, y) for x, y in zip(got, expected))
        del others, got


# ------------------------------------------------------------------ matrices that fail their checks
@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("fault", ["column ids", "one column id", "row pointers", "duplicate"])
def test_bad_csr_writes_nothing_outside_the_workspace(B, fault, mode):
    """Three radix passes (n = 2^17 + 3).  The workspace holds words of an earlier use: valid column ids and, as
    often, positions that would lead behind the workspace, where words that must not change lie."""
    a = random_csr(3000, (1 << 17) + 3, 8, np.float64, 1)
    nnz = a.colidx.size
    rng = np.random.default_rng(2)
    rowptr, colidx, vals = dev(a)
    if fault == "column ids":
        colidx[torch.from_numpy(rng.integers(0, nnz, nnz // 4)).cuda()] = a.n + 5
    elif fault == "one column id":
        colidx[7] = a.n + 5
    elif fault == "row pointers":
        rowptr[100], rowptr[200] = int(rowptr[150]), 3
    else:
        p = int(rowptr[40])
        colidx[p + 1] = colidx[p]
    size = B.spsyrk_plan_workspace_bytes(a.m, a.n, nnz, torch.float64, mode)
    total = 4 * size
    buf = torch.empty(total, dtype=torch.uint8, device="cuda")
    words = buf.view(torch.int32)
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    near = torch.randint(0, a.n, words.shape, generator=g, device="cuda", dtype=torch.int32)
    far = torch.randint(size // 8 + 1, (total - size) // 8 - 1, words.shape, generator=g, device="cuda", dtype=torch.int32)
    words.copy_(torch.where(torch.rand(words.shape, generator=g, device="cuda") < 0.5, near, far))
    behind = buf[size:].clone()
    with pytest.raises(B.SpsyrkError) as e:
        B.spsyrk_plan(a.m, a.n, rowptr, colidx, vals, mode=mode, workspace=buf[:size])
    assert e.value.status == 2
    assert torch.equal(buf[size:], behind)
    plan = B.spsyrk_plan(a.m, a.n, *dev(a), mode=mode, workspace=buf[:size])  # the next plan in the same workspace
    run_and_compare(B, a, mode, plan=plan)
    assert torch.equal(buf[size:], behind)


# ------------------------------------------------------------------ similarities
@pytest.mark.parametrize("m,n,per_row", [(900, 3000, 120), (20000, 700, 20), (12000, 400, 3)])
def test_similarities_of_values_other_than_one(B, m, n, per_row):
    """The fused similarity is spsyrk_jaccard's to the bit for any int32 values: the denominators are negative or zero for
    many entries (direct, rank and light rows)."""
    a = random_csr(m, n, per_row, np.int32, m)
    d = dev(a)
    rp, ci, cv, plan = B.tril_syrk(a.m, a.n, *d)
    jac = torch.full((cv.numel(),), -7.0, dtype=torch.float32, device="cuda")
    B.spsyrk_plan_set_jaccard(plan, jac)
    B.spsyrk_numeric(plan, rp, ci, cv)
    want = B.spsyrk_jaccard(a.m, 0, a.m, d[0], rp, ci, cv)
    assert torch.equal(jac.view(torch.int32), want.view(torch.int32))
    denominator = (d[0][1:] - d[0][:-1])
    rows = torch.repeat_interleave(torch.arange(m, device="cuda"), rp[1:] - rp[:-1])
    assert int((denominator[rows] + denominator[ci.long()] - cv < 0).sum()) > 1000


# ------------------------------------------------------------------ streams and threads
def test_nothing_of_a_plan_is_under_way_when_it_returns(B):
    """Binary matrix with many columns (its heavy columns are looked for among 2^26): the stream is idle when the plan returns,
    so the product may be taken on another stream."""
    m, n = 4000, 1 << 26
    rng = np.random.default_rng(4)
    a = random_csr(m, 300, 40, np.float32, 4, ones=True)
    spread = np.sort(rng.choice(n, 300, replace=False)).astype(np.int32)
    a = W.CSR(m, n, a.rowptr, spread[a.colidx], a.vals)
    d = dev(a)
    ref = oracle.syrk(m, n, a.rowptr, a.colidx, a.vals, oracle.TRIL)
    torch.cuda.synchronize()
    other = torch.cuda.Stream()
    for _ in range(3):
        plan = B.spsyrk_plan(m, n, *d)
        assert torch.cuda.current_stream().query()
        with torch.cuda.stream(other):
            rp, ci, cv, _ = B.tril_syrk(m, n, *d, plan=plan)
        torch.cuda.synchronize()
        assert np.array_equal(rp.cpu().numpy(), ref.rowptr) and np.array_equal(ci.cpu().numpy(), ref.colidx)
        assert np.array_equal(cv.cpu().numpy().astype(np.float64), ref.vals)


@pytest.mark.parametrize("mode", [0, 1])
def test_plan_of_no_rows_then_all(B, mode):
    """The binary analysis belongs to the plan, not to its row range: a plan of no rows, of one row, then of all."""
    a = random_csr(700, 5000, 60, np.int32, 9, ones=True)
    a.colidx[a.rowptr[:-1]] = 0  # a column that every row stores: heavy, and every row of the lower triangle is dense
    d = dev(a)
    for r0, r1 in ((0, 0), (350, 351), (700, 700)):
        plan = B.spsyrk_plan(a.m, a.n, *d, mode=mode, row_begin=r0, row_end=r1)
        run_and_compare(B, a, mode, r0, r1, plan=plan)
        B.spsyrk_plan_set_rows(plan, 0, a.m)
        run_and_compare(B, a, mode, plan=plan)


def heavy_matrix(m, dtype, seed):
    """Rows with more than 32 nonzeros over columns of about 40 entries, in every part of the range, among rows with one
    nonzero; a few rows that outgrow the smaller slot counts."""
    rng = np.random.default_rng(seed)
    n = max(m // 40, 64)
    rows = {i: np.array([rng.integers(n)]) for i in range(m)}
    for i in rng.choice(m, 300, replace=False):
        rows[i] = np.sort(rng.choice(n, 34, replace=False))
    for i in rng.choice(np.arange(m // 2, m), 20, replace=False):
        rows[i] = np.sort(rng.choice(n, min(400, n), replace=False))
    rowptr = np.zeros(m + 1, dtype=np.int64)
    np.cumsum([rows[i].size for i in range(m)], out=rowptr[1:])
    vals = rng.integers(1, 9, rowptr[-1]) if dtype == np.int32 else rng.uniform(-1, 1, rowptr[-1])
    return W.CSR(m, n, rowptr, np.concatenate([rows[i] for i in range(m)]).astype(np.int32), vals.astype(dtype))


def test_plans_of_several_threads(B):
    """Every thread has its own matrix, plan and stream; the kernels of the heavy rows are launched with many sizes of shared
    memory side by side, the mirror's with several."""
    sizes = (150000, 140000, 70000, 20000)
    mats = [heavy_matrix(m, np.int32, m) for m in sizes]
    want = []
    for a in mats:
        rp, ci, cv, _ = B.tril_syrk(a.m, a.n, *dev(a))
        want.append((rp, ci, cv) + tuple(B.spsyrk_mirror(a.m, rp, ci, cv)))
    torch.cuda.synchronize()
    failures = []

    def work(k):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                a = mats[k]
                d = dev(a)
                rp, ci, cv, plan = B.tril_syrk(a.m, a.n, *d)
                ci.fill_(-1)
                for _ in range(1500):
                    B.spsyrk_numeric(plan, rp, ci, cv)
                f = B.spsyrk_mirror(a.m, rp, ci, cv)
                torch.cuda.current_stream().synchronize()
                if not all(torch.equal(x, y) for x, y in zip((rp, ci, cv) + tuple(f), want[k])):
                    failures.append((k, "another result"))
        except Exception as e:  # noqa: BLE001 (reported by the assertion)
            failures.append((k, repr(e)))

    threads = [threading.Thread(target=work, args=(k,)) for k in range(len(sizes))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failures


@pytest.mark.parametrize("mode", [0, 1])
def test_one_plan_on_two_streams(B, mode):
    """Two numeric passes of one plan, and passes over row ranges of it, under way at the same time: every entry is written in
    all of them."""
    a = W.rmat(14, 16, 7)
    rp, ci, cv, plan = B.tril_syrk(a.m, a.n, *dev(a), mode=mode)
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in range(2)]
    outs = [(torch.full_like(ci, -1), torch.zeros_like(cv)) for _ in range(4)]
    torch.cuda.synchronize()
    for st, out in zip(streams, outs):
        B.spsyrk_numeric(plan, rp, *out, stream=st)
    for k in range(4):
        for st, out in zip(streams, outs[2:]):
            B.spsyrk_numeric_rows(plan, a.m * k // 4, a.m * (k + 1) // 4, rp, *out, stream=st)
    torch.cuda.synchronize()
    scale = cv.abs().clamp(min=1e-30)
    for c, v in outs:
        assert torch.equal(c, ci)
        assert float(((v - cv).abs() / scale).max()) <= 1e-5  # (sums of positive products: any order of additions)


@pytest.mark.parametrize("dtype", [torch.float32, torch.int32])
def test_heavy_rows_through_the_host_entry(B, dtype):
    """A power-law product large enough to be computed and downloaded in six row blocks, against the same on the device."""
    a = W.rmat(15, 16, 7)
    vals = torch.from_numpy(a.vals).to(dtype) if dtype == torch.float32 else torch.arange(a.vals.size, dtype=torch.int32) % 5
    d = (torch.from_numpy(a.rowptr), torch.from_numpy(a.colidx), vals)
    rp, ci, cv, _ = B.tril_syrk(a.m, a.n, *(t.cuda() for t in d))
    assert ci.numel() > 24 << 20  # a block per 4 << 20 entries
    h_rp, h_ci, h_cv = B.spsyrk_host_tril(a.m, a.n, *d)
    assert torch.equal(h_rp, rp.cpu()) and torch.equal(h_ci, ci.cpu())
    if dtype == torch.int32:
        assert torch.equal(h_cv, cv.cpu())
    else:  # (sums of positive products: any order of additions)
        assert float(((h_cv - cv.cpu()).abs() / cv.cpu()).max()) <= 1e-5


# ------------------------------------------------------------------ mirror: where the entries lie, how many rows there are
def lower_triangle(m, rows, cols, dtype, seed=1):
    """CSR of the distinct (row, column) pairs, on the GPU; values are distinct small numbers."""
    code = torch.unique(rows * m + cols)
    r = torch.div(code, m, rounding_mode="floor")
    rp = torch.searchsorted(r, torch.arange(m + 1, device="cuda"))
    vals = (torch.arange(code.numel(), device="cuda") % 1_000_003 + seed).to(dtype)
    return rp, (code - r * m).to(torch.int32), vals


def check_mirror(B, m, c, f=None):
    """F against the union of C_L and its reflection, sorted."""
    rp, ci, cv = c
    f_rp, f_ci, f_cv = B.spsyrk_mirror(m, *c) if f is None else f
    rows = torch.repeat_interleave(torch.arange(m, device="cuda"), rp[1:] - rp[:-1])
    below = ci < rows
    code = torch.cat([rows * m + ci, ci[below].long() * m + rows[below]])
    order = torch.argsort(code)
    code = code[order]
    r = torch.div(code, m, rounding_mode="floor")
    assert torch.equal(f_rp, torch.searchsorted(r, torch.arange(m + 1, device="cuda")))
    assert torch.equal(f_ci.long(), code - r * m)
    assert torch.equal(f_cv, torch.cat([cv, cv[below]])[order])


def arange(m):
    return torch.arange(m, device="cuda")


def pattern(name, m, k):
    g = torch.Generator(device="cuda")
    g.manual_seed(m + k)
    rows = torch.randint(0, m, (k,), generator=g, device="cuda")
    share = torch.rand(k, generator=g, device="cuda", dtype=torch.float64)
    if name == "spread":
        cols = (share * (rows + 1)).long()
    elif name == "one column":
        rows, cols = arange(m), torch.zeros_like(arange(m))
    elif name == "every 512th column":
        cols = (share * (rows // 512 + 1)).long() * 512
    elif name == "few rows":
        rows = rows % 7 * (m // 7)
        cols = (share * (rows + 1)).long()
    cols = torch.minimum(cols, rows)
    return torch.cat([rows, arange(m)[:: 1 if name != "few rows" else m // 5]]), torch.cat([cols, arange(m)[:: 1 if name != "few rows" else m // 5]])


@pytest.mark.parametrize("name", ["spread", "one column", "every 512th column", "few rows"])
@pytest.mark.parametrize("m,k,dtype", [(1 << 18, 1 << 21, torch.float32), ((1 << 19) + 1, 20_000_000, torch.int32), ((1 << 20) - 3, 1_000_000, torch.float32),
                                       (65536, 1 << 21, torch.float64), ((1 << 24) + 1, 3_000_000, torch.float32)])
def test_mirror_wherever_the_entries_lie(B, name, m, k, dtype):
    """Buckets that are cut into pieces and buckets that are not, two passes and three, radix passes for few entries and for
    more than 2^24 rows, rows that are searched for."""
    check_mirror(B, m, lower_triangle(m, *pattern(name, m, k), dtype))


def test_mirror_takes_about_the_same_time_wherever_the_entries_lie(B):
    """2^18 rows: entries in one column, in every 512th column, or two entries in all, against entries all over."""
    m = 1 << 18

    def microseconds(c):
        B.spsyrk_mirror(m, *c)
        best = 1e9
        for _ in range(5):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            B.spsyrk_mirror(m, *c)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b) * 1e3)
        return best

    spread = microseconds(lower_triangle(m, *pattern("spread", m, 1 << 22), torch.float32))
    ends = torch.tensor([3, m - 1], device="cuda")
    for c in (lower_triangle(m, *pattern("one column", m, 0), torch.float32), lower_triangle(m, *pattern("every 512th column", m, 1 << 22), torch.float32),
              lower_triangle(m, ends, ends, torch.float32)):
        assert microseconds(c) < 3 * spread


@pytest.mark.parametrize("m,k", [(5000, 50_000), ((1 << 19) + 1, 20_000_000), ((1 << 24) + 1, 1_000_000)])
@pytest.mark.parametrize("shift", [1, 2, 3])
def test_mirror_of_4_byte_values_into_unaligned_arrays(B, m, k, shift):
    """F's arrays may begin at any multiple of four bytes (8-byte values: multiples of sixteen)."""
    import ctypes
    c = lower_triangle(m, *pattern("spread", m, k), torch.float32)
    rp, ci, cv = c
    nnz_f = 2 * ci.numel() - m
    lib, code = B._lib, B._DTYPE_CODE[torch.float32]
    size = ctypes.c_size_t(0)
    B._check(lib.spsyrk_mirror(m, ci.numel(), code, None, None, None, None, None, None, None, None, ctypes.byref(size), None), "size")
    ws = torch.empty(size.value, dtype=torch.uint8, device="cuda")
    f_rp = torch.empty(m + 1, dtype=torch.int64, device="cuda")
    f_ci = torch.full((nnz_f + 2 * shift,), -9, dtype=torch.int32, device="cuda")
    f_cv = torch.full((nnz_f + 2 * shift,), -9.0, device="cuda")
    nnz = ctypes.c_int64(0)
    args = (m, ci.numel(), code, B._p(rp), B._p(ci), B._p(cv), B._p(f_rp))
    B._check(lib.spsyrk_mirror(*args, None, None, ctypes.byref(nnz), B._p(ws), ctypes.byref(size), B._stream(None)), "sizes")
    assert nnz.value == nnz_f
    ci_out, cv_out = f_ci[shift : shift + nnz_f], f_cv[shift : shift + nnz_f]
    B._check(lib.spsyrk_mirror(*args, B._p(ci_out), B._p(cv_out), ctypes.byref(nnz), B._p(ws), ctypes.byref(size), B._stream(None)), "fill")
    check_mirror(B, m, c, (f_rp, ci_out, cv_out))
    for t in (f_ci, f_cv):
        assert bool((t[:shift] == -9).all()) and bool((t[shift + nnz_f :] == -9).all())
