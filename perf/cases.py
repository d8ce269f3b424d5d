"""What a user of the library has it do, as timed cases over the public entry points of the binding.

Every pass of the product starts from a matrix A that the library has not seen: a program that squares a
matrix plans it once and multiplies once, so the plan is part of the pass.  Inputs are the seeded shapes of
``paper_2608_09713_b200/workloads.py`` (Erdos-Renyi, bounded-Zipf binary, R-MAT, hypergraph incidence), drawn
on the GPU so that many of them can be made quickly.

A case is ``{"kind": matrix family, "op": what is done with it, "dtype": value type, sizes...}``.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2608_09713_b200 import binding as B

_DT = {"f64": torch.float64, "f32": torch.float32, "i32": torch.int32}
_SV = {"f64": 8, "f32": 4, "i32": 4}


def listed():
    return [
        # The smallest call: a product and its full symmetric form, all launch latency.
        {"name": "er_4096_d8_f64_mirror", "kind": "er", "op": "mirror", "dtype": "f64", "m": 4096, "n": 4096, "d": 8},
        # Similarities of a few thousand sets (one batch of samples): every output row is dense.
        {"name": "zipf_3001_d100_i32_jaccard", "kind": "zipf", "op": "jaccard", "dtype": "i32", "m": 3001, "n": 1 << 17, "d": 100},
        # Common neighbours in a small power-law graph, single precision, rows of every weight.
        {"name": "rmat_s13_f32_tril", "kind": "rmat", "op": "tril", "dtype": "f32", "scale": 13, "ef": 16},
        # A ragged mid-size product whose consumer needs only the triangle.
        {"name": "er_60001_d16_f64_tril", "kind": "er", "op": "tril", "dtype": "f64", "m": 60001, "n": 60001, "d": 16},
        # Algorithm 2 on one process: two column panels, two products, one accumulation.
        {"name": "rmat_s15_f32_panels", "kind": "rmat", "op": "panels", "dtype": "f32", "scale": 15, "ef": 16},
        # Host buffers in, host buffers out (the call of a program that keeps its data on the CPU).
        {"name": "er_262144_d16_f64_host", "kind": "er", "op": "host", "dtype": "f64", "m": 1 << 18, "n": 1 << 18, "d": 16},
        # Both triangles at once: the full-output mode on an incidence matrix.
        {"name": "hyper_500003_f64_full", "kind": "hyper", "op": "full", "dtype": "f64", "m": 500_003, "n": 125_000},
        # Iterating on C without materialising it: a block of eight vectors through a triangle that is kept.
        {"name": "er_1048576_d16_f64_symm8", "kind": "er", "op": "symm", "dtype": "f64", "m": 1 << 20, "n": 1 << 20, "d": 16, "p": 8},
        # The large hypergraph overlap matrix with its symmetric form.
        {"name": "hyper_2000000_f64_mirror", "kind": "hyper", "op": "mirror", "dtype": "f64", "m": 2_000_000, "n": 500_000},
        # The large power-law graph: heavy rows carry most of the work.
        {"name": "rmat_s18_f32_mirror", "kind": "rmat", "op": "mirror", "dtype": "f32", "scale": 18, "ef": 16},
        # All-pairs similarity of a large binary matrix.
        {"name": "zipf_50000_d100_i32_jaccard", "kind": "zipf", "op": "jaccard", "dtype": "i32", "m": 50_000, "n": 1 << 22, "d": 100},
        # The headline workload: the large random matrix, product and symmetric form, double precision.
        {"name": "er_4194304_d16_f64_mirror", "kind": "er", "op": "mirror", "dtype": "f64", "m": 1 << 22, "n": 1 << 22, "d": 16},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: the families, operations, types and size ranges that the listed cases stand for."""
    family = rng.choice(("er", "er", "hyper", "rmat", "zipf", "consume", "host"))
    if family == "er":
        m = _log_int(rng, 2_000, 3_000_000)
        n = max(64, int(m * rng.uniform(0.5, 2.0)))
        d = rng.randint(4, 20)
        if d * d * m * m / n > 5e8:  # about 2.5e8 partial products at most
            m, n = int(5e8 / (d * d * m / n)), int(5e8 / (d * d * m / n) * n / m)
        return {"kind": "er", "op": rng.choice(("tril", "mirror", "mirror", "full")), "dtype": rng.choice(("f64", "f64", "f32")), "m": m, "n": n, "d": d}
    if family == "hyper":
        m = _log_int(rng, 20_000, 1_500_000)
        return {"kind": "hyper", "op": rng.choice(("tril", "mirror", "full")), "dtype": rng.choice(("f64", "f32")), "m": m, "n": m // 4 + 8192}
    if family == "rmat":
        return {"kind": "rmat", "op": rng.choice(("tril", "mirror", "panels")), "dtype": rng.choice(("f32", "f32", "f64")), "scale": rng.randint(11, 16), "ef": 16}
    if family == "zipf":
        return {"kind": "zipf", "op": "jaccard", "dtype": "i32", "m": _log_int(rng, 1_000, 40_000), "n": 1 << rng.randint(16, 21), "d": rng.randint(60, 140)}
    if family == "consume":
        m = _log_int(rng, 10_000, 1_000_000)
        return {"kind": "er", "op": "symm", "dtype": rng.choice(("f64", "f32")), "m": m, "n": m, "d": 16, "p": rng.choice((1, 3, 8))}
    m = _log_int(rng, 10_000, 300_000)
    return {"kind": "er", "op": "host", "dtype": rng.choice(("f64", "f32")), "m": m, "n": m, "d": 16}


# ------------------------------------------------------------------------------------------
# Inputs, on the GPU, from the seed alone.
# ------------------------------------------------------------------------------------------
def _csr(m, n, code):
    """Canonical CSR (row pointers, column ids) of the positions row * n + column, duplicates merged."""
    code = torch.unique(code)
    rows = torch.div(code, n, rounding_mode="floor")
    col = (code - rows * n).to(torch.int32)
    rowptr = torch.searchsorted(rows, torch.arange(m + 1, device="cuda"))
    return rowptr, col


def _positions_er(c, g):
    m, n, d = c["m"], c["n"], c["d"]
    cols = torch.randint(0, n, (m, d), generator=g, device="cuda")
    return m, n, (cols + torch.arange(m, device="cuda")[:, None] * n).reshape(-1)


def _positions_hyper(c, g):
    m, n = c["m"], c["n"]
    band = min(4096, n)
    rows = torch.arange(m, device="cuda")[:, None]
    deg = torch.randint(2, 9, (m, 1), generator=g, device="cuda")
    u = torch.rand((m, 8), generator=g, device="cuda", dtype=torch.float64)
    lo = (rows * n // m - band // 2).clamp(0, n - band)
    cols = torch.where(torch.rand((m, 8), generator=g, device="cuda") < 0.1, (u * n).long(), lo + (u * band).long())
    return m, n, (rows * n + cols)[torch.arange(8, device="cuda")[None, :] < deg]


def _positions_rmat(c, g):
    nv = 1 << c["scale"]
    rows = torch.zeros(c["ef"] * nv, dtype=torch.int64, device="cuda")
    cols = torch.zeros_like(rows)
    for _ in range(c["scale"]):
        u = torch.rand(rows.shape, generator=g, device="cuda")
        q = (u >= 0.57).long() + (u >= 0.76) + (u >= 0.95)
        rows, cols = rows * 2 + (q >> 1), cols * 2 + (q & 1)
    keep = rows != cols
    return nv, nv, rows[keep] * nv + cols[keep]


def _positions_zipf(c, g):
    """The first d distinct columns of a sequence of bounded-Zipf(1.1) draws per row."""
    m, n, d = c["m"], c["n"], c["d"]
    cdf = torch.cumsum(torch.arange(1, n + 1, device="cuda", dtype=torch.float64) ** -1.1, 0)
    cdf /= cdf[-1].clone()
    k = 3 * d
    out = []
    for r0 in range(0, m, 8192):
        rows = min(8192, m - r0)
        u = torch.rand((rows, k), generator=g, device="cuda", dtype=torch.float64)
        rank = torch.searchsorted(cdf, u, right=True).clamp_(max=n - 1)
        srt, order = torch.sort(rank, dim=1, stable=True)
        fresh = torch.ones_like(srt, dtype=torch.bool)
        fresh[:, 1:] = srt[:, 1:] != srt[:, :-1]
        first = torch.zeros_like(fresh).scatter_(1, order, fresh)  # the draw is the first of its rank in the row
        use = first & (torch.cumsum(first, 1) <= d)
        row = torch.arange(r0, r0 + rows, device="cuda")[:, None].expand(rows, k)
        out.append(row[use] * n + rank[use])
    return m, n, torch.cat(out)


def _relabelling(count, block, g):
    """A random permutation of 0..count-1, or, with a block size, one that keeps every label inside its block."""
    key = torch.rand(count, generator=g, device="cuda", dtype=torch.float64)
    if block:
        key += torch.arange(count, device="cuda") // block
    return torch.argsort(key)


def _matrix(case, seed):
    # The pattern is drawn once per set of sizes; the seed relabels its rows and columns and draws the values.  A and
    # C then have the same number of entries for every seed (a relabelling of A's rows is a symmetric one of C's), and
    # everything else about them is another input.  The banded family is relabelled inside blocks of 256.
    base = torch.Generator(device="cuda")
    base.manual_seed(20_260_809)
    m, n, code = globals()["_positions_" + case["kind"]](case, base)
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    block = 256 if case["kind"] == "hyper" else 0
    rperm, cperm = _relabelling(m, block, g), _relabelling(n, block, g)
    rows = torch.div(code, n, rounding_mode="floor")
    code = rperm[rows] * n + cperm[code - rows * n]
    del rows
    rowptr, col = _csr(m, n, code)
    del code
    dt = _DT[case["dtype"]]
    if case["kind"] in ("zipf", "hyper"):  # incidence: the stored values are ones
        vals = torch.ones(col.numel(), dtype=dt, device="cuda")
    elif case["kind"] == "rmat":
        vals = torch.rand(col.numel(), generator=g, device="cuda", dtype=dt) + 0.5
    else:
        vals = torch.rand(col.numel(), generator=g, device="cuda", dtype=dt) * 2 - 1
    return m, n, rowptr, col, vals, g


def prepare(case, seed):
    m, n, rowptr, col, vals, g = _matrix(case, seed)
    state = {"op": case["op"], "m": m, "n": n}
    if case["op"] == "symm":
        # an iterative program keeps the triangle and multiplies with new vectors
        c_rowptr, c_col, c_vals, plan = B.tril_syrk(m, n, rowptr, col, vals)
        del plan
        shape = (m, case["p"]) if case["p"] > 1 else (m,)
        x = torch.rand(shape, generator=g, device="cuda", dtype=vals.dtype) * 2 - 1
        state.update(c=(c_rowptr, c_col, c_vals), x=x)
    elif case["op"] == "host":
        # pinned buffers the program keeps: A, and room for C_L with a margin over the expected size
        room = int(_nnz_tril(case) * 1.05) + 4096
        a = [torch.empty(t.shape, dtype=t.dtype, pin_memory=True).copy_(t) for t in (rowptr, col, vals)]
        out = (torch.empty(m + 1, dtype=torch.int64, pin_memory=True), torch.empty(room, dtype=torch.int32, pin_memory=True),
               torch.empty(room, dtype=vals.dtype, pin_memory=True))
        state.update(a=a, out=out)
    else:
        state["a"] = (rowptr, col, vals)
    if torch.cuda.is_available():
        torch.cuda.synchronize()
    return state


def run(state):
    op, m, n = state["op"], state["m"], state["n"]
    if op == "symm":
        x = state["x"]
        return B.spsyrk_symm(m, *state["c"], x) if x.dim() == 2 else B.spsyrk_symv(m, *state["c"], x)
    a = state["a"]
    if op == "tril":
        return B.tril_syrk(m, n, *a)[:3]
    if op == "full":
        return B.tril_syrk(m, n, *a, mode=B.FULL)[:3]
    if op == "mirror":
        c_rowptr, c_col, c_vals, plan = B.tril_syrk(m, n, *a)
        f = B.spsyrk_mirror(m, c_rowptr, c_col, c_vals)
        return (c_rowptr, c_col, c_vals) + f
    if op == "jaccard":
        plan = B.spsyrk_plan(m, n, *a)
        dev = a[0].device
        B.spsyrk_plan_lend_map(plan, torch.empty(max(B.spsyrk_plan_map_bytes(plan), 256), dtype=torch.uint8, device=dev))
        c_rowptr = torch.empty(m + 1, dtype=torch.int64, device=dev)
        nnz = B.spsyrk_symbolic(plan, c_rowptr)
        c_col = torch.empty(nnz, dtype=torch.int32, device=dev)
        c_cnt = torch.empty(nnz, dtype=torch.int32, device=dev)
        jac = torch.empty(nnz, dtype=torch.float32, device=dev)
        B.spsyrk_plan_set_jaccard(plan, jac)
        B.spsyrk_numeric(plan, c_rowptr, c_col, c_cnt)
        return c_rowptr, c_col, c_cnt, jac
    if op == "panels":
        half = n // 2
        parts = [B.tril_syrk(m, n, *B.spsyrk_column_panel(m, *a, k0, k1))[:3] for k0, k1 in ((0, half), (half, n))]
        return B.spsyrk_accumulate(m, *parts[0], *parts[1])
    if op == "host":
        return B.spsyrk_host_tril(m, n, *a, out=state["out"])
    raise ValueError(op)


# ------------------------------------------------------------------------------------------
# What a pass cannot do without: every input read once, every output written once, one multiply-add (two
# operations) per partial product.  Expected sizes of the random inputs; the drawn ones differ by well under 1 %.
# ------------------------------------------------------------------------------------------
# R-MAT, edge factor 16: log2 of entries of A per possible edge is close to linear; entries and partial products of
# the lower triangle by scale, counted on matrices of the recipe (16 and 17 interpolated)
_RMAT_NNZ_A = {9: 5603, 10: 12006, 11: 25455, 12: 53458, 13: 110900, 14: 228713, 15: 468622, 16: 955000, 17: 1942000, 18: 3940001}
_RMAT_NNZ_C = {9: 43875, 10: 139248, 11: 410827, 12: 1187306, 13: 3490778, 14: 10126298, 15: 28934089, 16: 82200000, 17: 230000000, 18: 638000000}
_RMAT_MAC = {9: 137427, 10: 415323, 11: 1193172, 12: 3385393, 13: 9586077, 14: 26700893, 15: 73577029, 16: 201000000, 17: 545000000, 18: 1468000000}


def _shape(case):
    return (1 << case["scale"], 1 << case["scale"]) if case["kind"] == "rmat" else (case["m"], case["n"])


def _zipf_inclusion(case):
    """Probability that a row stores the column of each rank: draws until d distinct, the number of draws in expectation."""
    n, d = case["n"], case["d"]
    p = np.arange(1, n + 1, dtype=np.float64) ** -1.1
    p /= p.sum()
    lo, hi = float(d), 20.0 * d
    for _ in range(40):
        mid = (lo + hi) / 2
        lo, hi = (mid, hi) if float(-np.expm1(mid * np.log1p(-p)).sum()) < d else (lo, mid)
    return -np.expm1(lo * np.log1p(-p))


def _sizes(case):
    """(nnz(A), partial products with j <= i, nnz(C_L))."""
    kind = case["kind"]
    if kind == "rmat":
        s = case["scale"]
        return _RMAT_NNZ_A[s], _RMAT_MAC[s], _RMAT_NNZ_C[s]
    m, n = _shape(case)
    if kind == "er":
        nnz = -m * n * math.expm1(case["d"] * math.log1p(-1.0 / n))
        lam = nnz / n
        pairs = m * (m - 1) / 2.0
        return nnz, n * lam * lam / 2 + nnz, m - pairs * math.expm1(n * math.log1p(-(nnz / m / n) ** 2))
    if kind == "hyper":
        nnz = m * 4.998
        lam = nnz / n
        return nnz, n * lam * lam / 2 + nnz, m + 0.998 * n * lam * lam / 2
    q = _zipf_inclusion(case)
    nnz = float(m) * case["d"]
    return nnz, float((m * q) ** 2 @ np.ones_like(q)) / 2 + nnz / 2, m * (m + 1) / 2.0


def _nnz_tril(case):
    return _sizes(case)[2]


def work(case):
    m, _ = _shape(case)
    sv = _SV[case["dtype"]]
    nnz, macs, nnz_c = _sizes(case)
    op = case["op"]
    a_bytes = 8 * (m + 1) + nnz * (4 + sv)
    c_bytes = 8 * (m + 1) + nnz_c * (4 + sv)
    f_bytes = 8 * (m + 1) + (2 * nnz_c - m) * (4 + sv)
    if op == "symm":
        return {"bytes": c_bytes + 2 * m * case["p"] * sv, "flops": 4 * nnz_c * case["p"]}
    if op == "mirror":
        return {"bytes": a_bytes + c_bytes + f_bytes, "flops": 2 * macs}
    if op == "full":
        return {"bytes": a_bytes + f_bytes, "flops": 4 * macs}
    if op == "jaccard":
        return {"bytes": a_bytes + c_bytes + 4 * nnz_c, "flops": 2 * macs}
    return {"bytes": a_bytes + c_bytes, "flops": 2 * macs}  # tril, panels (their sum), host


def tolerance(case):
    # Whole numbers (row pointers, column ids, counts) are exact.  Measured as 2-norms, stated about four times wider:
    # a product of doubles against another library's order of summation 1.1e-15 on heavy rows (1.2e-16 on light ones);
    # single precision accumulated in double and rounded once 2.7e-8 (after the addition of two panels 3.7e-8);
    # symm / symv against another order 5.3e-16 in double, against double arithmetic 2.7e-7 in single; a similarity is
    # one single-precision division.
    if case["op"] == "symm":
        return {"rel": 2e-15} if case["dtype"] == "f64" else {"rel": 1.1e-6}
    return {"rel": 4e-15} if case["dtype"] == "f64" else {"rel": 1.5e-7}
