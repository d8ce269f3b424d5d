"""The asynchronous fill steps of the mirror and of the sparse sum captured into a CUDA graph and replayed."""
import ctypes

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2608_09713_b200 import binding
    return binding


def _product(B, m, d, dtype):
    g = torch.Generator(device="cuda")
    g.manual_seed(m)
    code = torch.unique(torch.randint(0, m, (m, d), generator=g, device="cuda") + torch.arange(m, device="cuda")[:, None] * m)
    rowptr = torch.searchsorted(torch.div(code, m, rounding_mode="floor"), torch.arange(m + 1, device="cuda"))
    return B.tril_syrk(m, m, rowptr, (code % m).to(torch.int32), torch.rand(code.numel(), generator=g, device="cuda", dtype=dtype) - 0.5)[:3]


def _replays(call, outputs, expected):
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        call()  # outside the capture first (function attributes)
    torch.cuda.current_stream().wait_stream(side)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        call()
    for _ in range(2):
        for t in outputs:
            t.fill_(-1)
        graph.replay()
        torch.cuda.synchronize()
        for t, e in zip(outputs, expected):
            assert torch.equal(t, e)


# by buckets in two passes (small and of several tiles), by records, by radix passes, by buckets in three passes
@pytest.mark.parametrize("m,d,dtype", [(500, 4, torch.float64), (9000, 8, torch.float64), (9000, 8, torch.float32), (70_000, 6, torch.float64),
                                       (300_000, 4, torch.float64), (300_000, 4, torch.float32), (300_000, 12, torch.float32)])
def test_mirror_fill_replays(B, m, d, dtype):
    c = _product(B, m, d, dtype)
    expected = B.spsyrk_mirror(m, *c)
    outputs = [torch.empty_like(t) for t in expected]
    sz = ctypes.c_size_t(B.spsyrk_mirror_workspace_bytes(m, c[1].numel(), dtype))
    ws = B._workspace(sz.value, torch.device("cuda"))
    nnz = ctypes.c_int64(0)
    code = B._DTYPE_CODE[dtype]
    args = lambda col, val: (m, c[1].numel(), code, *map(B._p, c), B._p(outputs[0]), col, val, ctypes.byref(nnz), B._p(ws), ctypes.byref(sz), B._stream(None))
    assert B._lib.spsyrk_mirror(*args(None, None)) == 0

    def call():
        assert B._lib.spsyrk_mirror(*args(B._p(outputs[1]), B._p(outputs[2]))) == 0
    _replays(call, outputs, expected)


@pytest.mark.parametrize("m,d", [(9000, 4), (2000, 40)])  # some lanes per row, a warp per row with rows of a CTA each
def test_accumulate_fill_replays(B, m, d):
    x, y = _product(B, m, d, torch.float32), _product(B, m, d + 1, torch.float32)
    expected = B.spsyrk_accumulate(m, *x, *y)
    outputs = [torch.empty_like(t) for t in expected[1:]]
    sz, nnz = ctypes.c_size_t(0), ctypes.c_int64(0)
    head = lambda: (m, B._DTYPE_CODE[torch.float32], x[1].numel(), *map(B._p, x), y[1].numel(), *map(B._p, y), B._p(expected[0]))
    assert B._lib.spsyrk_accumulate(*head(), None, None, None, None, ctypes.byref(sz), None) == 0
    ws = B._workspace(sz.value, torch.device("cuda"))

    def call():
        assert B._lib.spsyrk_accumulate(*head(), *map(B._p, outputs), ctypes.byref(nnz), B._p(ws), ctypes.byref(sz), B._stream(None)) == 0
    _replays(call, outputs, expected[1:])
