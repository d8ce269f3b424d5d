"""The sparse sum at the edges of its windows and tiles: a warp merges 32 entries of either row at a time, a CTA 2048 of both; rows
of more than 1024 entries of both inputs go to a CTA, where there are many entries those of more than 4096."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2608_09713_b200 import binding
    return binding


def _pair(kind, size, rng):
    """Ascending ids of one row of X and of Y, `size` entries together (of identical rows: of each)."""
    if kind == "same":  # every tile ends between the two entries of a pair, or could
        a = np.sort(rng.choice(3 * size + 1, size, replace=False))
        return a, a
    if kind == "shifted":  # one more id in front of Y: the pairs straddle the borders of threads and tiles differently
        a = np.arange(1, size + 1)
        return a, np.arange(size)
    if kind == "blocks":  # long runs of one row between ids of the other
        ids = np.arange(size)
        own = (ids // 700) % 2 == 0
        return ids[own], ids[~own]
    if kind == "one":  # only X
        return np.arange(size), np.zeros(0, dtype=np.int64)
    mask = rng.integers(0, 3, size=size)  # random: X only, Y only, both
    ids = np.sort(rng.choice(5 * size + 1, size, replace=False))
    return ids[mask != 1], ids[mask != 0]


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32, torch.int32])
@pytest.mark.parametrize("empty_rows", [0, 8000], ids=["warp", "group"])  # many empty rows: few lanes per row
@pytest.mark.parametrize("kind", ["same", "shifted", "blocks", "one", "random"])
def test_accumulate_at_tile_edges(B, kind, empty_rows, dtype):
    rng = np.random.default_rng(7)
    pairs = [_pair(kind, s, rng) for s in (1, 7, 8, 9, 31, 32, 33, 63, 64, 65, 127, 128, 129, 255, 256, 257, 511, 512, 513, 1023, 1024, 1025, 2047, 2048, 2049, 4095, 4096, 4097, 8191, 8192, 8193, 20_011)]
    pairs += [(np.zeros(0, dtype=np.int64),) * 2] * empty_rows + [pairs[-1], pairs[4]]
    m = len(pairs)
    npdt = {torch.float64: np.float64, torch.float32: np.float32, torch.int32: np.int32}[dtype]

    def csr(side):
        rows = [p[side] for p in pairs]
        rp = np.concatenate(([0], np.cumsum([r.size for r in rows]))).astype(np.int64)
        v = rng.integers(-9, 10, size=rp[-1]) if dtype == torch.int32 else rng.standard_normal(rp[-1])
        return rp, np.concatenate(rows).astype(np.int32), v.astype(npdt)

    x, y = csr(0), csr(1)
    zr, zc, zv = (t.cpu().numpy() for t in B.spsyrk_accumulate(m, *[torch.from_numpy(t).cuda() for t in x], *[torch.from_numpy(t).cuda() for t in y]))
    er, ec, ev = oracle.add(m, x[0], x[1], x[2].astype(np.float64), y[0], y[1], y[2].astype(np.float64))
    assert np.array_equal(zr, er) and np.array_equal(zc, ec)
    assert np.array_equal(zv, ev.astype(npdt))  # one rounded addition: the double sum of two floats rounds to the float sum


def test_accumulate_of_many_entries(B):
    """So many entries that a warp merges rows of up to 4096: rows on both sides of that, among rows of 2000."""
    rng = np.random.default_rng(17)
    lengths = [np.where(np.arange(7400) % 100 == 0, rng.integers(2040, 2056, 7400), rng.integers(900, 1100, 7400)) for _ in range(2)]
    x, y = (_device_csr(ln, 51 + i) for i, ln in enumerate(lengths))
    assert (x[1].numel() + y[1].numel()) // (148 * 24) >= 4096
    got = [t.cpu().numpy() for t in B.spsyrk_accumulate(7400, *x, *y)]
    ref = oracle.add(7400, *(t.cpu().numpy() for t in x), *(t.cpu().numpy() for t in y))
    assert all(np.array_equal(a, b) for a, b in zip(got, ref))


@pytest.mark.parametrize("m", [65_536, 65_537, 1 << 20, (1 << 20) + 3])  # long rows are looked for row by row, by units of 4 rows, of 32
@pytest.mark.parametrize("mean", [2, 20], ids=["lanes", "warps"])
def test_long_rows_wherever_they_stand(B, m, mean):
    """The first, the last, neighbours, rows at the ends of a unit, and a unit that is long in all but not in any row."""
    rng = np.random.default_rng(m)
    csr = []
    for side in range(2):
        lengths = rng.integers(0, mean + 1, size=m)
        lengths[[0, 1, 31, 32, 127, 128, m // 2, m // 2 + 1, m - 4, m - 1]] = rng.integers(600, 5000, size=10)
        lengths[4096:4096 + 32] = 60
        csr.append(_device_csr(lengths, m + side))
    got = [t.cpu().numpy() for t in B.spsyrk_accumulate(m, *csr[0], *csr[1])]
    ref = oracle.add(m, *(t.cpu().numpy() for t in csr[0] + csr[1]))
    assert all(np.array_equal(a, b) for a, b in zip(got, ref))


@pytest.mark.parametrize("size", [300, 5000])
@pytest.mark.parametrize("side", [0, 1])
def test_accumulate_refuses_rows_that_do_not_ascend(B, size, side):
    """The check across the borders of tiles: one equal pair of neighbours anywhere in the row."""
    for at in (1, 31, 32, size // 2, 255, 256, 257, size - 1):
        good = np.arange(size, dtype=np.int32)
        bad = good.copy()
        bad[at] = bad[at - 1]
        cols = [bad, good] if side == 0 else [good, bad]
        rp = torch.tensor([0, size], dtype=torch.int64, device="cuda")
        v = torch.ones(size, dtype=torch.float64, device="cuda")
        with pytest.raises(B.SpsyrkError) as e:
            B.spsyrk_accumulate(1, rp, torch.from_numpy(cols[0]).cuda(), v, rp, torch.from_numpy(cols[1]).cuda(), v)
        assert e.value.status == 2


def _device_csr(lengths, seed):
    """Rows of the given lengths, ascending with small random gaps, and their values on the GPU."""
    rng = np.random.default_rng(seed)
    rp = np.concatenate(([0], np.cumsum(lengths))).astype(np.int64)
    gaps = np.cumsum(rng.integers(1, 5, size=rp[-1]))
    col = gaps - np.repeat(np.concatenate(([0], gaps))[rp[:-1]], lengths)
    return tuple(torch.from_numpy(t).cuda() for t in (rp, col.astype(np.int32), rng.standard_normal(rp[-1])))


class _Sum:
    """The steps of one sum by the C calls, with a workspace of the caller's."""

    def __init__(self, B, x, y):
        import ctypes
        self.B, self.x, self.y, self.m = B, x, y, x[0].numel() - 1
        self.rowptr, self.bytes, self.nnz = torch.empty_like(x[0]), ctypes.c_size_t(0), ctypes.c_int64(0)
        assert self._call(None, None, None, None) == 0

    def _call(self, col, val, ws, stream):
        import ctypes
        p = self.B._p
        return self.B._lib.spsyrk_accumulate(self.m, 0, self.x[1].numel(), *map(p, self.x), self.y[1].numel(), *map(p, self.y), p(self.rowptr), p(col),
                                             p(val), ctypes.byref(self.nnz), p(ws), ctypes.byref(self.bytes), self.B._stream(stream))

    def sizes(self, ws):
        assert self._call(None, None, ws, None) == 0
        self.out = (torch.full((self.nnz.value,), -1, dtype=torch.int32, device="cuda"), torch.full((self.nnz.value,), -1.0, dtype=torch.float64, device="cuda"))

    def fill(self, ws, stream=None):
        assert self._call(*self.out, ws, stream) == 0

    def check(self):
        expected = self.B.spsyrk_accumulate(self.m, *self.x, *self.y)
        assert torch.equal(self.rowptr, expected[0]) and torch.equal(self.out[0], expected[1]) and torch.equal(self.out[1], expected[2])


def _sum(B, kind, seed):
    rng = np.random.default_rng(seed)
    m = 60_000 if kind == "short" else 6000
    def rows():
        lengths = rng.integers(0, 9, size=m) if kind == "short" else rng.integers(20, 300, size=m)
        lengths[rng.integers(0, m, 40)] = rng.integers(2000, 9000, 40)  # some of them long
        return lengths
    return _Sum(B, _device_csr(rows(), seed), _device_csr(rows(), seed + 1))


@pytest.mark.parametrize("kind", ["short", "wide"])
def test_fill_leaves_the_workspace_alone(B, kind):
    """What the size step left there is gone and something else stands in its place: the fill does not read it and does not write it."""
    s = _sum(B, kind, 11)
    ws = B._workspace(s.bytes.value, torch.device("cuda"))
    s.sizes(ws)
    ws.fill_(0x5a)
    s.fill(ws)
    s.check()
    assert bool((ws == 0x5a).all())


@pytest.mark.parametrize("kind", ["short", "wide"])
def test_two_fills_with_one_workspace(B, kind):
    sums = [_sum(B, kind, 21), _sum(B, kind, 31)]
    ws = B._workspace(max(s.bytes.value for s in sums), torch.device("cuda"))
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    for s in sums:
        s.sizes(ws)
    torch.cuda.synchronize()
    for _ in range(5):
        for s, st in zip(sums, streams):
            s.fill(ws, st)
    torch.cuda.synchronize()
    for s in sums:
        s.check()


def test_fill_on_another_stream_beside_new_tensors(B):
    """The workspace that the binding allocates is given up when the call returns, with the fill under way on another stream."""
    s = _sum(B, "wide", 41)
    expected = B.spsyrk_accumulate(s.m, *s.x, *s.y)
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    for _ in range(5):
        got = B.spsyrk_accumulate(s.m, *s.x, *s.y, stream=side)
        others = [torch.full((s.bytes.value,), 0x5a, dtype=torch.uint8, device="cuda") for _ in range(3)]
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(got, expected))
        del others, got
