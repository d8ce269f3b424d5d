"""A kernel that does not start makes its call fail: every launch of a call in turn is refused by a stand-in for the CUDA
runtime, on the host (kernels do not run, device memory is host memory)."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

RUNTIME = r"""
#include <cstdlib>
#include <cstring>
typedef int err_t;
struct dim3_t { unsigned x, y, z; };
static long launches, refused = -1;
static int last_error;

static int launch() {
    if (launches++ != refused) return 0;
    return last_error = 701;  // too many resources requested for launch
}
extern "C" {
void fake_refuse(long n) { launches = 0; refused = n; last_error = 0; }
long fake_launches() { return launches; }
err_t cudaLaunchKernel(const void*, dim3_t, dim3_t, void**, size_t, void*) { return launch(); }
err_t cudaLaunchKernelExC(const void*, const void*, void**) { return launch(); }
err_t cudaGetLastError() { const int e = last_error; last_error = 0; return e; }
err_t cudaHostAlloc(void** p, size_t n, unsigned) { *p = std::calloc(1, n); return 0; }
err_t cudaHostGetDevicePointer(void** d, void* h, unsigned) { *d = h; return 0; }
err_t cudaFreeHost(void* p) { std::free(p); return 0; }
err_t cudaMalloc(void** p, size_t n) { *p = std::calloc(1, n); return 0; }
err_t cudaFree(void* p) { std::free(p); return 0; }
err_t cudaMemsetAsync(void* p, int v, size_t n, void*) { std::memset(p, v, n); return 0; }
err_t cudaMemcpyAsync(void* d, const void* s, size_t n, int, void*) { std::memcpy(d, s, n); return 0; }
err_t cudaStreamSynchronize(void*) { return 0; }
err_t cudaStreamCreate(void** s) { *s = nullptr; return 0; }
err_t cudaStreamDestroy(void*) { return 0; }
err_t cudaStreamWaitEvent(void*, void*, unsigned) { return 0; }
err_t cudaEventCreate(void** e) { *e = nullptr; return 0; }
err_t cudaEventCreateWithFlags(void** e, unsigned) { *e = nullptr; return 0; }
err_t cudaEventDestroy(void*) { return 0; }
err_t cudaEventElapsedTime(float* t, void*, void*) { *t = 0; return 0; }
err_t cudaEventQuery(void*) { return 0; }
err_t cudaEventRecord(void*, void*) { return 0; }
err_t cudaEventSynchronize(void*) { return 0; }
err_t cudaGetDevice(int* d) { *d = 0; return 0; }
err_t cudaDeviceGetAttribute(int* v, int, int) { *v = 148; return 0; }
err_t cudaFuncGetAttributes(void* a, const void*) { std::memset(a, 0, 16); return 0; }
err_t cudaFuncSetAttribute(const void*, int, int) { return 0; }
err_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) { *n = 1; return 0; }
err_t cudaGetSymbolAddress(void** p, const void*) { *p = std::calloc(1, 16u << 20); return 0; }
static struct { dim3_t g, b; size_t s; void* st; } pushed;
unsigned __cudaPushCallConfiguration(dim3_t g, dim3_t b, size_t s, void* st) { pushed = {g, b, s, st}; return 0; }
err_t __cudaPopCallConfiguration(dim3_t* g, dim3_t* b, size_t* s, void* st) {
    *g = pushed.g; *b = pushed.b; *s = pushed.s; *(void**)st = pushed.st;
    return 0;
}
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, void*, void*, void*, void*, int*) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
}
"""

# Calls that get as far with kernels that do nothing; each prints its number of launches and those whose refusal it did not report
CALLS = r"""
import ctypes, sys
fake, lib = ctypes.CDLL(sys.argv[1]), ctypes.CDLL(sys.argv[2])
i64, vp = ctypes.c_int64, ctypes.c_void_p
fake.fake_launches.restype = ctypes.c_long
keep = []
def mem(n):
    keep.append(ctypes.create_string_buffer(n + 256))
    at = ctypes.addressof(keep[-1])
    return vp((at + 255) // 256 * 256)
m, n, nnz = 5000, 70_000, 40_000
rp, ci, cv = mem(8 * (m + 1)), mem(4 * nnz), mem(8 * nnz)

def plan(mode, rows=m):
    sz = ctypes.c_size_t(0)
    args = lambda h, ws: (h, i64(m), i64(n), i64(nnz), rp, ci, cv, 0, mode, i64(0), i64(rows), ws, ctypes.byref(sz), None)
    assert lib.spsyrk_plan(*args(None, None)) == 0
    ws, h = mem(sz.value), vp()
    return lambda: lib.spsyrk_plan(*args(ctypes.byref(h), ws)), h

def with_plan(mode, f):
    call, h = plan(mode)
    assert call() == 0
    return lambda: f(h)

def three_steps(f, out, fill):
    sz = ctypes.c_size_t(0)
    assert f(None, None, None, ctypes.byref(sz)) == 0
    ws = mem(sz.value)
    return lambda: f(*(out if fill else (None, None)), ws, ctypes.byref(sz))

total = i64(0)
col, val, rowptr = mem(8 * nnz), mem(16 * nnz), mem(8 * (m + 1))
mirror = lambda rows, dt: lambda c, v, ws, sz: lib.spsyrk_mirror(i64(rows), i64(nnz), dt, mem(8 * (rows + 1)), ci, cv, mem(8 * (rows + 1)), c, v, ctypes.byref(total), ws, sz, None)
def accumulate(nx):
    return lambda c, v, ws, sz: lib.spsyrk_accumulate(i64(m), 0, i64(nx), rp, ci, cv, i64(nx), rp, ci, cv, rowptr, c, v, ctypes.byref(total), ws, sz, None)
CALLS = {
    "plan": plan(0)[0], "plan full": plan(1)[0], "plan of no rows": plan(0, 0)[0],
    "set_rows": with_plan(0, lambda h: lib.spsyrk_plan_set_rows(h, i64(3), i64(4000), None)),
    "set_rows full": with_plan(1, lambda h: lib.spsyrk_plan_set_rows(h, i64(3), i64(4000), None)),
    "set_block": with_plan(1, lambda h: lib.spsyrk_plan_set_block(h, i64(3), i64(4000), i64(5), i64(4500), None)),
    "symbolic": with_plan(0, lambda h: lib.spsyrk_symbolic(h, rowptr, ctypes.byref(total), None)),
    "symbolic full": with_plan(1, lambda h: lib.spsyrk_symbolic(h, rowptr, ctypes.byref(total), None)),
    "one pass slots": with_plan(0, lambda h: lib.spsyrk_onepass_slots(h, ctypes.byref(total), None)),
    "partition": with_plan(0, lambda h: lib.spsyrk_plan_partition(h, i64(4), (i64 * 5)(), None)),
    "permute": three_steps(lambda c, v, ws, sz: lib.spsyrk_permute(i64(m), i64(n), i64(nnz), 0, rp, ci, cv, mem(4 * m), None, rowptr, c, v, ws, sz, None), (col, val), True),
    "column panel": three_steps(lambda c, v, ws, sz: lib.spsyrk_column_panel(i64(m), i64(nnz), 0, rp, ci, cv, i64(0), i64(9), rowptr, c, v, ctypes.byref(total), ws, sz, None), None, False),
    "mirror row pointers": lambda: lib.spsyrk_mirror_rowptr_noalloc(i64(m), rp, ci, rowptr, ctypes.byref(total), None),
    "symv": lambda: lib.spsyrk_symv(i64(m), i64(nnz), 0, rp, ci, cv, col, val, None),
    "symm": lambda: lib.spsyrk_symm(i64(m), i64(3), i64(nnz), 0, rp, ci, cv, mem(24 * m), mem(24 * m), None),
    "mirror sizes": three_steps(mirror(5000, 0), None, False),
}
for rows, dt in ((5000, 0), (5000, 1), (300_000, 0), (300_000, 1), (40_000, 1)):
    CALLS[f"mirror {rows} {dt}"] = three_steps(mirror(rows, dt), (col, val), True)
for nx in (10_000, 300_000):
    CALLS[f"sum sizes {nx}"] = three_steps(accumulate(nx), None, False)
    CALLS[f"sum {nx}"] = three_steps(accumulate(nx), (col, val), True)
for name, call in CALLS.items():
    fake.fake_refuse(ctypes.c_long(-1))
    assert call() == 0, name
    launches = fake.fake_launches()
    lost = []
    for k in range(launches):
        fake.fake_refuse(ctypes.c_long(k))
        if call() != 6:
            lost.append(k)
    print(name, launches, lost, sep="|")
"""


@pytest.fixture(scope="module")
def outcomes(tmp_path_factory):
    from paper_2608_09713_b200 import build
    lib = build.build_cuda()
    d = tmp_path_factory.mktemp("runtime")
    (d / "fake.cpp").write_text(RUNTIME)
    fake = str(d / "libfake.so")
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-w", "-shared", "-fPIC", "-o", fake, str(d / "fake.cpp")])
    out = subprocess.run([sys.executable, "-c", CALLS, fake, lib], env=dict(os.environ, LD_PRELOAD=fake), capture_output=True, text=True, timeout=600)
    assert out.returncode == 0, out.stdout[-2000:] + out.stderr[-2000:]
    return [line.split("|") for line in out.stdout.splitlines()]


def test_every_launch_that_fails_is_reported(outcomes):
    assert len(outcomes) > 15
    for name, launches, lost in outcomes:
        assert int(launches) > 0, name
        assert lost == "[]", f"{name}: launches {lost} of {launches} failed unnoticed"
