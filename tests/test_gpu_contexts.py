"""Calls before and after cudaDeviceReset: what the library keeps between calls
belongs to a context and must not be used in the next one. Each test runs in a
process of its own, on memory from the CUDA runtime (PyTorch's own state does
not survive the reset)."""
from __future__ import annotations

import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HEAD = r"""
import ctypes, sys
import numpy as np
from paper_2010_08526_gb300 import _capi as C
lib = C.load()
rt = ctypes.CDLL("libcudart.so.13")

def ok(e):
    assert e == 0, e

def dev(a):
    a = np.ascontiguousarray(a)
    p = ctypes.c_void_p()
    ok(rt.cudaMalloc(ctypes.byref(p), ctypes.c_size_t(max(a.nbytes, 8))))
    ok(rt.cudaMemcpy(p, a.ctypes.data_as(ctypes.c_void_p), ctypes.c_size_t(a.nbytes), 1))
    return p.value

def host(p, n, dt):
    a = np.empty(n, dt)
    ok(rt.cudaMemcpy(a.ctypes.data_as(ctypes.c_void_p), ctypes.c_void_p(p), ctypes.c_size_t(a.nbytes), 2))
    return a

def csc(m, n, ptr, rows, vals, ptr_type=C.I32):
    return C.SpgemmCsc(m, n, 0 if rows is None else len(rows), dev(ptr), 0 if rows is None else dev(rows),
                       0 if rows is None else dev(vals), ptr_type, C.I32, C.F32)

M, N, PER = 50000, 900, 700            # 700 rows a column: tables above 48 KB
rng = np.random.default_rng(1)
start = rng.integers(0, M, N)
rows = ((start[:, None] + 3 * np.arange(PER)) % M).astype(np.int32)
vals = rng.integers(1, 9, (N, PER)).astype(np.float32)
ptr = (PER * np.arange(N + 1)).astype(np.int32)

def transposed():
    A = csc(M, N, ptr, rows.ravel(), vals.ravel())
    T = csc(N, M, np.zeros(M + 1, np.int32), np.zeros(N * PER, np.int32), np.zeros(N * PER, np.float32))
    C.check(lib.spgemm_transpose(ctypes.byref(A), ctypes.byref(T), None))
    tp = host(T.colptr, M + 1, np.int32)
    tr = host(T.rowidx, N * PER, np.int32)
    col = np.repeat(np.arange(M), np.diff(tp))
    order = np.lexsort((col, tr))
    want = np.lexsort((rows.ravel(), np.repeat(np.arange(N), PER)))
    assert np.array_equal(col[order], rows.ravel()[want])
    assert np.array_equal(host(T.vals, N * PER, np.float32)[order], vals.ravel()[want])
"""


def run(body):
    r = subprocess.run([sys.executable, "-c", HEAD + body + "\nprint('done')\n"], cwd=ROOT, capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0 and "done" in r.stdout, r.stdout + r.stderr


def test_transpose_after_a_reset():
    run("""
for _ in range(3):
    transposed()
    transposed()
    ok(rt.cudaDeviceReset())
""")


PRODUCT = """
def product():
    # six of A's columns a column: about 4,100 rows, tables of 128 KB
    A = csc(M, N, ptr, rows.ravel(), vals.ravel())
    n = 40
    pick = np.concatenate([rng.choice(N, 6, replace=False) for _ in range(n)]).astype(np.int32)
    B = csc(N, n, (6 * np.arange(n + 1)).astype(np.int32), pick, np.ones(6 * n, np.float32))
    o = C.SpgemmOpts()
    o.budget_bytes = 1 << 33
    o.kstages = 1
    o.sort_output = 1
    h = ctypes.c_void_p()
    C.check(lib.spgemm_plan_create(ctypes.byref(A), ctypes.byref(B), ctypes.byref(o), 1, None, ctypes.byref(h)))
    C.check(lib.spgemm_symbolic(h, None))
    info = C.SpgemmPlanInfo()
    C.check(lib.spgemm_plan_query(h, ctypes.byref(info)))
    out = csc(M, n, np.zeros(n + 1, np.int64), np.zeros(info.nnz_c, np.int32), np.zeros(info.nnz_c, np.float32), C.I64)
    C.check(lib.spgemm_numeric(h, 0, ctypes.byref(out), None))
    C.check(lib.spgemm_plan_check(h, None))
    C.check(lib.spgemm_plan_destroy(h))
    cp = host(out.colptr, n + 1, np.int64)
    r, v = host(out.rowidx, info.nnz_c, np.int32), host(out.vals, info.nnz_c, np.float32)
    for j in range(n):
        dense = np.zeros(M, np.float32)
        for k in pick[6 * j:6 * j + 6]:
            dense[rows[k]] += vals[k]
        where = np.flatnonzero(dense)
        assert np.array_equal(r[cp[j]:cp[j + 1]], where) and np.array_equal(v[cp[j]:cp[j + 1]], dense[where])
    # and the prune, whose selection stages 100 KB
    for fill in (False, True):
        if not fill:
            res = C.SpgemmCsc(M, n, 0, dev(np.zeros(n + 1, np.int64)), 0, 0, C.I64, C.I32, C.F32)
        else:
            res.rowidx, res.vals = dev(np.zeros(res.nnz, np.int32)), dev(np.zeros(res.nnz, np.float32))
        C.check(lib.spgemm_prune(ctypes.byref(out), ctypes.c_double(0.0), 100, ctypes.byref(res), None))
    pv = host(res.vals, res.nnz, np.float32)
    for j in range(n):
        assert np.array_equal(np.sort(pv[100 * j:100 * j + 100]), np.sort(v[cp[j]:cp[j + 1]])[-100:])
"""


def test_product_and_prune_after_a_reset():
    run(PRODUCT + """
for _ in range(3):
    product()
    ok(rt.cudaDeviceReset())
""")


def test_first_calls_of_several_threads():
    """Every thread waits until the kernels' limits are set."""
    run(PRODUCT + """
import threading
failed = []
gate = threading.Barrier(6)

def go():
    gate.wait()
    try:
        product()
    except BaseException as e:
        failed.append(e)

threads = [threading.Thread(target=go) for _ in range(6)]
[t.start() for t in threads]
[t.join() for t in threads]
assert not failed, failed
""")


def test_a_second_context_of_the_device():
    """A context of the caller's own beside the runtime's, and back."""
    run(PRODUCT + """
product()
transposed()
drv = ctypes.CDLL("libcuda.so.1")
mine, first = ctypes.c_void_p(), ctypes.c_void_p()
ok(drv.cuCtxGetCurrent(ctypes.byref(first)))
ok(drv.cuCtxCreate_v4(ctypes.byref(mine), None, 0, 0))
product()
transposed()
ok(rt.cudaDeviceSynchronize())
ok(drv.cuCtxSetCurrent(first))
product()
transposed()
ok(rt.cudaDeviceSynchronize())
ok(drv.cuCtxDestroy_v2(mine))
ok(drv.cuCtxSetCurrent(first))
product()
transposed()
""")


MERGE = """
def merged():
    n = 300
    parts = (C.SpgemmCsc * 2)(*[csc(M, n, ptr[:n + 1], rows[i * n:(i + 1) * n].ravel(), vals[i * n:(i + 1) * n].ravel())
                                for i in range(2)])
    out = C.SpgemmCsc(M, n, 0, dev(np.zeros(n + 1, np.int64)), 0, 0, C.I64, C.I32, C.F32)
    C.check(lib.spgemm_merge_noalloc(parts, 2, ctypes.byref(out), None))
    out.rowidx, out.vals = dev(np.zeros(out.nnz, np.int32)), dev(np.zeros(out.nnz, np.float32))
    C.check(lib.spgemm_merge_noalloc(parts, 2, ctypes.byref(out), None))
    cp = host(out.colptr, n + 1, np.int64)
    r, v = host(out.rowidx, out.nnz, np.int32), host(out.vals, out.nnz, np.float32)
    for j in range(n):
        dense = np.zeros(M, np.float32)
        for i in range(2):
            dense[rows[i * n + j]] += vals[i * n + j]
        got = np.zeros(M, np.float32)
        got[r[cp[j]:cp[j + 1]]] = v[cp[j]:cp[j + 1]]
        assert np.array_equal(got, dense) and cp[j + 1] - cp[j] == np.count_nonzero(dense)
"""


def test_merge_without_allocation_in_other_contexts():
    run(MERGE + """
merged()
drv = ctypes.CDLL("libcuda.so.1")
mine, first = ctypes.c_void_p(), ctypes.c_void_p()
ok(drv.cuCtxGetCurrent(ctypes.byref(first)))
ok(drv.cuCtxCreate_v4(ctypes.byref(mine), None, 0, 0))
merged()
ok(drv.cuCtxSetCurrent(first))
merged()
ok(drv.cuCtxDestroy_v2(mine))
ok(drv.cuCtxSetCurrent(first))
ok(rt.cudaDeviceReset())
merged()
""")
