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
