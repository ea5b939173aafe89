"""Row order written by the hash tiers themselves (sort_output), at the sizes
where the table sort changes its form: one entry, a warp's 32 and 33, each
tier's capacity and one below and above it; spread-out rows, consecutive
rows, and a far outlier that puts all others into one bucket (the bitonic
fallback). Values are small integers, so every type compares exactly."""
from __future__ import annotations

import numpy as np
import pytest

from workloads.csc import CSC

from helpers import to_dev

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2010_08526_gb300 as spg  # noqa: E402

SIZES = [1, 2, 31, 32, 33, 63, 64, 65, 127, 128, 129, 255, 256, 257, 511, 512, 513, 1023, 1024, 1025, 2047, 2048,
         2049, 4096, 4097, 8191, 8192]


def column_rows(rng, m, count, layout):
    if layout == "spread":
        return rng.permutation(np.unique(np.append(rng.integers(0, m, 3 * count), np.arange(count)))[-count:])
    base = int(rng.integers(0, m - count - 1))
    rows = base + rng.permutation(count)
    if layout == "outlier":
        rows[rng.integers(0, count)] = m - 1
    return rows


@pytest.mark.parametrize("layout", ["spread", "run", "outlier"])
@pytest.mark.parametrize("m", [20011, (1 << 30) + 7])
@pytest.mark.parametrize("vt,it,semiring,stages", [
    (np.float32, np.int32, "plus_times", 1), (np.float64, np.int64, "plus_times", 2),
    (np.int64, np.int32, "plus_times", 1), (np.float64, np.int32, "min_plus", 1)])
def test_hash_tiers_write_ascending_rows(layout, m, vt, it, semiring, stages):
    rng = np.random.default_rng(len(SIZES) * m % 1000)
    n = len(SIZES)
    # columns j and n + j of A: the rows of C(:, j), and every other one of them again
    cols, vals = [], []
    for count in SIZES:
        cols.append(column_rows(rng, m, count, layout))
    for j in range(n):
        cols.append(cols[j][::2])
    vals = [rng.integers(1, 9, c.size) for c in cols]
    ptr = np.concatenate([[0], np.cumsum([c.size for c in cols])])
    A = CSC(m, 2 * n, ptr.astype(it), np.concatenate(cols).astype(it), np.concatenate(vals).astype(vt))
    one = 0 if semiring == "min_plus" else 1
    B = CSC(2 * n, n, (2 * np.arange(n + 1)).astype(it),
            np.stack([np.arange(n), n + np.arange(n)], 1).reshape(-1).astype(it), np.full(2 * n, one).astype(vt))
    C = spg.spgemm(to_dev(A), to_dev(B), sort_output=True, semiring=semiring, kstages=stages)
    colptr, rows, got = (x.cpu().numpy() for x in (C.colptr, C.rowidx, C.vals))
    assert np.array_equal(np.diff(colptr), SIZES)
    for j in range(n):
        want = dict(zip(cols[j].tolist(), vals[j].tolist()))
        for r, v in zip(cols[n + j].tolist(), vals[n + j].tolist()):
            want[r] = min(want[r], v) if semiring == "min_plus" else want[r] + v
        order = np.sort(cols[j])
        assert np.array_equal(rows[colptr[j]:colptr[j + 1]], order), f"column of {SIZES[j]}"
        assert np.array_equal(got[colptr[j]:colptr[j + 1]], np.array([want[r] for r in order.tolist()], dtype=vt))


@pytest.mark.parametrize("vt,it", [(np.float32, np.int32), (np.float64, np.int32), (np.int64, np.int64)])
@pytest.mark.parametrize("cap", [256, 8192])
def test_heavy_columns_write_ascending_rows(vt, it, cap):
    """Hash-range items over many sparse panels, some with clusters far from
    the rest (the bitonic fallback), between dense panels."""
    rng = np.random.default_rng(cap)
    m = 1 << 20
    cols = []
    for count in (257, 600, 3000, 8193, 20000):
        far = rng.integers(m // 2, m, count // 3)
        cluster = 300000 + np.arange(min(1500, count // 3))          # one bucket of a wide item
        near = rng.integers(0, 40000, count)                          # denser panels
        rows = np.unique(np.concatenate([far, cluster, near]))
        cols.append(rng.permutation(rows)[:count])
    ptr = np.concatenate([[0], np.cumsum([c.size for c in cols])])
    vals = [rng.integers(1, 9, c.size) for c in cols]
    n = len(cols)
    A = CSC(m, n, ptr.astype(it), np.concatenate(cols).astype(it), np.concatenate(vals).astype(vt))
    I = CSC(n, n, np.arange(n + 1).astype(it), np.arange(n).astype(it), np.ones(n, vt))
    C = spg.spgemm(to_dev(A), to_dev(I), sort_output=True, tuning=spg.Tuning(hash_max_cap=cap))
    colptr, rows, got = (x.cpu().numpy() for x in (C.colptr, C.rowidx, C.vals))
    for j in range(n):
        order = np.argsort(cols[j])
        assert np.array_equal(rows[colptr[j]:colptr[j + 1]], cols[j][order])
        assert np.array_equal(got[colptr[j]:colptr[j + 1]], vals[j][order].astype(vt))
