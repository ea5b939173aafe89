"""Columns of the CTA tiers with table order: both ways the warps share a
column (rounds of B entries from 64 entries per warp on, else windows of every
round), at both sides of that line for each CTA size, with empty columns of A
among the entries and stages of k that skip entries. Values are small integers,
so every type compares exactly."""
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

ROWS = [513, 1000, 2000, 2049, 4000, 8000]            # distinct rows of a column of C
ENTRIES = [1, 2, 33, 255, 256, 511, 512, 545, 1023, 1024, 2047, 2048, 2081]   # entries of a column of B


@pytest.mark.parametrize("stages", [1, 3])
@pytest.mark.parametrize("vt,it", [(np.float32, np.int32), (np.int64, np.int64), (np.float64, np.int32)])
def test_cta_tiers_share_a_column(vt, it, stages):
    rng = np.random.default_rng(11)
    m = 20011
    shapes = [(r, e) for r in ROWS for e in ENTRIES]
    arows, brows, bptr = [], [], [0]
    for r, e in shapes:
        pool = rng.permutation(m)[:r]
        # e columns of A that cover the pool: every fifth one empty (when there
        # are enough), the others a share of it and a few rows twice
        used = [i for i in range(e) if e < 5 or i % 5 != 2]
        cols = [np.empty(0, np.int64)] * e
        for i, part in zip(used, np.array_split(pool, len(used))):
            cols[i] = np.unique(np.append(part, pool[rng.integers(0, r, 2)]))
        brows.append(len(arows) + rng.permutation(e))
        arows += cols
        bptr.append(bptr[-1] + e)
    aptr = np.concatenate([[0], np.cumsum([c.size for c in arows])])
    A = CSC(m, len(arows), aptr.astype(it), np.concatenate(arows).astype(it), rng.integers(1, 9, aptr[-1]).astype(vt))
    B = CSC(len(arows), len(shapes), np.array(bptr).astype(it), np.concatenate(brows).astype(it),
            rng.integers(1, 9, bptr[-1]).astype(vt))
    C = spg.spgemm(to_dev(A), to_dev(B), sort_output=False, kstages=stages)
    colptr, rows, vals = (x.cpu().numpy() for x in (C.colptr, C.rowidx, C.vals))
    for j, (r, e) in enumerate(shapes):
        want = np.zeros(m, vt)
        for q in range(bptr[j], bptr[j + 1]):
            k = int(B.rowidx[q])
            want[A.rowidx[aptr[k]:aptr[k + 1]]] += A.vals[aptr[k]:aptr[k + 1]] * B.vals[q]
        got_rows, got = rows[colptr[j]:colptr[j + 1]], vals[colptr[j]:colptr[j + 1]]
        order = np.argsort(got_rows)
        assert np.array_equal(got_rows[order], np.flatnonzero(want)), f"rows {r}, entries {e}"
        assert np.array_equal(got[order], want[np.flatnonzero(want)]), f"rows {r}, entries {e}"
