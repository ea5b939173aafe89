"""Transposes around the warp's windows of entries: columns cut by a window,
many columns in one, runs of empty columns, long columns of neighbouring rows."""
from __future__ import annotations

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2010_08526_gb300 as spg  # noqa: E402


def band(m, counts, it, vt=torch.int64):
    """Column j: counts[j] neighbouring rows from row 3 j on."""
    n = counts.numel()
    ptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    ptr[1:] = torch.cumsum(counts, 0)
    col = torch.repeat_interleave(torch.arange(n, device="cuda"), counts)
    rows = (3 * col + torch.arange(col.numel(), device="cuda") - ptr[col]) % m
    return spg.Csc(m, n, ptr.to(it), rows.to(it), torch.arange(col.numel(), device="cuda").to(vt)), col


@pytest.mark.parametrize("it", [torch.int32, torch.int64])
@pytest.mark.parametrize("counts", [
    [0, 1], [127], [128], [129], [0, 0, 31, 1, 0, 95, 2, 0, 0, 127, 129, 0], [1] * 128 + [0] * 500 + [1] * 129,
    [256, 0, 255, 1, 257], [5000], [2, 0] * 700, [0] * 100000 + [3] + [0] * 100000 + [200]])
def test_windows_of_entries(counts, it):
    A, col = band(6007, torch.tensor(counts, device="cuda"), it)
    T = spg.transpose(A)
    got = torch.repeat_interleave(torch.arange(A.nrows, device="cuda"), T.colptr.long().diff())
    a, oa = torch.sort(A.rowidx.long() * A.ncols + col)
    b, ob = torch.sort(got * A.ncols + T.rowidx.long())
    assert torch.equal(a, b) and torch.equal(A.vals[oa], T.vals[ob])


@pytest.mark.parametrize("extra", [-1, 0, 1, 200])
def test_windows_of_many_entries(extra):
    """Around the size from which a warp takes twice as many."""
    counts = torch.full(((1 << 22) // 64,), 64, device="cuda")
    counts[5] += extra if extra > 0 else 0
    counts[9] += extra if extra < 0 else 0
    A, col = band(300007, counts, torch.int32)
    T = spg.transpose(A)
    got = torch.repeat_interleave(torch.arange(A.nrows, device="cuda"), T.colptr.long().diff())
    a, oa = torch.sort(A.rowidx.long() * A.ncols + col)
    b, ob = torch.sort(got * A.ncols + T.rowidx.long())
    assert torch.equal(a, b) and torch.equal(A.vals[oa], T.vals[ob])
