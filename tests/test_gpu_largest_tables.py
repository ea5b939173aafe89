"""Columns of the largest hash table (4097 to 8192 rows): the unsorted whole
product and the stages of a k-split walk them by different kernels, the
sorted product by a third route."""
from __future__ import annotations

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2010_08526_gb300 as spg  # noqa: E402


@pytest.mark.parametrize("vt,it", [(torch.float32, torch.int64), (torch.float64, torch.int32), (torch.int64, torch.int32)])
@pytest.mark.parametrize("kw", [dict(), dict(sort_output=True), dict(kstages=3), dict(semiring="or_and")])
def test_columns_of_the_largest_table(vt, it, kw):
    g = torch.Generator(device="cuda")
    g.manual_seed(6)
    m, k, n = 20000, 300, 40
    lens = torch.randint(0, 200, (k,), generator=g, device="cuda")
    lens[:4] = torch.tensor([4097, 8192, 8191, 5000], device="cuda")
    ptr = torch.zeros(k + 1, dtype=torch.int64, device="cuda")
    ptr[1:] = torch.cumsum(lens, 0)
    col = torch.repeat_interleave(torch.arange(k, device="cuda"), lens)
    rows = (torch.randint(0, m, (k,), generator=g, device="cuda")[col] + 2 * (torch.arange(col.numel(), device="cuda") - ptr[col])) % m
    A = spg.Csc(m, k, ptr.to(it), rows.to(it), torch.randint(1, 5, (col.numel(),), generator=g, device="cuda").to(vt))
    # columns of B: one of A's four long columns alone, and 30 to 70 short ones
    counts = torch.full((n,), 1, device="cuda")
    counts[4:] = torch.randint(30, 71, (n - 4,), generator=g, device="cuda")
    bp = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    bp[1:] = torch.cumsum(counts, 0)
    bcol = torch.repeat_interleave(torch.arange(n, device="cuda"), counts)
    brow = 4 + (torch.randint(0, k - 4, (n,), generator=g, device="cuda")[bcol] + torch.arange(bcol.numel(), device="cuda") - bp[bcol]) % (k - 4)
    brow[:4] = torch.arange(4, device="cuda")
    B = spg.Csc(k, n, bp.to(it), brow.to(it), torch.randint(1, 5, (brow.numel(),), generator=g, device="cuda").to(vt))
    C = spg.spgemm(A, B, tuning=spg.Tuning(hash_max_cap=8192), **kw)
    da = torch.zeros(k, m, dtype=torch.float64, device="cuda")
    da[col, rows] = A.vals.double()
    db = torch.zeros(n, k, dtype=torch.float64, device="cuda")
    db[bcol, brow] = B.vals.double()
    want = db @ da
    reached = want > 0
    if kw.get("semiring"):
        want = reached.double()
    assert torch.equal(C.colptr.diff(), reached.sum(1)) and int(C.colptr.diff().max()) == 8192
    assert int((C.colptr.diff() > 4096).sum()) > 8 and C.plan_info["heavy_columns"] == 0
    ccol = torch.repeat_interleave(torch.arange(n, device="cuda"), C.colptr.diff())
    got = torch.zeros(n, m, dtype=torch.float64, device="cuda")
    got[ccol, C.rowidx.long()] = C.vals.double()
    assert torch.equal(got, want)
    if kw.get("sort_output"):
        assert torch.equal(ccol * m + C.rowidx, torch.nonzero(reached.reshape(-1)).reshape(-1))
