"""B row indices outside [0, k) are skipped by the kernels (unvalidated input):
no product, no gradient and no access beyond A's arrays comes of them."""
from __future__ import annotations

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2010_08526_gb300 as spg  # noqa: E402


def random_csc(nrows, counts, g, vt, it):
    """Columns of counts[j] distinct rows; small integers, so sums are exact."""
    n = counts.numel()
    ptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    ptr[1:] = torch.cumsum(counts, 0)
    col = torch.repeat_interleave(torch.arange(n, device="cuda"), counts)
    at = torch.arange(col.numel(), device="cuda") - ptr[col]
    rows = (torch.randint(0, nrows, (n,), generator=g, device="cuda")[col] + 3 * at) % nrows
    vals = torch.randint(1, 5, (col.numel(),), generator=g, device="cuda").to(vt)
    return spg.Csc(nrows, n, ptr.to(it), rows.to(it), vals), col


def with_bad_rows(B, col, bad_values, g):
    """(B with a fifth of its row indices out of range, B without those entries, which they are)."""
    bad = torch.rand(B.nnz, generator=g, device="cuda") < 0.2
    rows = B.rowidx.clone()
    pick = torch.randint(0, len(bad_values), (B.nnz,), generator=g, device="cuda")
    rows[bad] = torch.tensor(bad_values, device="cuda").to(rows.dtype)[pick[bad]]
    ptr = torch.zeros(B.ncols + 1, dtype=torch.int64, device="cuda")
    ptr[1:] = torch.cumsum(torch.bincount(col[~bad], minlength=B.ncols), 0)
    clean = spg.Csc(B.nrows, B.ncols, ptr.to(B.colptr.dtype), B.rowidx[~bad].contiguous(), B.vals[~bad].contiguous())
    return spg.Csc(B.nrows, B.ncols, B.colptr, rows, B.vals), clean, bad


@pytest.mark.parametrize("vt,it", [(torch.float32, torch.int32), (torch.float64, torch.int64)])
def test_backward_skips_indices_out_of_range(vt, it):
    g = torch.Generator(device="cuda")
    g.manual_seed(21)
    m, k = 500, 401
    A, _ = random_csc(m, torch.randint(0, 6, (k,), generator=g, device="cuda"), g, vt, it)
    B, col = random_csc(k, torch.tensor([0, 1, 8, 31, 32, 33, 90], device="cuda").repeat(8), g, vt, it)
    broken, clean, bad = with_bad_rows(B, col, [-1, -(1 << 20), k, k + 1, (1 << 31) - 2], g)
    C = spg.spgemm(A, clean)
    G = spg.Csc(m, B.ncols, C.colptr, C.rowidx, torch.randint(-4, 5, (C.nnz,), generator=g, device="cuda").to(vt))
    assert int(C.colptr.diff().max()) <= 512     # the warp tiers
    want_a, want_b = spg.backward(A, clean, G)
    dA, dB = spg.backward(A, broken, G)
    assert torch.equal(dA, want_a)
    assert torch.equal(dB[~bad], want_b) and not dB[bad].any()
    D = spg.spgemm(A, broken, sort_output=True)  # the forward pass skips them too
    W = spg.spgemm(A, clean, sort_output=True)
    assert torch.equal(D.colptr, W.colptr) and torch.equal(D.rowidx, W.rowidx) and torch.equal(D.vals, W.vals)


def test_batched_products_skip_negative_indices():
    g = torch.Generator(device="cuda")
    g.manual_seed(22)
    As, Bs, Ws = [], [], []
    for m, k in ((40, 60), (900, 400)):
        A, _ = random_csc(m, torch.randint(0, 9, (k,), generator=g, device="cuda"), g, torch.int64, torch.int64)
        B, col = random_csc(k, torch.randint(0, 50, (70,), generator=g, device="cuda"), g, torch.int64, torch.int64)
        broken, clean, _ = with_bad_rows(B, col, [-1, -(1 << 20)], g)
        As.append(A)
        Bs.append(broken)
        Ws.append(clean)
    out = []
    for rhs in (Bs, Ws):
        multi = spg.Multi(As, rhs)
        multi.run()
        colptr, rows, vals = multi.output()
        col = torch.repeat_interleave(torch.arange(multi.total_cols, device="cuda"), colptr.diff())
        key, order = torch.sort(col * 1000 + rows)
        out.append((colptr.clone(), key, vals[order].clone()))
        multi.close()
    for a, b in zip(*out):
        assert torch.equal(a, b)
