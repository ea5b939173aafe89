"""Products whose entries or inner dimension reach 2^31: the kernels with 64-bit
offsets (k_sym_warp, k_sym_block, k_num_warp, k_num_block and k_bwd_warp on
products), which smaller products do not run. Columns of every hash tier, at
both ends of A, against dense sums; integer values, so the sums are exact."""
from __future__ import annotations

import pytest

pytestmark = [pytest.mark.gpu, pytest.mark.slow]

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2010_08526_gb300 as spg  # noqa: E402

M = 1 << 20                     # rows; a filler column holds them all
SIZES = [0, 1, 5, 33, 60, 130, 300, 700, 1500, 3000, 6000]


def small_columns(per, g):
    """(counts, rows, vals) of columns of the SIZES, `per` of each, distinct rows."""
    counts = torch.tensor(SIZES, device="cuda").repeat(per)
    counts = counts[torch.randperm(counts.numel(), generator=g, device="cuda")]
    ptr = torch.cumsum(counts, 0) - counts
    col = torch.repeat_interleave(torch.arange(counts.numel(), device="cuda"), counts)
    at = torch.arange(col.numel(), device="cuda") - ptr[col]
    rows = (torch.randint(0, M, (counts.numel(),), generator=g, device="cuda")[col] + 5 * at) % M
    return counts, col, rows, torch.randint(1, 5, (col.numel(),), generator=g, device="cuda")


def many_entries(vt, it, g):
    """Small columns before and behind 2048 full ones (2^31 entries; int32: 4096 fewer)."""
    counts, col, rows, vals = small_columns(4, g)
    short = counts.numel() // 2
    head = int(counts[:short].sum())
    full = 2048
    last = M if it == torch.int64 else M - 4096 - rows.numel()      # entries of the last full column
    filler = (full - 1) * M + last
    ai = torch.empty(rows.numel() + filler, dtype=it, device="cuda")
    av = torch.ones(ai.numel(), dtype=vt, device="cuda")
    ai[head:head + filler - last].view(full - 1, M)[:] = torch.arange(M, dtype=it, device="cuda")
    ai[head + filler - last:head + filler] = torch.arange(last, dtype=it, device="cuda")
    for part, to in ((slice(0, head), slice(0, head)), (slice(head, None), slice(head + filler, None))):
        ai[to] = rows[part].to(it)
        av[to] = vals[part].to(vt)
    lens = torch.cat([counts[:short], torch.full((full - 1,), M, device="cuda"),
                      torch.tensor([last], device="cuda"), counts[short:]])
    ap = torch.zeros(lens.numel() + 1, dtype=torch.int64, device="cuda")
    ap[1:] = torch.cumsum(lens, 0)
    assert int(ap[-1]) >= (1 << 31) - 8192
    ids = torch.cat([torch.arange(short, device="cuda"), torch.arange(short, counts.numel(), device="cuda") + full])
    entry = torch.arange(rows.numel(), device="cuda")
    entry[head:] += filler
    return spg.Csc(M, lens.numel(), ap.to(it), ai, av), ids, entry, (counts, col, rows, vals)


def many_columns(vt, it, g):
    """Small columns spread over 2^31 - 4000 mostly empty ones."""
    counts, col, rows, vals = small_columns(4, g)
    k = (1 << 31) - 4000
    ids = torch.arange(counts.numel(), device="cuda") * ((k - 1) // (counts.numel() - 1))
    ap = torch.zeros(k + 1, dtype=it, device="cuda")
    upto = torch.cumsum(counts, 0)
    for j in range(counts.numel()):
        ap[int(ids[j]) + 1:] = int(upto[j])
    return spg.Csc(M, k, ap, rows.to(it), vals.to(vt)), ids, torch.arange(rows.numel(), device="cuda"), (counts, col, rows, vals)


@pytest.mark.parametrize("make,vt,it", [(many_entries, torch.float32, torch.int64), (many_entries, torch.float32, torch.int32),
                                        (many_columns, torch.float64, torch.int32)])
def test_wide_products(make, vt, it):
    g = torch.Generator(device="cuda")
    g.manual_seed(11)
    A, ids, entry, (counts, col, rows, vals) = make(vt, it, g)
    k = ids.numel()
    # B: single columns, then up to 40 of the short and two longer ones (at most
    # 6,600 products: no heavy column)
    small = torch.nonzero(counts <= 130).reshape(-1)
    longer = torch.nonzero(counts <= 700).reshape(-1)
    lists = [[j] for j in range(k)]
    for n in (2, 7, 20, 33, 40):
        for _ in range(3):
            pick = small[torch.randperm(small.numel(), generator=g, device="cuda")[:n]].tolist()
            more = longer[torch.randint(0, longer.numel(), (2,), generator=g, device="cuda")].tolist()
            lists.append(sorted(set(pick + more)))
    bp = torch.tensor([0] + [len(x) for x in lists], device="cuda").cumsum(0)
    bk = torch.tensor([j for x in lists for j in x], device="cuda")
    bcol = torch.repeat_interleave(torch.arange(len(lists), device="cuda"), bp.diff())
    bv = torch.randint(1, 5, (bk.numel(),), generator=g, device="cuda")
    B = spg.Csc(A.ncols, len(lists), bp.to(it), ids[bk].to(it), bv.to(vt))
    dense_a = torch.zeros(k, M, dtype=torch.float64, device="cuda")
    dense_a[col, rows] = vals.double()
    dense_b = torch.zeros(len(lists), k, dtype=torch.float64, device="cuda")
    dense_b[bcol, bk] = bv.double()
    want = dense_b @ dense_a
    for sort, tuning in ((False, None), (True, None), (True, spg.Tuning(hybrid_sort=1))):
        plan = spg.Plan(A, B, budget=160 << 30, sort_output=sort, tuning=tuning)
        info = plan.symbolic()
        assert info["nbatches"] == 1 and info["heavy_columns"] == 0
        C = plan.numeric(0)
        plan.check_errors()
        ccol = torch.repeat_interleave(torch.arange(len(lists), device="cuda"), C.colptr.diff())
        assert torch.equal(C.colptr.diff(), (want > 0).sum(1))
        got = torch.zeros_like(want)
        got[ccol, C.rowidx.long()] = C.vals.double()
        assert torch.equal(got, want)
        if sort:
            assert bool((C.rowidx.long().diff()[ccol.diff() == 0] > 0).all())
        if sort and tuning is None:   # gradients, with a G that stores two entries of three
            keep = torch.rand(C.nnz, generator=g, device="cuda") < 0.67
            gp = torch.zeros(len(lists) + 1, dtype=torch.int64, device="cuda")
            gp[1:] = torch.cumsum(torch.bincount(ccol[keep], minlength=len(lists)), 0)
            gv = torch.randint(-4, 5, (int(keep.sum()),), generator=g, device="cuda")
            G = spg.Csc(M, len(lists), gp, C.rowidx[keep].contiguous(), gv.to(vt))
            assert int((gp.diff() <= 512).sum()) > 30 and int((gp.diff() > 512).sum()) > 5
            dA, dB = plan.backward(G)
            dense_g = torch.zeros_like(want)
            dense_g[ccol[keep], C.rowidx[keep].long()] = gv.double()
            assert torch.equal(dA[entry].double(), (dense_b.T @ dense_g)[col, rows])
            assert torch.equal(dB.double(), (dense_g @ dense_a.T)[bcol, bk])
            dA[entry] = 0
            assert not any(bool(x.any()) for x in dA.split(1 << 28))       # nothing anywhere else
        plan.close()


def test_wide_product_with_a_heavy_column():
    """A's panel copies, items and the generic heavy kernel with offsets past 2^31."""
    g = torch.Generator(device="cuda")
    g.manual_seed(12)
    A, ids, _, (counts, col, rows, vals) = many_entries(torch.float32, torch.int64, g)
    k = ids.numel()
    full = 2047 + k // 2                       # the last filler column: ones
    pick = torch.cat([ids[[0, 1, k - 2, k - 1]], torch.tensor([full], device="cuda")])
    B = spg.Csc(A.ncols, 1, torch.tensor([0, 5], device="cuda"), torch.sort(pick).values, torch.ones(5, device="cuda"))
    want = torch.ones(M, device="cuda")
    for j in (0, 1, k - 2, k - 1):
        want.index_add_(0, rows[col == j], vals[col == j].float())
    C = spg.spgemm(A, B, budget=200 << 30, sort_output=True)
    assert C.plan_info["heavy_columns"] == 1
    assert torch.equal(C.rowidx, torch.arange(M, device="cuda")) and torch.equal(C.vals, want)
