"""The symbolic step's front end: multiplications per column, their total and
the column offsets, at the sizes where the scans change form (one tile, one
launch, folded partials, three launches) and for ragged columns of B (runs of
empty columns, one column of thousands of entries)."""
from __future__ import annotations

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2010_08526_gb300 as spg  # noqa: E402


def diagonal(n, it):
    i = torch.arange(n + 1, device="cuda", dtype=it)
    return spg.Csc(n, n, i, i[:n].clone(), torch.ones(n, device="cuda"))


@pytest.mark.parametrize("it", [torch.int32, torch.int64])
@pytest.mark.parametrize("n", [1, 31, 1024, 1025, 2047, 2048, 2049, 8192, 8193, 16384, 16385, 57344, 57345, 70001, (1 << 23) + 8191])
def test_offsets_and_flops_of_ragged_columns(n, it):
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    k = 4096
    counts = torch.randint(0, 4, (n,), generator=g, device="cuda")
    counts[torch.rand(n, generator=g, device="cuda") < 0.4] = 0
    counts[n // 3:n // 3 + 700] = 0
    counts[n // 2] = k                       # one long column
    ptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    ptr[1:] = torch.cumsum(counts, 0)
    nnz = int(ptr[-1])
    # rows of a column: consecutive from a random start, so they are distinct
    start = torch.randint(0, k, (n,), generator=g, device="cuda")
    start[n // 2] = 0
    col = torch.repeat_interleave(torch.arange(n, device="cuda"), counts)
    rows = (start[col] + torch.arange(nnz, device="cuda") - ptr[col]) % k
    B = spg.Csc(k, n, ptr.to(it), rows.to(it), torch.ones(nnz, device="cuda"))
    plan = spg.Plan(diagonal(k, it), B)
    info = plan.symbolic()
    assert info["flops"] == nnz and info["nnz_c"] == nnz
    assert torch.equal(plan.column_counts(), counts)
    for t in range(plan.nbatches):
        c0, c1, _ = plan.batch(t)
        C = plan.numeric(t)
        assert torch.equal(C.colptr, ptr[c0:c1 + 1] - ptr[c0])
    plan.check_errors()
    plan.close()


@pytest.mark.parametrize("ordered", [True, False])
@pytest.mark.parametrize("entries", [257, 383, 384, 385, 511, 512, 513, 5000])
def test_panel_copies_at_window_edges(entries, ordered):
    """Heavy columns read the panelised copies of A, built in windows of 128
    entries: totals around a window, runs cut by it, empty columns between."""
    rng = np.random.default_rng(entries)
    m = 6000
    counts = [0, 257, 0, 0, min(entries - 257, m - 1), 0]
    rows = [rng.permutation(m)[:c] for c in counts]
    if ordered:
        rows = [np.sort(r) for r in rows]
    ptr = np.concatenate([[0], np.cumsum(counts)])
    vals = rng.integers(1, 9, int(ptr[-1])).astype(np.float32)
    n = len(counts)

    def csc(nrows, ncols, p, r, v):
        t = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (p.astype(np.int32), r.astype(np.int32), v)]
        return spg.Csc(nrows, ncols, *t)

    A = csc(m, n, ptr, np.concatenate(rows), vals)
    B = csc(n, 1, np.array([0, n]), np.arange(n), np.ones(n, np.float32))     # the sum of all columns
    C = spg.spgemm(A, B, sort_output=True, tuning=spg.Tuning(hash_max_cap=256, panel_rows=1024))
    dense = np.zeros(m)
    np.add.at(dense, np.concatenate(rows), vals)
    where = np.flatnonzero(dense)
    assert np.array_equal(C.rowidx.cpu().numpy(), where)
    assert np.array_equal(C.vals.cpu().numpy(), dense[where].astype(np.float32))


@pytest.mark.parametrize("merge", ["end", "incremental"])
@pytest.mark.parametrize("stages", [1, 3])
def test_tier_counts_over_batches(stages, merge):
    """The tier populations of a batch are added up from blocks of 256 columns
    and single columns at its ends: batches cut anywhere, every hash tier."""
    n, m = 1500, 9000
    g = torch.Generator(device="cuda")
    g.manual_seed(stages)
    sizes = torch.tensor([0, 1, 33, 130, 300, 700, 1500, 3000, 5000], device="cuda")
    counts = sizes[torch.randint(0, 9, (n,), generator=g, device="cuda")]
    ptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    ptr[1:] = torch.cumsum(counts, 0)
    col = torch.repeat_interleave(torch.arange(n, device="cuda"), counts)
    start = torch.randint(0, m, (n,), generator=g, device="cuda")
    rows = (start[col] + torch.arange(col.numel(), device="cuda") - ptr[col]) % m
    vals = torch.randint(1, 9, (col.numel(),), generator=g, device="cuda").to(torch.float64)
    A = spg.Csc(m, n, ptr.int(), rows.int(), vals)
    i = torch.arange(n + 1, device="cuda").int()
    I = spg.Csc(n, n, i, i[:n].clone(), torch.ones(n, dtype=torch.float64, device="cuda"))
    whole = spg.spgemm(A, I, sort_output=True)
    probe = spg.Plan(A, I, budget=1 << 33, kstages=stages, merge=merge, sort_output=True)
    spent = (1 << 33) - 2 * probe.symbolic()["batch_cap_bytes"]
    probe.close()
    for cut in (3, 17):
        C = spg.spgemm(A, I, sort_output=True, kstages=stages, merge=merge,
                       budget=spent + 2 * max(12 * 5000 * 4, 24 * whole.nnz // cut))
        assert C.plan_info["nbatches"] > 1
        assert torch.equal(C.colptr, whole.colptr)
        assert torch.equal(C.rowidx, whole.rowidx) and torch.equal(C.vals, whole.vals)
    order = torch.sort(col * m + rows)
    assert torch.equal(whole.rowidx.long(), order.values % m) and torch.equal(whole.vals, vals[order.indices])


def ragged(m, n, seed, dtype=torch.int32):
    """Columns of 0, 1, 2 and a few hundred distinct rows."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    counts = torch.tensor([0, 0, 1, 2, 2, 300], device="cuda")[torch.randint(0, 6, (n,), generator=g, device="cuda")]
    ptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    ptr[1:] = torch.cumsum(counts, 0)
    col = torch.repeat_interleave(torch.arange(n, device="cuda"), counts)
    start = torch.randint(0, m, (n,), generator=g, device="cuda")
    rows = (start[col] + 7 * (torch.arange(col.numel(), device="cuda") - ptr[col])) % m
    vals = torch.randint(-9, 9, (col.numel(),), generator=g, device="cuda")
    return spg.Csc(m, n, ptr.to(dtype), rows.to(dtype), vals), col


def check_transpose(A, col, T):
    key, order = torch.sort(A.rowidx.long() * A.ncols + col)
    got = torch.repeat_interleave(torch.arange(A.nrows, device="cuda"), T.colptr.long().diff()) * A.ncols
    k2, o2 = torch.sort(got + T.rowidx.long())
    assert torch.equal(key, k2) and torch.equal(A.vals[order], T.vals[o2])


@pytest.mark.parametrize("m,n", [(1, 40), (31, 33), (5003, 4001), ((1 << 21) + 3, 900)])
def test_transpose_of_ragged_columns(m, n):
    """The last shape needs more scratch than the block kept between calls."""
    if m < 2200:
        col = torch.arange(n, device="cuda")
        A = spg.Csc(m, n, torch.arange(n + 1, device="cuda").int(), (col % m).int(), col.clone())
    else:
        A, col = ragged(m, n, m)
    check_transpose(A, col, spg.transpose(A))


def test_transposes_on_threads_and_streams():
    import threading
    work = [ragged(5003 + 100 * i, 3001, i) for i in range(4)]
    torch.cuda.synchronize()
    done = [None] * 4

    def go(i):
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            for _ in range(8):
                done[i] = spg.transpose(work[i][0])
            s.synchronize()

    threads = [threading.Thread(target=go, args=(i,)) for i in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for (A, col), T in zip(work, done):
        check_transpose(A, col, T)


@pytest.mark.parametrize("m,cols", [(1000, 5), (1000, 16500), (200000, 40), (200000, 1300), ((1 << 24) + 5000, 3)])
def test_item_lists_of_every_form(m, cols):
    """Heavy items cut by one CTA (one and several panels), by many CTAs with
    bins in shared memory, and with more bins than fit there."""
    g = torch.Generator(device="cuda")
    g.manual_seed(m + cols)
    count = 400
    start = torch.randint(0, m, (cols,), generator=g, device="cuda")
    step = torch.where(torch.arange(cols, device="cuda") % 2 == 0, 1, max(1, (m - 1) // count))
    rows = (start[:, None] + step[:, None] * torch.arange(count, device="cuda")[None, :]) % m
    vals = torch.randint(1, 9, (cols, count), generator=g, device="cuda").float()
    ptr = (torch.arange(cols + 1, device="cuda") * count).int()
    A = spg.Csc(m, cols, ptr, rows.reshape(-1).int(), vals.reshape(-1).contiguous())
    C = spg.spgemm(A, diagonal(cols, torch.int32), sort_output=True,
                   tuning=spg.Tuning(hash_max_cap=256, panel_rows=0 if m == 200000 else 1024))
    order = torch.sort(rows, dim=1)
    assert torch.equal(C.rowidx.long(), order.values.reshape(-1))
    assert torch.equal(C.vals, torch.gather(vals, 1, order.indices).reshape(-1))


@pytest.mark.parametrize("m", [900, 5000, 20000])
def test_heavy_rule_keeps_the_batch_plan(m):
    """Which columns are heavy depends on the row count by default; whatever the
    budget, the plan has the batches (or the refusal) of the fixed 8192-row line,
    and the product is the same."""
    n = 600
    g = torch.Generator(device="cuda")
    g.manual_seed(m)
    counts = torch.randint(1, m // 2, (n,), generator=g, device="cuda")
    ptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    ptr[1:] = torch.cumsum(counts, 0)
    col = torch.repeat_interleave(torch.arange(n, device="cuda"), counts)
    start = torch.randint(0, m, (n,), generator=g, device="cuda")
    rows = (start[col] + torch.arange(col.numel(), device="cuda") - ptr[col]) % m
    vals = torch.randint(1, 5, (col.numel(),), generator=g, device="cuda").double()
    A = spg.Csc(m, n, ptr.int(), rows.int(), vals)
    B, _ = ragged(n, 700, m)
    B = spg.Csc(n, 700, B.colptr, B.rowidx, B.vals.double())
    whole = spg.spgemm(A, B, sort_output=True, tuning=spg.Tuning(hash_max_cap=8192))
    need = 12 * whole.nnz
    batches = set()
    for budget in [1 << 20] + [int(need * f) + (60 << 20) for f in (0.2, 0.5, 1, 2, 4, 10, 40)]:
        seen = []
        for tun in (None, spg.Tuning(hash_max_cap=8192)):
            try:
                C = spg.spgemm(A, B, sort_output=True, budget=budget, tuning=tun)
            except spg.SpgemmError as e:
                seen.append(str(e.status))
                continue
            seen.append(C.plan_info["nbatches"])
            assert torch.equal(C.colptr, whole.colptr) and torch.equal(C.rowidx, whole.rowidx)
            assert torch.equal(C.vals, whole.vals)
        assert seen[0] == seen[1]
        batches.add(seen[0])
    assert len(batches) > 1


@pytest.mark.parametrize("vt", [torch.float32, torch.int64])
@pytest.mark.parametrize("stages,sort", [(1, True), (1, False), (3, True)])
def test_light_columns_with_many_short_segments(vt, stages, sort):
    """Columns of B around a warp's 32 entries and several rounds of them, over
    columns of A with 0 to 3 entries (empty segments between), every warp tier."""
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    m, k = 700, 2000
    ca = torch.randint(0, 4, (k,), generator=g, device="cuda")
    ap = torch.zeros(k + 1, dtype=torch.int64, device="cuda")
    ap[1:] = torch.cumsum(ca, 0)
    cola = torch.repeat_interleave(torch.arange(k, device="cuda"), ca)
    ra = (torch.randint(0, m, (k,), generator=g, device="cuda")[cola] + 11 * (torch.arange(cola.numel(), device="cuda") - ap[cola])) % m
    A = spg.Csc(m, k, ap.int(), ra.int(), torch.randint(1, 5, (cola.numel(),), generator=g, device="cuda").to(vt))
    cb = torch.tensor([0, 1, 5, 31, 32, 33, 63, 64, 65, 128, 200, 300], device="cuda").repeat(9)
    n = cb.numel()
    bp = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    bp[1:] = torch.cumsum(cb, 0)
    colb = torch.repeat_interleave(torch.arange(n, device="cuda"), cb)
    rb = (torch.randint(0, k, (n,), generator=g, device="cuda")[colb] + 3 * (torch.arange(colb.numel(), device="cuda") - bp[colb])) % k
    B = spg.Csc(k, n, bp.int(), rb.int(), torch.randint(1, 5, (colb.numel(),), generator=g, device="cuda").to(vt))
    C = spg.spgemm(A, B, sort_output=sort, kstages=stages, tuning=spg.Tuning(hash_max_cap=8192))
    da = torch.zeros(m, k, dtype=torch.float64, device="cuda")
    da[ra, cola] = A.vals.double()
    db = torch.zeros(k, n, dtype=torch.float64, device="cuda")
    db[rb, colb] = B.vals.double()
    want, reached = (da @ db).T, ((da != 0).double() @ (db != 0).double()).T > 0
    colc = torch.repeat_interleave(torch.arange(n, device="cuda"), C.colptr.diff())
    got = torch.zeros(n, m, dtype=torch.float64, device="cuda")
    got[colc, C.rowidx.long()] = C.vals.double()
    assert torch.equal(C.colptr.diff(), reached.sum(1)) and torch.equal(got, want)
    if sort:
        assert torch.equal(colc * m + C.rowidx, torch.nonzero(reached.reshape(-1)).reshape(-1))


@pytest.mark.parametrize("vt,it", [(torch.float32, torch.int32), (torch.float64, torch.int64)])
@pytest.mark.parametrize("kept", [1.0, 0.5, 0.0])
def test_backward_of_light_columns(vt, it, kept):
    """Short and empty segments, several rounds of 32 B entries, and a G that
    stores only some of C's entries; integer values, so the sums are exact."""
    g = torch.Generator(device="cuda")
    g.manual_seed(8)
    m, k = 600, 1500
    ca = torch.randint(0, 6, (k,), generator=g, device="cuda")
    ap = torch.zeros(k + 1, dtype=torch.int64, device="cuda")
    ap[1:] = torch.cumsum(ca, 0)
    cola = torch.repeat_interleave(torch.arange(k, device="cuda"), ca)
    ra = (torch.randint(0, m, (k,), generator=g, device="cuda")[cola] + 7 * (torch.arange(cola.numel(), device="cuda") - ap[cola])) % m
    A = spg.Csc(m, k, ap.to(it), ra.to(it), torch.randint(-4, 5, (cola.numel(),), generator=g, device="cuda").to(vt))
    cb = torch.tensor([0, 1, 7, 31, 32, 33, 64, 65, 150], device="cuda").repeat(9)
    n = cb.numel()
    bp = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    bp[1:] = torch.cumsum(cb, 0)
    colb = torch.repeat_interleave(torch.arange(n, device="cuda"), cb)
    rb = (torch.randint(0, k, (n,), generator=g, device="cuda")[colb] + 3 * (torch.arange(colb.numel(), device="cuda") - bp[colb])) % k
    B = spg.Csc(k, n, bp.to(it), rb.to(it), torch.randint(-4, 5, (colb.numel(),), generator=g, device="cuda").to(vt))
    C = spg.spgemm(A, B)
    col = torch.repeat_interleave(torch.arange(n, device="cuda"), C.colptr.diff())
    keep = torch.rand(C.nnz, generator=g, device="cuda") < kept
    gp = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    gp[1:] = torch.cumsum(torch.bincount(col[keep], minlength=n), 0)
    G = spg.Csc(m, n, gp, C.rowidx[keep].contiguous(), torch.randint(-4, 5, (int(keep.sum()),), generator=g, device="cuda").to(vt))
    dA, dB = spg.backward(A, B, G)
    da = torch.zeros(m, k, dtype=torch.float64, device="cuda")
    da[ra, cola] = A.vals.double()
    db = torch.zeros(k, n, dtype=torch.float64, device="cuda")
    db[rb, colb] = B.vals.double()
    dg = torch.zeros(m, n, dtype=torch.float64, device="cuda")
    dg[G.rowidx.long(), col[keep]] = G.vals.double()
    assert torch.equal(dA.double(), (dg @ db.T)[ra, cola])
    assert torch.equal(dB.double(), (da.T @ dg)[rb, colb])


@pytest.mark.parametrize("warp_cap,cap,threads", [(32, 256, 128), (128, 1024, 128), (256, 1024, 256), (512, 8192, 512)])
def test_batched_products_of_uneven_columns(warp_cap, cap, threads):
    """Warp and CTA items at every table size, short and empty segments, columns
    above the shared tables, and int64 sums that wrap and change sign."""
    g = torch.Generator(device="cuda")
    g.manual_seed(threads + cap)
    As, Bs, want = [], [], []
    for i, (m, k, n) in enumerate([(40, 50, 30), (900, 700, 300), (20000, 400, 60)]):
        A, cola = ragged(m, k, i + 3)
        A.vals.copy_(torch.randint(-(1 << 62), 1 << 62, (A.nnz,), generator=g, device="cuda"))
        B, colb = ragged(k, n, i + 13)
        keep = torch.rand(B.nnz, generator=g, device="cuda") < 0.7
        ptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
        ptr[1:] = torch.cumsum(torch.bincount(colb[keep], minlength=n), 0)
        # distinct (row, column) pairs only, as ragged() gives for k > 2100 rows
        key = torch.unique(B.rowidx[keep].long() + colb[keep] * k)
        colb, rb = key // k, key % k
        ptr[1:] = torch.cumsum(torch.bincount(colb, minlength=n), 0)
        B = spg.Csc(k, n, ptr.int(), rb.int(), torch.randint(-9, 9, (key.numel(),), generator=g, device="cuda"))
        keya = torch.unique(A.rowidx.long() + cola * m)
        cola, ra = keya // m, keya % m
        pa = torch.zeros(k + 1, dtype=torch.int64, device="cuda")
        pa[1:] = torch.cumsum(torch.bincount(cola, minlength=k), 0)
        A = spg.Csc(m, k, pa.int(), ra.int(), A.vals[:keya.numel()].contiguous())
        As.append(A)
        Bs.append(B)
        # products of every B entry, summed modulo 2^64 on the host's integers
        da = torch.zeros(k, m, dtype=torch.int64, device="cuda")
        da[cola, ra] = A.vals
        sa = torch.zeros(k, m, dtype=torch.bool, device="cuda")
        sa[cola, ra] = True
        c = torch.zeros(n, m, dtype=torch.int64, device="cuda")
        s = torch.zeros(n, m, dtype=torch.bool, device="cuda")
        for e in range(key.numel()):
            c[colb[e]] += da[rb[e]] * B.vals[e]
            s[colb[e]] |= sa[rb[e]]
        want.append((c, s))
    multi = spg.Multi(As, Bs, tuning=spg.Tuning(hash_max_cap=cap, warp_max_cap=warp_cap, block_tier_threads=threads))
    for _ in range(2):
        multi.run()
        colptr, rows, vals = multi.output()
        c0 = 0
        for (c, s), B in zip(want, Bs):
            ptr = colptr[c0:c0 + B.ncols + 1]
            assert torch.equal(ptr.diff(), s.sum(1))
            a, z = int(ptr[0]), int(ptr[-1])
            col = torch.repeat_interleave(torch.arange(B.ncols, device="cuda"), ptr.diff())
            got = torch.zeros_like(c)
            got[col, rows[a:z].long()] = vals[a:z]
            assert torch.equal(got, c)
            c0 += B.ncols
    multi.close()
