"""Sorted output of columns whose rows come in clusters far apart, so that many
rows share a bucket of the counting sort: on both sides of the lines from which
a warp's and a CTA's table goes to the bitonic network, and what it costs."""
from __future__ import annotations

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2010_08526_gb300 as spg  # noqa: E402

M = (1 << 31) - 1


def clustered(clusters, width, n, vt, spread=False):
    """n columns of `clusters` runs of `width` rows (or the same number, spread) and row M - 1."""
    g = torch.Generator(device="cuda")
    g.manual_seed(clusters * 1000 + width)
    if spread:
        gap = (M - 1) // (clusters * width)
        rows = torch.arange(clusters * width, device="cuda") * gap + torch.randint(
            0, gap, (n, clusters * width), generator=g, device="cuda")
    else:
        at = torch.arange(clusters, device="cuda") * ((M - 1) // clusters) // (1 << 20) * (1 << 20)
        rows = (at[None, :, None] + torch.randint(0, 300, (n, 1, 1), generator=g, device="cuda")
                + torch.arange(width, device="cuda")).reshape(n, -1)
    rows = torch.cat([rows, torch.full((n, 1), M - 1, device="cuda")], 1)
    rows = torch.gather(rows, 1, torch.rand(rows.shape, generator=g, device="cuda").argsort(1))   # any stored order
    vals = torch.randint(1, 1000, rows.shape, generator=g, device="cuda").to(vt)
    ptr = (torch.arange(n + 1, device="cuda") * rows.shape[1]).int()
    A = spg.Csc(M, n, ptr, rows.reshape(-1).int(), vals.reshape(-1).contiguous())
    i = torch.arange(n + 1, device="cuda", dtype=torch.int32)
    return A, spg.Csc(n, n, i, i[:n].clone(), torch.ones(n, device="cuda", dtype=vt)), rows, vals


@pytest.mark.parametrize("vt", [torch.float32, torch.float64, torch.int64])
@pytest.mark.parametrize("clusters,width", [
    (1, 127), (1, 128), (1, 129), (2, 130), (1, 511), (3, 128),             # warps
    (2, 255), (2, 256), (2, 257), (4, 500), (16, 500), (30, 256), (60, 129)])  # CTAs
def test_clusters_in_row_order(clusters, width, vt):
    A, I, rows, vals = clustered(clusters, width, 23, vt)
    order = rows.argsort(1)
    want_r, want_v = torch.gather(rows, 1, order).reshape(-1), torch.gather(vals, 1, order).reshape(-1)
    C = spg.spgemm(A, I, sort_output=True)
    assert torch.equal(C.rowidx.long(), want_r) and torch.equal(C.vals, want_v)


def test_pruned_clusters_in_row_order():
    """The kept columns of a stream go through the same sort."""
    A, I, rows, vals = clustered(2, 400, 40, torch.float32)
    plan = spg.Plan(A, I, budget=1 << 34, sort_output=True, prune=(0.0, 700))
    plan.symbolic()
    seen = []
    spg.run_batched(plan, lambda b, c0, c1, p: seen.append((c0, c1, p[0].copy(), p[1].copy(), p[2].copy())) and None)
    plan.close()
    for c0, c1, cp, ri, va in seen:
        for j in range(c0, c1):
            r, v = rows[j], vals[j]
            order = torch.argsort(r)
            r, v = r[order], v[order]
            keep = torch.sort(torch.argsort(v, descending=True, stable=True)[:700]).values
            a, z = cp[j - c0], cp[j - c0 + 1]
            assert ri[a:z].tolist() == r[keep].tolist() and va[a:z].tolist() == v[keep].tolist()


@pytest.mark.parametrize("clusters,width,n", [(1, 500, 40000), (2, 500, 20000)])
def test_clusters_cost_a_few_times_spread_rows(clusters, width, n):
    """Measured 2.8 times; ranking a whole cluster by counting takes 4.6 and 6.3 times."""
    best = []
    for spread in (False, True):
        A, I, _, _ = clustered(clusters, width, n, torch.float32, spread)
        plan = spg.Plan(A, I, budget=1 << 36, sort_output=True)
        plan.symbolic()
        C = plan.alloc_batch(0)
        times = []
        for _ in range(12):
            a, z = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            plan.numeric(0, C)
            z.record()
            z.synchronize()
            times.append(a.elapsed_time(z))
        best.append(min(times))
        plan.close()
    print(best)
    assert best[0] < 3.5 * best[1]
