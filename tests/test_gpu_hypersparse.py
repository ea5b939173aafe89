"""Matrices with long runs of empty columns (the blocks of a matrix spread over
many processes): results, and that a run costs the logarithm of its length and
not a step per column in one thread. The time limits are some hundred times
what the calls take, and half of what a step per column takes or less."""
from __future__ import annotations

import time

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2010_08526_gb300 as spg  # noqa: E402


def csc(m, n, counts, rows, vals, it):
    ptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(counts, 0, out=ptr[1:])
    return spg.Csc(m, n, ptr.to(it), rows.to(it), vals)


def seconds(call):
    call()
    torch.cuda.synchronize()
    t = time.perf_counter()
    call()
    torch.cuda.synchronize()
    return time.perf_counter() - t


@pytest.mark.parametrize("it", [torch.int32, torch.int64])
@pytest.mark.parametrize("places", [[0, 39_999_999], [39_999_999], [5, 6, 7, 8, 20_000_001, 20_000_002, 39_999_998]])
def test_flops_across_empty_columns(places, it):
    n, k = 40_000_000, 1000
    per = 9                                   # more than a thread's share of eight entries
    cols = torch.tensor(places, device="cuda")
    counts = torch.zeros(n, dtype=torch.int64, device="cuda")
    counts[cols] = per
    nnz = per * len(places)
    B = csc(k, n, counts, (torch.arange(nnz, device="cuda") * 7) % k, torch.ones(nnz, device="cuda"), it)
    lens = torch.arange(k, device="cuda") % 4
    first = torch.zeros(k + 1, dtype=torch.int64, device="cuda")
    first[1:] = torch.cumsum(lens, 0)
    rows = torch.arange(int(first[-1]), device="cuda") - torch.repeat_interleave(first[:-1], lens)
    rows = rows + 4 * torch.repeat_interleave(torch.arange(k, device="cuda"), lens)     # all distinct
    A = csc(4 * k, k, lens, rows, torch.ones(rows.numel(), device="cuda"), it)
    plan = spg.Plan(A, B, budget=1 << 36)
    assert seconds(plan.symbolic) < 0.5
    want = lens[B.rowidx.long()].reshape(len(places), per).sum(1)
    got = plan.column_counts()
    assert plan.info["flops"] == int(want.sum()) and int(got.sum()) == int(want.sum())
    assert torch.equal(got[cols], want)
    plan.close()


@pytest.mark.parametrize("it", [torch.int32, torch.int64])
@pytest.mark.parametrize("ordered", [True, False])
def test_panel_copies_across_empty_columns(ordered, it):
    """A product with a heavy column copies A by row panels: columns of one entry
    and of thousands, neighbours and 20,000,000 columns apart."""
    g = torch.Generator(device="cuda")
    g.manual_seed(4)
    ka, m = 40_000_000, 100_000
    cols = torch.tensor([0, 1, 2, 9, 20_000_000, 20_000_001, 39_999_990, 39_999_999], device="cuda")
    lens = torch.tensor([60_000, 1, 1, 3, 1, 30_000, 2, 60_000], device="cuda")
    counts = torch.zeros(ka, dtype=torch.int64, device="cuda")
    counts[cols] = lens
    rows = [torch.randperm(m, generator=g, device="cuda")[:int(x)] for x in lens]
    if ordered:
        rows = [torch.sort(r).values for r in rows]
    rows = torch.cat(rows)
    vals = torch.randint(1, 9, (rows.numel(),), generator=g, device="cuda").float()
    A = csc(m, ka, counts, rows, vals, it)
    scale = torch.arange(1, 9, device="cuda").float()
    B = csc(ka, 1, torch.tensor([8], device="cuda"), cols, scale, it)
    plan = spg.Plan(A, B, budget=1 << 36, sort_output=True)
    assert seconds(plan.symbolic) < 0.5
    assert plan.info["heavy_columns"] == 1
    C = plan.numeric(0)
    plan.check_errors()
    dense = torch.zeros(m, device="cuda").index_add_(0, rows, vals * torch.repeat_interleave(scale, lens))
    where = torch.nonzero(dense).reshape(-1)
    assert torch.equal(C.rowidx.long(), where) and torch.equal(C.vals, dense[where])
    plan.close()
