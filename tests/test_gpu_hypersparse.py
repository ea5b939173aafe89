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
