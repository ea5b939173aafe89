"""Which columns are heavy by default: the line, the budgets it applies to and
what the plan reports of it."""
from __future__ import annotations

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2010_08526_gb300 as spg  # noqa: E402


def columns(nrows, counts, g, vt=torch.float32):
    """Columns of counts[j] distinct rows in a run from a random start."""
    ptr = torch.zeros(counts.numel() + 1, dtype=torch.int64, device="cuda")
    ptr[1:] = torch.cumsum(counts, 0)
    col = torch.repeat_interleave(torch.arange(counts.numel(), device="cuda"), counts)
    start = torch.randint(0, nrows, (counts.numel(),), generator=g, device="cuda")
    rows = (start[col] + torch.arange(col.numel(), device="cuda") - ptr[col]) % nrows
    vals = torch.randint(1, 5, (col.numel(),), generator=g, device="cuda").to(vt)
    return spg.Csc(nrows, counts.numel(), ptr.int(), rows.int(), vals)


def operands(m, most, seed, k=600, n=500, per=40):
    """A product whose columns have up to min(m, most + a few hundred) rows and many products each."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    A = columns(m, torch.randint(1, most, (k,), generator=g, device="cuda"), g)
    B = columns(k, torch.randint(0, per, (n,), generator=g, device="cuda"), g)
    return A, B


def info_at(A, B, budget, **kw):
    plan = spg.Plan(A, B, budget=budget, **kw)
    try:
        return plan.symbolic()
    except spg.SpgemmError as e:
        return dict(status=e.status, heavy_columns=0)
    finally:
        plan.close()


def line_budget(A, B):
    """(lo, hi): the default line applies at hi bytes and not at lo, 4 KiB below."""
    lo, hi = 1 << 20, 1 << 34
    assert info_at(A, B, hi)["heavy_columns"] > 0 and info_at(A, B, lo)["heavy_columns"] == 0
    while hi - lo > 4096:
        mid = (lo + hi) // 2
        if info_at(A, B, mid)["heavy_columns"] > 0:
            hi = mid
        else:
            lo = mid
    return lo, hi


@pytest.mark.parametrize("m", [5000, 40000])
def test_repeated_symbolic_steps_plan_the_same(m):
    """The workspace that one symbolic step leaves on a plan does not change the
    next one's heavy columns, batches or cap, at budgets around the one from
    which the default line applies."""
    A, B = operands(m, m // 2 if m < 8192 else 7000, m)
    if m > 8192:   # one B entry a column: no column above the fixed line
        g = torch.Generator(device="cuda")
        g.manual_seed(3)
        B = columns(B.nrows, torch.ones(8000, dtype=torch.int64, device="cuda"), g)
    lo, hi = line_budget(A, B)
    for budget in (lo, hi, hi + (64 << 10), hi + (1 << 20), hi + (32 << 20)):
        want = info_at(A, B, budget)
        plan = spg.Plan(A, B, budget=budget)
        for _ in range(3):
            try:
                got = plan.symbolic()
            except spg.SpgemmError as e:
                got = dict(status=e.status, heavy_columns=0)
            assert got == want, budget - hi
        plan.close()


@pytest.mark.parametrize("m,most,k", [(5000, 2500, 600), (16000, 8000, 600), (40000, 12000, 600), (300000, 12000, 3000)])
@pytest.mark.parametrize("sort", [False, True])
def test_cap_per_batch_is_the_fixed_lines(m, most, k, sort):
    """No column above 8192 rows, some of them, in one panel and in several:
    the cap of a batch is the one of the 8192-row line, after a first and a
    second symbolic step."""
    A, B = operands(m, most, m, k=k, n=4 * k, per=20 if m == 5000 else 6)
    fixed = info_at(A, B, 1 << 34, sort_output=sort, tuning=spg.Tuning(hash_max_cap=8192))
    plan = spg.Plan(A, B, budget=1 << 34, sort_output=sort)
    for _ in range(2):
        info = plan.symbolic()
        assert info["heavy_columns"] > fixed["heavy_columns"]     # the lower line is in use
        assert info["batch_cap_bytes"] == fixed["batch_cap_bytes"]
    plan.close()


@pytest.mark.parametrize("m,vt,sizes,lower", [
    # columns of one size: by the mean multiplications (600 a B entry, n columns)
    (5000, torch.float32, [6], False), (5000, torch.float32, [7], True),
    (5000, torch.float64, [6], False), (5000, torch.float64, [7], True),
    (5000, torch.int64, [6], False), (5000, torch.int64, [7], True),
    # columns of several sizes, few products: 600 to 1,800 and 1,200 to 1,800
    (5000, torch.float32, [1, 1, 3], True), (5000, torch.float32, [2, 3], False),
    # several panels: 4-byte values up to 2^19 rows, 8-byte ones up to two panels, and
    # doubles of several sizes up to 2^16 rows
    (40000, torch.float64, [6, 6, 22], True), (40000, torch.int64, [6, 6, 22], False),
    (65537, torch.float64, [6, 6, 22], False),
    (40000, torch.float32, [8], True), (40000, torch.float64, [8], False), (40000, torch.int64, [8], False),
    (16384, torch.float64, [8], True), (16385, torch.float64, [8], False),
    ((1 << 19) + 1, torch.float32, [8], False)])
def test_lower_line_where_it_pays(m, vt, sizes, lower):
    """The lower line is taken by how the multiplications of the columns above it
    spread, by their mean and total, the value width and the panels; C is the
    same either way. Few and many columns (both binning kernels)."""
    for n in (6000, 17000):
        g = torch.Generator(device="cuda")
        g.manual_seed(m)
        k = 64
        A = columns(m, torch.full((k,), 600 if m < 8192 else 700, device="cuda"), g, vt)
        B = columns(k, torch.tensor(sizes, device="cuda").repeat(n // len(sizes)), g, vt)
        out = []
        for tuning in (None, spg.Tuning(hash_max_cap=8192)):
            plan = spg.Plan(A, B, budget=1 << 36, sort_output=True, tuning=tuning)
            info = plan.symbolic()
            assert info["nbatches"] == 1
            out.append((info["heavy_columns"], info["batch_cap_bytes"], plan.numeric(0)))
            plan.check_errors()
            plan.close()
        (heavy, cap, C), (none, cap8, W) = out
        assert (heavy > none) == lower and cap == cap8
        assert torch.equal(C.colptr, W.colptr) and torch.equal(C.rowidx, W.rowidx) and torch.equal(C.vals, W.vals)


def test_few_products_in_all_do_not_lower_the_line():
    """Columns of 4,200 products each, 300 of them."""
    g = torch.Generator(device="cuda")
    g.manual_seed(10)
    A = columns(5000, torch.full((64,), 600, device="cuda"), g)
    B = columns(64, torch.full((300,), 7, device="cuda"), g)
    assert info_at(A, B, 1 << 36)["heavy_columns"] == 0


def test_a_few_hubs_do_not_lower_the_line():
    """Ten columns of a million products among a thousand of 1,500."""
    g = torch.Generator(device="cuda")
    g.manual_seed(9)
    m, k, n = 5000, 2000, 1010
    A = columns(m, torch.full((k,), 500, device="cuda"), g)
    counts = torch.full((n,), 3, device="cuda")
    counts[::101] = k
    info = info_at(A, columns(k, counts, g), 1 << 36)
    assert info["flops"] == 500 * (3 * (n - 10) + 10 * k) and info["heavy_columns"] == 0
