"""The work users of this library have it do, as measurable cases.

Every case is one call (or one step) through the package's public entry
points on seeded synthetic matrices: the recipes and sizes are those of
workloads/generators.py, bench.py and the tests, drawn on the GPU. Products
return C with sorted columns (the paper's final form of C, Sec. IV-D), the
only form in which two runs of one product can be compared entry by entry;
the unsorted forms run inside the gradient step, the k-split's stages, the
pruned stream and the batched products.

A case is a dict of plain values:
  kind      which call (see run())
  graph     recipe of A: "er" (d distinct uniform rows per column), "paths"
            (binomial column counts of mean d), "rmat", "protein" (lognormal
            degrees of mean d) or "kmer" (2 rows per column)
  n, d      columns of A and entries per column (edge factor for "rmat")
  val, idx  value type ("f32", "f64", "i64") and index type ("i32", "i64")
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2010_08526_gb300 as spg

DEV = "cuda"
VAL = {"f32": torch.float32, "f64": torch.float64, "i64": torch.int64}
IDX = {"i32": torch.int32, "i64": torch.int64}
# fixed, so that the batch plan does not depend on what else holds memory
BUDGET = 96 << 30


def listed():
    return [
        # the smallest call: a 64 x 64 double product, as in gradient checks and
        # coarse levels; all latency (plan, launches, readbacks)
        dict(name="tiny_f64", kind="product", graph="er", n=64, d=8, val="f64", idx="i32"),
        # a small uniform product from scratch (benchmark configuration 1)
        dict(name="er4k_f64", kind="product", graph="er", n=4096, d=8, val="f64", idx="i32"),
        # counting 2-paths of one mid-sized graph, bit-exact (an element of configuration 4)
        dict(name="paths50k_i64", kind="plan", graph="paths", n=50021, d=16, val="i64", idx="i32"),
        # a batch of small graphs of uneven sizes, counted into dense matrices
        # (configuration 4's shape: one persistent pass in a CUDA graph)
        dict(name="multi64_i64", kind="multi", graph="paths", n=2000, nmin=500, count=64, d=32, val="i64", idx="i32"),
        # a skewed (social) graph of ordinary size: every column tier at once
        dict(name="rmat14_f32", kind="plan", graph="rmat", n=16384, d=16, val="f32", idx="i32"),
        # the headline workload's recipe at the largest size that fits three times over
        dict(name="rmat18_f32", kind="plan", graph="rmat", n=262144, d=16, val="f32", idx="i32"),
        # protein similarity (configuration 3): 64-bit indices, hardly any compression
        dict(name="protein100k_f32", kind="plan", graph="protein", n=100000, d=40, val="f32", idx="i64"),
        # inner dimension split into 4 stages with the hash merge (configuration 2's second half)
        dict(name="ksplit4_rmat15_f32", kind="plan", graph="rmat", n=30011, d=16, val="f32", idx="i32", stages=4),
        # 2-hop shortest distances on a skewed graph
        dict(name="minplus_rmat13_f64", kind="plan", graph="rmat", n=7919, d=12, val="f64", idx="i32",
             semiring="min_plus"),
        # overlap candidates: reads x k-mers times its transpose, shared k-mer counts
        dict(name="overlap_aat_i64", kind="aat", graph="kmer", n=400009, d=2, reads=40009, val="i64", idx="i64"),
        # a training step through A * B (configuration 5): forward and masked backward
        dict(name="fwdbwd_f32", kind="grad", graph="er", n=200000, d=16, cols=100000, db=8, val="f32", idx="i32"),
        # Markov clustering's expansion under a memory budget: column batches, pruned to
        # the largest entries of each column, sorted and streamed to the host
        dict(name="topk_stream_f32", kind="stream", graph="protein", n=20011, d=40, val="f32", idx="i64",
             topk=100, batches=4),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["product", "paths", "multi", "rmat", "protein", "ksplit", "semiring", "aat", "grad", "stream"])
    idx = rng.choice(["i32", "i64"])
    if kind == "product":
        return dict(kind="product", graph="er", n=_log(rng, 64, 30000), d=rng.randint(2, 16),
                    val=rng.choice(["f64", "f32", "i64"]), idx=idx)
    if kind == "paths":
        return dict(kind="plan", graph="paths", n=_log(rng, 1000, 200000), d=rng.randint(2, 32),
                    val=rng.choice(["i64", "f64"]), idx=idx)
    if kind == "multi":
        n = _log(rng, 1000, 6000)
        return dict(kind="multi", graph="paths", n=n, nmin=500, count=rng.randint(8, max(9, 60000 // n)),
                    d=rng.randint(8, 32), val="i64", idx=idx)
    if kind == "rmat":
        return dict(kind="plan", graph="rmat", n=_log(rng, 3000, 200000), d=rng.randint(6, 16),
                    val=rng.choice(["f32", "f32", "f64"]), idx=idx)
    if kind == "protein":
        return dict(kind="plan", graph="protein", n=_log(rng, 5000, 120000), d=rng.randint(10, 40),
                    val="f32", idx="i64")
    if kind == "ksplit":
        return dict(kind="plan", graph="rmat", n=_log(rng, 3000, 60000), d=rng.randint(6, 16),
                    val=rng.choice(["f32", "f64"]), idx=idx, stages=rng.choice([2, 3, 4, 7]))
    if kind == "semiring":
        return dict(kind="plan", graph="rmat", n=_log(rng, 2000, 60000), d=rng.randint(4, 16),
                    val=rng.choice(["f32", "f64"]), idx=idx, semiring=rng.choice(["min_plus", "or_and"]))
    if kind == "aat":
        n = _log(rng, 20000, 2000000)
        return dict(kind="aat", graph="kmer", n=n, d=2, reads=max(500, n // rng.randint(5, 40)), val="i64", idx=idx)
    if kind == "grad":
        n = _log(rng, 2000, 250000)
        return dict(kind="grad", graph="er", n=n, d=rng.randint(4, 24), cols=max(500, n // rng.randint(1, 4)),
                    db=rng.randint(2, 12), val=rng.choice(["f32", "f64"]), idx=idx)
    return dict(kind="stream", graph="protein", n=_log(rng, 5000, 30000), d=rng.randint(10, 40), val="f32",
                idx="i64", topk=rng.choice([10, 50, 100, 300]), batches=rng.randint(4, 7))


# ---------------------------------------------------------------- matrices
# The shape of a graph comes from the case alone (generator h); the seed
# (generator g) relabels its vertices and draws the values. So C has the same
# number of entries for every seed, at other places and with other values.
def _labels(n, g, within=None):
    """A random relabelling of n ids, inside runs of `within` ids if given."""
    key = torch.rand(n, generator=g, device=DEV, dtype=torch.float64)
    if within:
        key += torch.arange(n, device=DEV) // within
    return torch.argsort(key)


def _csc(nrows, ncols, cols, rows, vals, idx, ascending=False):
    """A Csc from its entries; rows ascending in each column, or in the order given."""
    cols, order = torch.sort(cols * nrows + rows if ascending else cols, stable=True)
    if ascending:
        cols = cols // nrows
    rows, vals = rows[order], vals[order]
    colptr = torch.zeros(ncols + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(torch.bincount(cols, minlength=ncols), 0, out=colptr[1:])
    it = IDX[idx]
    return spg.Csc(nrows, ncols, colptr.to(it), rows.to(it).contiguous(), vals.contiguous())


def _values(count, val, g, dist):
    if dist == "ones":
        return torch.ones(count, dtype=VAL[val], device=DEV)
    if val == "i64":
        return torch.randint(-3, 4, (count,), generator=g, device=DEV, dtype=torch.int64)
    f = torch.randn if dist == "normal" else torch.rand
    return f(count, generator=g, device=DEV, dtype=VAL[val])


def _distinct(nrows, counts, g):
    """(cols, rows): counts[j] distinct uniform rows of column j, in draw order."""
    cols = torch.repeat_interleave(torch.arange(counts.numel(), device=DEV), counts)
    rows = torch.randint(0, nrows, (cols.numel(),), generator=g, device=DEV)
    while True:
        key, order = torch.sort(cols * nrows + rows, stable=True)
        bad = order[1:][key[1:] == key[:-1]]
        if bad.numel() == 0:
            return cols, rows
        rows[bad] = torch.randint(0, nrows, (bad.numel(),), generator=g, device=DEV)


def _er(nrows, ncols, d, val, idx, h, g, dist):
    counts = torch.full((ncols,), min(d, max(1, nrows // 4)), dtype=torch.int64, device=DEV)
    cols, rows = _distinct(nrows, counts, h)
    to = _labels(nrows, g)
    cols = to[cols] if nrows == ncols else cols
    return _csc(nrows, ncols, cols, to[rows], _values(rows.numel(), val, g, dist), idx)


def _paths(n, d, val, idx, h, g):
    p = torch.full((n,), d / n, dtype=torch.float64, device=DEV)
    counts = torch.binomial(torch.full_like(p, float(n)), p, generator=h).to(torch.int64).clamp_(max=max(1, n // 4))
    cols, rows = _distinct(n, counts, h)
    to = _labels(n, g)
    return _csc(n, n, to[cols], to[rows], _values(rows.numel(), val, g, "ones"), idx)


def _rmat(n, ef, val, idx, h, g):
    """A = X + X^T of R-MAT edges (a=.57 b=c=.19), duplicates summed, without
    the vertices >= n of the enclosing power of two."""
    scale = max(1, (n - 1).bit_length())
    e = ef << scale
    r = torch.zeros(e, dtype=torch.int64, device=DEV)
    c = torch.zeros(e, dtype=torch.int64, device=DEV)
    for _ in range(scale):
        u = torch.rand(e, generator=h, device=DEV)
        r = 2 * r + (u >= 0.76)
        c = 2 * c + (((u >= 0.57) & (u < 0.76)) | (u >= 0.95))
    x = torch.rand(e, generator=g, device=DEV).to(torch.float64)   # exact sums in any order
    keep = (r < n) & (c < n)
    r, c, x = r[keep], c[keep], x[keep]
    to = _labels(n, g, within=64)   # the low ids stay the hubs, as R-MAT leaves them
    r, c = to[r], to[c]
    key, inv = torch.unique(torch.cat([c * n + r, r * n + c]), return_inverse=True)
    vals = torch.zeros(key.numel(), dtype=torch.float64, device=DEV).index_add_(0, inv, torch.cat([x, x]))
    return _csc(n, n, key // n, key % n, vals.to(VAL[val]), idx)


def _protein(n, d, val, idx, h, g):
    """Symmetric, lognormal degrees (mean d, sigma 1.2, cap 5000), Chung-Lu
    partners, similarities U(0.3, 1.0); a repeated pair keeps its largest."""
    z = torch.randn(n, generator=h, device=DEV, dtype=torch.float64)
    deg = torch.exp(math.log(d) - 0.72 + 1.2 * z).round_().clamp_(1, min(5000, n // 4)).to(torch.int64)
    src = torch.repeat_interleave(torch.arange(n, device=DEV), (deg + 1) // 2)
    cum = torch.cumsum(deg, 0)
    u = torch.rand(src.numel(), generator=h, device=DEV, dtype=torch.float64)
    dst = torch.searchsorted(cum, (u * cum[-1]).to(torch.int64), right=True).clamp_(max=n - 1)
    x = 0.3 + 0.7 * torch.rand(src.numel(), generator=g, device=DEV)
    keep = dst != src
    lo, hi, x = torch.minimum(src, dst)[keep], torch.maximum(src, dst)[keep], x[keep]
    key, inv = torch.unique(lo * n + hi, return_inverse=True)
    half = torch.zeros(key.numel(), device=DEV).scatter_reduce_(0, inv, x, "amax")
    to = _labels(n, g)
    lo, hi = to[key // n], to[key % n]
    return _csc(n, n, torch.cat([lo, hi]), torch.cat([hi, lo]), torch.cat([half, half]).to(VAL[val]), idx,
                ascending=True)


def _generators(case, seed):
    h, g = torch.Generator(device=DEV), torch.Generator(device=DEV)
    h.manual_seed(case["n"] * 64 + case["d"])
    g.manual_seed(seed)
    return h, g


def _matrix(case, h, g, dist="uniform"):
    n, d, val, idx = case["n"], case["d"], case["val"], case["idx"]
    if case["graph"] == "er":
        return _er(n, n, d, val, idx, h, g, dist)
    if case["graph"] == "paths":
        return _paths(n, d, val, idx, h, g)
    if case["graph"] == "rmat":
        return _rmat(n, d, val, idx, h, g)
    if case["graph"] == "protein":
        return _protein(n, d, val, idx, h, g)
    return _er(case["reads"], n, d, val, idx, h, g, "ones")   # kmer


# ---------------------------------------------------------------- the calls
def prepare(case, seed):
    h, g = _generators(case, seed)
    kind = case["kind"]
    st = dict(kind=kind)
    if kind == "multi":
        # sizes log-uniform in [nmin, n], degrees U(2, d), the same in every seed
        rng = np.random.default_rng(case["n"] * 1000 + case["count"])
        ns = np.rint(np.exp(rng.uniform(math.log(case["nmin"]), math.log(case["n"]), case["count"]))).astype(int)
        ds = rng.uniform(2, case["d"], case["count"])
        st["As"] = [_paths(int(a), float(b), case["val"], case["idx"], h, g) for a, b in zip(ns, ds)]
        st["multi"] = spg.Multi(st["As"], st["As"])
        # place of every column of every graph in the packed dense matrices
        n = torch.from_numpy(ns).to(DEV)
        place = torch.repeat_interleave(n, n)
        st["place"] = torch.cumsum(place, 0) - place
        st["size"] = int((ns.astype(np.int64) ** 2).sum())
    elif kind == "grad":
        st["A"] = _matrix(case, h, g, "normal")
        st["B"] = _er(case["n"], case["cols"], case["db"], case["val"], case["idx"], h, g, "normal")
        st["a"] = st["A"].vals.clone().requires_grad_()
        st["b"] = st["B"].vals.clone().requires_grad_()
    elif kind == "stream":
        A = st["A"] = _matrix(case, h, g)
        # steps of 1/128: sums are exact in any order, so the selection has one answer
        A.vals.mul_(128).round_().div_(128)
        probe = spg.Plan(A, A, budget=BUDGET, sort_output=True, prune=(0.0, case["topk"]))
        info = probe.symbolic()
        probe.close()
        # a device ring of two batches, each at most a `batches`-th of C
        spent = BUDGET - 2 * info["batch_cap_bytes"]
        whole = (info["nnz_c"] + A.ncols * case["topk"]) * info["bytes_per_nnz"] + 56 * A.ncols
        st["plan"] = spg.Plan(A, A, budget=spent + 2 * whole // case["batches"], sort_output=True,
                              prune=(0.0, case["topk"]), host_slot_bytes=64 << 20)
        room = A.ncols * case["topk"]
        st["colptr"] = np.zeros(A.ncols + 1, dtype=np.int64)
        st["rows"] = np.zeros(room, dtype=np.int64 if case["idx"] == "i64" else np.int32)
        st["vals"] = np.zeros(room, dtype=np.float32)
    else:
        A = st["A"] = _matrix(case, h, g)
        if kind == "plan":
            st["plan"] = spg.Plan(A, A, budget=BUDGET, kstages=case.get("stages", 1), sort_output=True,
                                  semiring=case.get("semiring", "plus_times"))
    return st


def run(st):
    kind = st["kind"]
    if kind == "product":           # one call from two matrices to C
        C = spg.spgemm(st["A"], st["A"], sort_output=True)
        return [C.colptr, C.rowidx, C.vals]
    if kind == "aat":
        C = spg.spgemm_aat(st["A"], sort_output=True)
        return [C.colptr, C.rowidx, C.vals]
    if kind == "plan":              # a kept plan: symbolic step, then every batch
        plan = st["plan"]
        plan.symbolic()
        out = []
        for t in range(plan.nbatches):
            C = plan.numeric(t)
            out += [C.colptr, C.rowidx, C.vals]
        return out
    if kind == "multi":             # all graphs in one pass, then dense counts per graph
        m = st["multi"]
        m.run()
        colptr, rows, vals = m.output()
        at = torch.repeat_interleave(st["place"], colptr.diff(), output_size=rows.numel()) + rows
        dense = torch.zeros(st["size"], dtype=vals.dtype, device=vals.device)
        dense[at] = vals
        return [colptr, dense]
    if kind == "grad":              # loss = |A B|^2 / 2, gradients of both operands' values
        st["a"].grad = st["b"].grad = None
        c = spg.SpGEMMFn.apply(st["a"], st["b"], st["A"], st["B"])
        loss = 0.5 * (c * c).sum()
        loss.backward()
        return [loss.detach(), st["a"].grad, st["b"].grad]
    plan, colptr, rows, vals = st["plan"], st["colptr"], st["rows"], st["vals"]
    end = 0

    def sink(batch, c0, c1, piece):
        nonlocal end
        cp, ri, va = piece
        rows[end:end + len(ri)] = ri
        vals[end:end + len(va)] = va
        colptr[c0 + 1:c1 + 1] = end + cp[1:]
        end += len(ri)

    plan.symbolic()
    spg.run_batched(plan, sink)
    return [colptr, rows[:end], vals[:end]]


# ---------------------------------------------------------------- bytes and flops
def _entry_bytes(M):
    return M.rowidx.element_size() + M.vals.element_size()


def _csc_bytes(M):
    return M.nnz * _entry_bytes(M) + (M.ncols + 1) * M.colptr.element_size()


def work(case):
    """Every input read once, every output written once; 2 operations a product."""
    st = prepare(case, 1)
    if case["kind"] == "multi":
        st["multi"].run()
        colptr, rows, vals = st["multi"].output()
        flops = 2 * sum(_flops(A, A) for A in st["As"])
        moved = sum(_csc_bytes(A) for A in st["As"]) + colptr.numel() * 8 + st["size"] * 8
        return {"bytes": moved, "flops": flops}
    A = st["A"]
    B = st["B"] if case["kind"] == "grad" else spg.transpose(A) if case["kind"] == "aat" else A
    B = spg.Csc(B.nrows, B.ncols, B.colptr.to(A.colptr.dtype), B.rowidx, B.vals)
    plan = spg.Plan(A, B, budget=BUDGET)
    nnz, flops = plan.symbolic()["nnz_c"], 2 * _flops(A, B)
    counts = plan.column_counts()
    plan.close()
    moved = _csc_bytes(A) + (_csc_bytes(B) if case["kind"] == "grad" else 0)
    if case["kind"] == "grad":      # the gradients; C is formed and read once by the backward
        moved += (A.nnz + B.nnz) * A.vals.element_size() + 2 * nnz * _entry_bytes(A)
        flops *= 3
    else:
        if case["kind"] == "stream":
            nnz = int(counts.clamp(max=case["topk"]).sum())
        moved += nnz * _entry_bytes(A) + (B.ncols + 1) * 8
    return {"bytes": moved, "flops": flops}


def _flops(A, B):
    return int(A.colptr.diff().to(torch.int64)[B.rowidx.to(torch.int64)].sum())


# ---------------------------------------------------------------- 64-bit values
def _products(A, B, most=150_000_000):
    """The products of A B in column chunks of at most `most`: (entry of A,
    entry of B, position of C's entry within the chunk, entries of C in the
    chunk); C's entries by ascending column, then row."""
    ap, bp = A.colptr.to(torch.int64), B.colptr.to(torch.int64)
    ai, bi = A.rowidx.to(torch.int64), B.rowidx.to(torch.int64)
    bcol = torch.repeat_interleave(torch.arange(B.ncols, device=DEV), bp.diff())
    size = ap.diff()[bi]
    upto = torch.zeros(B.nnz + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(size, 0, out=upto[1:])
    done = upto[bp].cpu()           # products before each column
    c = 0
    while c < B.ncols:
        z = max(c + 1, int(torch.searchsorted(done, done[c] + most, right=True)) - 1)
        e0, e1 = int(bp[c]), int(bp[z])
        pe = torch.repeat_interleave(torch.arange(e0, e1, device=DEV), size[e0:e1])
        q = torch.arange(pe.numel(), device=DEV) - (upto[pe] - int(done[c])) + ap[bi[pe]]
        key, order = torch.sort(bcol[pe] * A.nrows + ai[q])
        new = torch.ones_like(key, dtype=torch.bool)
        new[1:] = key[1:] != key[:-1]
        at = torch.cumsum(new, 0) - 1
        yield q[order], pe[order], at, int(new.sum())
        c = z


def exact(case, seed):
    if case["kind"] == "multi" or case["val"] == "i64" or case["kind"] == "stream":
        return None                 # whole numbers; or a selection, whose values C's own tests cover
    h, g = _generators(case, seed)
    A = B = _matrix(case, h, g, "normal" if case["kind"] == "grad" else "uniform")
    if case["kind"] == "grad":
        B = _er(case["n"], case["cols"], case["db"], case["val"], case["idx"], h, g, "normal")
    a, b = A.vals.double(), B.vals.double()
    semiring = case.get("semiring", "plus_times")
    vals = []
    da, db, loss = torch.zeros_like(a), torch.zeros_like(b), 0.0
    for q, pe, at, n in _products(A, B):
        if semiring == "min_plus":
            c = torch.full((n,), math.inf, dtype=torch.float64, device=DEV).scatter_reduce_(0, at, a[q] + b[pe], "amin")
        elif semiring == "or_and":
            both = ((a[q] != 0) & (b[pe] != 0)).double()
            c = torch.zeros(n, dtype=torch.float64, device=DEV).scatter_reduce_(0, at, both, "amax")
        else:
            c = torch.zeros(n, dtype=torch.float64, device=DEV).index_add_(0, at, a[q] * b[pe])
        if case["kind"] == "grad":
            loss = loss + 0.5 * (c * c).sum()
            da.index_add_(0, q, c[at] * b[pe])
            db.index_add_(0, pe, c[at] * a[q])
        else:
            vals.append(c)
    if case["kind"] == "grad":
        return [loss, da, db]
    return [None, None, torch.cat(vals)]
