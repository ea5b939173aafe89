"""The top-k selection at the sizes where it changes form (a warp's 128 entries, a
CTA's step of 2048, the staged keys' limit) against the oracle, bit-exact:
spread, crowded, equal and special values."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from workloads.csc import CSC

from helpers import to_dev

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2010_08526_gb300 as spg  # noqa: E402

SIZES = [0, 1, 2, 31, 33, 127, 128, 129, 511, 513, 2047, 2048, 2049, 4097, 6143, 12799, 12800, 12801, 25599, 25600, 25601, 29000]


def values(rng, n, vt, kind):
    if kind == "spread":
        v = rng.standard_normal(n) * 10.0 ** rng.integers(-3, 4, n)
    elif kind == "crowded":
        v = rng.integers(0, 5, n) / 4.0
    elif kind == "equal":
        v = np.full(n, 3.0)
    else:
        v = rng.standard_normal(n)
        v[rng.random(n) < 0.1] = np.inf
        v[rng.random(n) < 0.1] = -np.inf
        v[rng.random(n) < 0.1] = 0.0
        v[rng.random(n) < 0.1] = np.nan
    if np.dtype(vt) == np.int64:
        if kind == "special":
            v = rng.choice(np.array([np.iinfo(np.int64).min, -1, 0, 1, np.iinfo(np.int64).max]), n)
            return v.astype(np.int64)
        return np.rint(v * 1000).astype(np.int64)
    return v.astype(vt)


@pytest.mark.parametrize("kind", ["spread", "crowded", "equal", "special"])
@pytest.mark.parametrize("vt", [np.float32, np.float64, np.int64])
@pytest.mark.parametrize("topk,thr", [(1, float("-inf")), (100, float("-inf")), (100, 0.25), (3000, -1.0), (0, 0.5)])
def test_prune_matches_oracle(kind, vt, topk, thr):
    rng = np.random.default_rng(topk + len(kind))
    m = 30000
    ptr = np.concatenate([[0], np.cumsum(SIZES)])
    rows = np.concatenate([rng.choice(m, s, replace=False) for s in SIZES] or [np.zeros(0)])
    A = CSC(m, len(SIZES), ptr.astype(np.int64), rows.astype(np.int64), values(rng, int(ptr[-1]), vt, kind))
    P = spg.prune(to_dev(A), threshold=thr, topk=topk)
    ref = oracle.prune(A, thr, topk)
    assert np.array_equal(P.colptr.cpu().numpy(), np.asarray(ref.colptr))
    assert np.array_equal(P.rowidx.cpu().numpy(), np.asarray(ref.rowidx))
    assert np.array_equal(P.vals.cpu().numpy(), np.asarray(ref.vals))
