"""The longest column there is, 2^31 - 1 rows, pruned: the places that the
selection steps to lie past 2^31. (17 GB of input, some twenty seconds.)"""
from __future__ import annotations

import pytest

pytestmark = [pytest.mark.gpu, pytest.mark.slow]

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2010_08526_gb300 as spg  # noqa: E402


def test_prune_of_the_longest_column():
    n = (1 << 31) - 1
    rows = torch.arange(n, dtype=torch.int32, device="cuda")
    vals = (rows % 65521).float()
    special = {3: 70000.0, 1 << 30: 90000.0, n - 2: 80000.0, n - 1: 100000.0}
    for at, v in special.items():
        vals[at] = v
    C = spg.Csc(n, 1, torch.tensor([0, n], dtype=torch.int32, device="cuda"), rows, vals)
    P = spg.prune(C, topk=9)
    # the four largest, and the first five of the equal 65520s, in stored order
    ties = [65520 + 65521 * i for i in range(5)]
    want = sorted(list(special) + ties)
    assert P.colptr.tolist() == [0, 9] and P.rowidx.tolist() == want
    assert P.vals.tolist() == [special.get(i, 65520.0) for i in want]
