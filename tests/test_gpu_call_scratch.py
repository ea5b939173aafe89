"""The device block that transposes, prunes and merges keep between calls."""
from __future__ import annotations

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2010_08526_gb300 as spg  # noqa: E402


class Refusing(spg.TorchAllocator):
    """Refuses the allocations of one kind, counting them."""

    def __init__(self, kind):
        super().__init__()
        self.kind = kind
        self.refused = 0

    def allocate(self, nbytes, kind):
        if kind == self.kind:
            self.refused += 1
            return None
        return super().allocate(nbytes, kind)


def diagonal(n):
    i = torch.arange(n + 1, device="cuda", dtype=torch.int32)
    return spg.Csc(n, n, i, i[:n].clone(), torch.ones(n, device="cuda"))


def free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def test_a_refused_allocation_gives_the_block_back():
    """PyTorch's allocator refusing device memory: the call fails as before, asked
    once (the device has memory), and the 32 MiB are the device's again."""
    A = diagonal(1000)
    for first in (True, False):                # the first time loads code and fills PyTorch's pools, too
        T = spg.transpose(A)                   # takes the block (again)
        assert torch.equal(T.rowidx, A.rowidx)
        held = free()
        al = Refusing(0)
        with pytest.raises(spg.SpgemmError) as e:
            spg.Plan(A, A, allocator=al)
        assert e.value.status == 2 and al.refused == 1 and al.live == 0
        assert first or free() - held >= 32 << 20


def test_refused_host_memory_keeps_the_block():
    A = diagonal(1000)
    spg.transpose(A)
    held = free()
    al = Refusing(1)
    with pytest.raises(spg.SpgemmError) as e:
        spg.Plan(A, A, allocator=al)
    assert e.value.status == 2 and al.live == 0 and free() <= held + (4 << 20)
