"""A caller's allocator whose pointers are off the 256-byte boundary: the
context aligns them, and steps as with its own memory."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1809_10895_gb300 import rf
from paper_1809_10895_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1809_10895_gb300 import build as B
    B.build()
    rf.load()
    torch.cuda.set_device(0)


class Offset(rf.TorchAllocator):
    def _do_alloc(self, nbytes, user):
        t = self.torch.empty(int(nbytes) + 8, dtype=self.torch.uint8, device=self.device)
        self.blocks[t.data_ptr() + 8] = t
        return t.data_ptr() + 8


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("attempts", [True, False])
def test_offset_pointers(monkeypatch, precision, attempts):
    case = W.heterogeneous_box(20, 13, 12, d=0.25, seed=7, water_table_depth=1.5, rain=5e-6, dt0=60.0)
    heads = []
    for alloc in (rf.TorchAllocator, Offset):
        monkeypatch.setattr(rf, "TorchAllocator", alloc)
        s = rf.Solver.from_case(case, precision=precision)
        assert (alloc is Offset) == all(p % 256 == 8 for p in s._allocator.blocks)
        s.set_one_launch(attempts=attempts)
        for _ in range(3):
            s.step()
        heads.append(s.get_state()[0])
        blocks = s._allocator.blocks
        s.close()
        assert not blocks
    assert np.array_equal(*heads)
