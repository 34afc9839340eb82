"""What a grid holds on the device: its scratch is the 73 doubles per cell that
the linearisation uses, in whole tiles of 32 cells, and nothing beside it."""
import pytest

from paper_2406_10862_gb300 import workloads as W

from _gpu_common import need_gpu

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nphase", [2, 3])
def test_memory_of_a_grid(nphase):
    need_gpu()
    from paper_2406_10862_gb300 import ocp as O

    O.Grid(W.tiny(4, 4, 4, nphase=nphase)[0])          # loads the kernels
    g, _ = W.tiny(100, 100, 100, nphase=nphase)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    grid = O.Grid(g)
    held = before - torch.cuda.mem_get_info()[0]
    # scratch 584, transmissibilities 24, their derivatives 48, porosity 8, well map 4,
    # row starts 4, columns 28 bytes a cell; 12 allocations in pages of 2 MB, and
    # 2.2 MB for the solver's slots
    assert 700 * g.N < held < 700 * g.N + (13 * 2 + 3) * (1 << 20)
    del grid
