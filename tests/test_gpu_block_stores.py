"""The linearisation's block stores on the GPU: grids whose last warp is
partial or has no + faces in a direction, and outputs that are aligned to 8
bytes only (the wide store of a 2x2 block needs 32), in every launch shape."""
import numpy as np
import pytest

from paper_2406_10862_gb300 import workloads as W

from _gpu_common import need_gpu

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SHAPES = [([64, 32, 32], 0), ([128, 128, 256], 0), ([32, 64, 64], 0), ([64, 64, 64], 1), ([64, 32, 32], 2),
          ([32, 32, 32], 3)]


@pytest.mark.parametrize("nphase", [2, 3])
@pytest.mark.parametrize("dims", [(1, 1, 1), (33, 1, 1), (1, 1, 40), (31, 3, 1), (32, 4, 2), (9, 7, 5)])
def test_same_bits_at_every_alignment_and_shape(dims, nphase):
    need_gpu()
    from paper_2406_10862_gb300 import ocp as O

    g, s = W.tiny(*dims, nphase=nphase)
    grid = O.Grid(g)
    T = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")
    args = (T(s.u_new.ravel()), T(s.flag_new), T(s.u_old.ravel()), T(s.flag_old), s.dt)
    nv, nr = grid.nnzb * nphase * nphase, nphase * grid.N
    want = None
    for tiles, ordered in SHAPES:
        grid.set_shape(dict(cells_per_tile=tiles, ctas_per_sm=[0, 0, 0], ordered=ordered))
        for off in range(4):
            guard = 7.25
            val = torch.full((nv + 8,), guard, dtype=torch.float64, device="cuda")
            res = torch.full((nr + 8,), guard, dtype=torch.float64, device="cuda")
            grid.linearize(*args, residual=res[off:off + nr], bsr_val=val[off:off + nv])
            assert grid.status() == 0
            v, r = val.cpu(), res.cpu()
            for x, n in ((v, nv), (r, nr)):
                assert (x[:off] == guard).all() and (x[off + n:] == guard).all()
            got = (v[off:off + nv], r[off:off + nr])
            if want is None:
                want = got
            assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
