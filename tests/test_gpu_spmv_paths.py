"""The block products' paths on the GPU -- staged by bulk copy, through
registers, transposed through shared memory or by wide loads -- give the same
bits whatever the matrix's alignment, and the oracle's product, at partial
warps, grids without a direction and odd matrix sizes."""
import numpy as np
import pytest

from _gpu_common import RTOL_SPMV, need_gpu
from oracle.spmv import bsr_spmv
from paper_2406_10862_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("transpose", [False, True])
@pytest.mark.parametrize("nb", [2, 3])
@pytest.mark.parametrize("dims", [(1, 1, 1), (33, 1, 1), (1, 1, 7), (1, 5, 4), (31, 3, 1), (8, 4, 2), (13, 5, 3),
                                  (17, 9, 7)])
def test_products_at_every_alignment(dims, nb, transpose):
    need_gpu()
    from paper_2406_10862_gb300 import ocp as O

    g, _ = W.tiny(*dims, nphase=nb, wells=False)
    grid = O.Grid(g)
    rp, ci = (t.cpu().numpy() for t in grid.pattern())
    rng = np.random.default_rng(sum(dims) + nb)
    n, nv = nb * grid.N, grid.nnzb * nb * nb
    val, x, y0 = rng.normal(size=nv), rng.normal(size=n), rng.normal(size=n)
    T = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")
    blocks = val.reshape(-1, nb, nb)
    for alpha, beta in ((1.0, 0.0), (-0.75, 0.0), (1.5, 0.25)):
        ref, mag = bsr_spmv(rp, ci, blocks, x, alpha, beta, y0.copy(), transpose)
        want = None
        for off in range(4):
            room = torch.full((nv + 8,), float("nan"), dtype=torch.float64, device="cuda")
            room[off:off + nv] = T(val)
            y = grid.spmv(room[off:off + nv], T(x), alpha, beta, T(y0), transpose=transpose).cpu()
            assert grid.status() == 0
            assert np.all(np.abs(y.numpy() - ref) <= RTOL_SPMV * mag + 1e-300)
            want = y if want is None else want
            assert torch.equal(y, want)
