"""The (P, N) reduction's block access on the GPU: partial warps, grids
without a direction, matrices aligned to 8 bytes only, with and without the
full system, against the oracle."""
import numpy as np
import pytest

from _gpu_common import RTOL_J, RTOL_R, assert_scaled_close, need_gpu
from oracle.pn import eliminate_volume_row, linearize_pn, natural_to_pn
from paper_2406_10862_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nphase", [2, 3])
@pytest.mark.parametrize("dims", [(1, 1, 1), (33, 1, 1), (1, 1, 7), (31, 3, 1), (8, 4, 2)])
def test_reduction_at_the_edges(dims, nphase):
    need_gpu()
    from paper_2406_10862_gb300 import ocp

    g, s = W.tiny(*dims, nphase=nphase, seed=8, frac_unsat=0.35 if nphase == 3 else 0.0, rs_hi=0.7)
    x_new, x_old = natural_to_pn(g, s.u_new, s.flag_new), natural_to_pn(g, s.u_old, s.flag_old)
    x_new[1] *= 1.002                    # off the volume-balance manifold
    full = linearize_pn(g, x_new, x_old, 1.5)
    red = eliminate_volume_row(g, full)
    grid = ocp.Grid(g)
    T = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")
    N, nb, L = g.N, nphase, nphase + 1
    for off in range(4):
        bufs = {"bsr_val": grid.nnzb * nb * nb, "bsr_val_full": grid.nnzb * L * L}
        room = {k: torch.full((n + 8,), 7.25, dtype=torch.float64, device="cuda") for k, n in bufs.items()}
        views = {k: room[k][off:off + n] for k, n in bufs.items()}
        o = grid.linearize_pn(T(x_new.ravel()), T(x_old.ravel()), 1.5, out=dict(views), full=True)
        red_only = grid.linearize_pn(T(x_new.ravel()), T(x_old.ravel()), 1.5)
        assert grid.status() == 0
        assert_scaled_close(o["residual"].cpu().numpy(), red["R"], red["R_mag"], RTOL_R, "reduced residual")
        assert_scaled_close(o["bsr_val"].cpu().numpy(), red["val"], red["val_mag"], RTOL_J, "reduced bsr_val")
        assert_scaled_close(o["residual_full"].cpu().numpy(), full["R"], full["R_mag"], RTOL_R, "full residual")
        assert_scaled_close(o["bsr_val_full"].cpu().numpy(), full["val"], full["val_mag"], RTOL_J, "full bsr_val")
        for k in ("residual", "bsr_val", "elim"):
            assert torch.equal(o[k], red_only[k])
        for k, n in bufs.items():
            x = room[k].cpu()
            assert (x[:off] == 7.25).all() and (x[off + n:] == 7.25).all()
