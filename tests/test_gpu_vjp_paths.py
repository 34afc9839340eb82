"""The adjoint product with its PVT table in shared memory (small grids) and
through L1 (from 64 cells per SM on) against the oracle, on both sides of the
line between them and with a partial last warp."""
import numpy as np
import pytest

from _gpu_common import RTOL_VJP, assert_scaled_close, dev_state, need_gpu
from oracle.linearize import linearize as oracle_linearize
from paper_2406_10862_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nphase", [2, 3])
@pytest.mark.parametrize("more", [-1, 0, 33])
def test_adjoint_on_both_sides_of_the_line(nphase, more):
    need_gpu()
    from paper_2406_10862_gb300 import ocp as O

    n = 64 * torch.cuda.get_device_properties(0).multi_processor_count + more
    g, s = W.tiny(n, 1, 1, nphase=nphase, seed=46)
    lam = np.random.default_rng(5).normal(size=(g.N, nphase))
    o = oracle_linearize(g, s.u_new, s.flag_new, s.u_old, s.flag_old, s.dt, mode="all", lam=lam)
    grid = O.Grid(g)
    un, fn, uo, fo = dev_state(s)
    _, v, ff = grid.linearize(un, fn, uo, fo, s.dt, want_face_flux=True)
    out = grid.adjoint_vjp(un, fn, uo, fo, s.dt, v, ff, torch.as_tensor(lam.ravel(), device="cuda"))
    assert grid.status() == 0
    for k in ("unew", "uold", "lnk", "phi"):
        assert_scaled_close(out[k].cpu().numpy(), o["g_" + k], o["g_%s_mag" % k], RTOL_VJP, "g_" + k)
