"""IMPEC's kernels at the edges of their warps on the GPU: partial warps and
grids without one or two directions, against the oracle; and no store past the
matrix."""
import numpy as np
import pytest

from _gpu_common import need_gpu
from oracle.impec import impec_step, pressure_system
from oracle.pn import natural_to_pn
from paper_2406_10862_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

RTOL = 1e-12          # relative to the entries' magnitude scales: a few dozen roundings


@pytest.mark.parametrize("nphase", [2, 3])
@pytest.mark.parametrize("dims", [(1, 1, 1), (33, 1, 1), (1, 1, 7), (1, 5, 4), (31, 3, 1), (8, 4, 2), (13, 5, 3)])
def test_matrix_and_update_at_the_edges(dims, nphase):
    need_gpu()
    from paper_2406_10862_gb300 import ocp

    g, s = W.tiny(*dims, nphase=nphase, seed=5, frac_unsat=0.3 if nphase == 3 else 0.0, rs_hi=0.7)
    x0, dt = natural_to_pn(g, s.u_new, s.flag_new), 0.5
    A, E0, A_mag, E0_mag, _ = pressure_system(g, x0, dt)
    x1, dP, _, _ = impec_step(g, x0, dt)
    grid = ocp.Grid(g)
    T = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")
    rp, ci = (t.cpu().numpy() for t in grid.pattern())
    rows = np.repeat(np.arange(g.N), np.diff(rp))
    room = torch.full((grid.nnzb + 8,), 7.25, dtype=torch.float64, device="cuda")
    val, rhs = grid.impec_pressure(T(x0.ravel()), dt, val=room[3:3 + grid.nnzb])
    assert grid.status() == 0
    ref, mag = A.toarray()[rows, ci], A_mag[rows, ci]
    assert np.all(np.abs(val.cpu().numpy() - ref) <= RTOL * mag + 1e-300)
    assert np.all(np.abs(rhs.cpu().numpy() + E0) <= RTOL * E0_mag + 1e-300)
    assert (room[:3] == 7.25).all() and (room[3 + grid.nnzb:] == 7.25).all()
    new = grid.impec_update(T(x0.ravel()), T(dP), dt).cpu().numpy().reshape(x0.shape)
    # the update is a difference of products of order 1e-12 of the amounts' own scale
    assert np.allclose(new[0], x1[0], rtol=0, atol=1e-9)
    for e in range(1, nphase + 1):
        assert np.allclose(new[e], x1[e], rtol=1e-11, atol=1e-11 * np.abs(x1[e]).max())
