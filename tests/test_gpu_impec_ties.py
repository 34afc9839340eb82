"""IMPEC at exact upwind ties on the GPU: uniform pressure and no capillary
pressure, so that the potential difference of every horizontal face is zero,
with saturations that differ from cell to cell.  Both rows of a face have to
take the same upstream cell (the lower-numbered one, as the oracle does), or
the update makes or loses mass."""
import dataclasses

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
@pytest.mark.parametrize("dims", [(33, 1, 1), (1, 9, 1), (7, 6, 1), (6, 5, 3)])
def test_rows_of_a_tied_face_agree(dims, nphase):
    need_gpu()
    from paper_2406_10862_gb300 import ocp

    g, s = W.tiny(*dims, nphase=nphase, seed=3, wells=False)
    g = dataclasses.replace(g, pcow_max=0.0, pcgo_max=0.0)
    u = s.u_new.copy()
    u[0] = 4000.0 + 2.0 * (np.arange(g.N) // (g.nx * g.ny))     # uniform in every layer
    flag = np.zeros(g.N, dtype=np.int8)
    rng = np.random.default_rng(4)
    u[1] = rng.uniform(0.2, 0.6, g.N)
    if nphase == 3:
        u[2] = rng.uniform(0.05, 0.3, g.N)
    x0, dt = natural_to_pn(g, u, flag), 0.5
    A, E0, A_mag, E0_mag, _ = pressure_system(g, x0, dt)
    grid = ocp.Grid(g)
    T = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")
    rp, ci = (t.cpu().numpy() for t in grid.pattern())
    rows = np.repeat(np.arange(g.N), np.diff(rp))
    val, rhs = grid.impec_pressure(T(x0.ravel()), dt)
    assert np.all(np.abs(val.cpu().numpy() - A.toarray()[rows, ci]) <= RTOL * A_mag[rows, ci] + 1e-300)
    assert np.all(np.abs(rhs.cpu().numpy() + E0) <= RTOL * E0_mag + 1e-300)
    # a pressure change that moves every phase through every face
    dP = rng.normal(0.0, 50.0, g.N)
    new = grid.impec_update(T(x0.ravel()), T(dP), dt).cpu().numpy().reshape(x0.shape)
    assert grid.status() == 0
    for e in range(1, nphase + 1):
        moved = new[e] - x0[e]
        # no wells: what leaves a cell enters another; each cell's sum of at most six
        # fluxes rounds within 8 units of the amounts and of the flux sums
        assert abs(moved.sum()) <= 8 * 2.0 ** -53 * (np.abs(x0[e]).sum() + np.abs(moved).sum()) * 6
        assert np.abs(moved).max() > 1e-6 * np.abs(x0[e]).max()
