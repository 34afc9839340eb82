"""The rounding of d(gas amount)/d S_g, phi (b_g - R_s b_o), on the GPU: the two
terms nearly cancel, so a rounding of either one shows.

One row of cells at rest at a knot of the PVT table, without capillary
pressure and rock compressibility and of unit volume: b_g, b_o, R_s and phi are
the doubles that the tables hold, every face's terms are zero, and the entry is
that derivative alone.  Its error is measured against exact rationals in units
of the variance of three independent roundings, of phi b_g, phi b_o and the
result: 1 if these are all there are, against 1.6 with the product by R_s
rounded too (the statistic scatters by 0.01 at 20 000 cells)."""
import dataclasses
from fractions import Fraction

import numpy as np
import pytest

from _gpu_common import need_gpu
from paper_2406_10862_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CELLS = 20000


def case():
    g, s = W.tiny(CELLS, 1, 1, wells=False, seed=8)
    g = dataclasses.replace(g, pcow_max=0.0, pcgo_max=0.0, cr=0.0, dx=5.614583, dy=1.0, dz=1.0)
    k = len(g.tab_p) - 3
    u = np.stack([np.full(CELLS, float(g.tab_p[k])), np.full(CELLS, 0.2), np.full(CELLS, 0.15)])
    return g, u, (1.0 / float(g.tab_Bg[k]), 1.0 / float(g.tab_Bo[k]), float(g.tab_Rs[k]))


def statistic(got, phi, fluid):
    """Mean of error^2 over its variance with three roundings."""
    bg, bo, rs = fluid
    total = Fraction(bg) - Fraction(rs) * Fraction(bo)
    err = np.array([float(Fraction(float(v)) - Fraction(float(p)) * total) for v, p in zip(got, phi)])
    var = (np.spacing(phi * bg) ** 2 + (rs * np.spacing(phi * bo)) ** 2 + np.spacing(np.abs(got)) ** 2) / 12.0
    return float(np.mean(err ** 2 / var))


@pytest.mark.parametrize("mixed", [False, True])
def test_the_product_by_rs_is_not_rounded(mixed):
    need_gpu()
    from paper_2406_10862_gb300 import ocp as O

    g, u, fluid = case()
    flag = np.zeros(CELLS, dtype=np.int8)
    if mixed:                       # an undersaturated cell in every warp: the general form
        flag[::32] = 1
        u[2, ::32] = 0.5 * fluid[2]
    grid = O.Grid(g)
    T = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")
    _, val, _ = grid.linearize(T(u.ravel()), T(flag), T(u.ravel()), T(flag), 1.0)
    assert grid.status() == 0
    rp, ci = (t.cpu().numpy() for t in grid.pattern())
    diag = np.flatnonzero(ci == np.repeat(np.arange(CELLS), np.diff(rp)))
    got = val.view(-1, 3, 3).cpu().numpy()[diag, 2, 2]
    rest = np.ones(CELLS, dtype=bool)
    if mixed:                       # the neighbours' faces hold flow terms: inner cells of each run
        at = np.arange(CELLS) % 32
        rest = (at > 1) & (at < 31)
    assert statistic(got[rest], np.asarray(g.phi)[rest], fluid) < 1.1
