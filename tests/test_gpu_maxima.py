"""The updates' and norms' maxima on the GPU: one atomic per CTA must give the
exact maximum over the cells, whatever the number of CTAs, and count every
switched cell."""
import numpy as np
import pytest

from paper_2406_10862_gb300 import workloads as W

from _gpu_common import need_gpu

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(1, 1, 1), (31, 1, 1), (8, 8, 4), (257, 1, 1), (40, 30, 7)])
@pytest.mark.parametrize("nphase", [2, 3])
def test_maxima_are_exact(dims, nphase):
    need_gpu()
    from paper_2406_10862_gb300 import ocp as O

    g, s = W.tiny(*dims, nphase=nphase, wells=False)
    grid = O.Grid(g)
    nb, N = nphase, g.N
    T = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")
    rng = np.random.default_rng(N + nb)
    u, f = T(s.u_new.ravel()).clone(), T(s.flag_new).clone()
    du = rng.normal(size=(N, nb)) * np.array([10.0, 0.05, 0.05])[:nb]
    dmax, nsw = torch.full((4,), -1.0, dtype=torch.float64, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    f0 = f.clone()
    grid.newton_update(u, f, T(du.ravel()), -1.0, 10.0, dmax, nsw)
    got = dmax.cpu().numpy()
    assert got[0] == np.abs(du[:, 0]).max() and got[1] == np.abs(du[:, 1]).max()
    if nb == 3:
        for k in (0, 1):
            of = np.abs(du[s.flag_new == k, 2])
            assert got[2 + k] == (of.max() if len(of) else 0.0)
        assert int(nsw.item()) == int((f != f0).sum())
    # (P, N): the update's and the norms' maxima
    pn = torch.zeros((nb + 1) * N, dtype=torch.float64, device="cuda")
    elim = T(np.concatenate([rng.normal(size=(nb + 1) * N)]))
    dm = torch.zeros(nb + 1, dtype=torch.float64, device="cuda")
    grid.pn_update(pn, T(du.ravel()), 2.0, elim, dm)
    assert np.array_equal(dm.cpu().numpy(), np.abs(pn.view(nb + 1, N).cpu().numpy()).max(axis=1))
    res = rng.normal(size=(N, nb + 1))
    norms = grid.pn_norms(T(res.ravel()), 0.5).cpu().numpy()
    pv = np.asarray(g.phi) * (g.dx * g.dy * g.dz / 5.614583 / 0.5)
    assert norms[3] == np.abs(res[:, nb]).max()
    for e in range(nb):
        # one rounding each in the pore volume's scale and product, and the quotient
        assert abs(norms[e] - (np.abs(res[:, e]) / pv).max()) <= 4e-16 * norms[e]
