"""The solver's forms that large systems take, on the GPU: vectors left out of
shared memory (from 345 000 three-phase cells on the published s, from 460 000
on the published p too), several unknowns a thread, and large systems whose
residual is formed by other code than the solver's."""
import numpy as np
import pytest
import scipy.sparse as sp

from paper_2406_10862_gb300 import workloads as W

from _gpu_common import need_gpu

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

RTOL, RES = 1e-11, 1e-10          # as in test_gpu_solver.py


def _system(dims, nb, wells=False):
    """A random block matrix with a dominant diagonal on the grid's pattern."""
    from paper_2406_10862_gb300 import ocp as O

    g, _ = W.tiny(*dims, nphase=max(nb, 2), wells=wells)
    grid = O.Grid(g)
    rng = np.random.default_rng(sum(dims) + nb)
    rp, ci = (t.cpu().numpy() for t in grid.pattern())
    rows = np.repeat(np.arange(grid.N), np.diff(rp))
    v = rng.normal(size=(grid.nnzb, nb, nb))
    v[ci == rows] += 8.0 * nb * np.eye(nb)
    return grid, v, rng.normal(size=grid.N * nb), rp, ci, np.flatnonzero(ci == rows)


def _solve(grid, nb, val, b, x, transpose=False):
    if nb == 1:
        return grid.bicgstab_scalar(val, b, x, RTOL, 400)
    return grid.bicgstab(val, b, x, RTOL, 400, transpose=transpose)


@pytest.mark.parametrize("nb,transpose", [(1, False), (2, False), (2, True), (3, False), (3, True)])
@pytest.mark.parametrize("dims", [(10, 10, 3), (19, 17, 13), (1, 40, 50)])
def test_same_bits_with_vectors_in_global_memory(dims, nb, transpose):
    need_gpu()
    grid, v, b, *_ = _system(dims, nb)
    T = lambda a: torch.as_tensor(a.ravel(), device="cuda")
    val, tb = T(v), T(b)
    for ctas in (0, 3, 40):           # the device's, several unknowns a thread, one unknown a thread
        want = None
        for spill in range(8):
            grid.probe_solver_limits(spill=spill, ctas=ctas)
            x = T(np.random.default_rng(1).normal(size=b.size))
            st, it, rr = _solve(grid, nb, val, tb, x, transpose)
            assert st == 0 and rr <= RTOL
            want = (x, it, rr) if want is None else want
            assert torch.equal(x, want[0]) and (it, rr) == want[1:]
    assert grid.status() == 0


@pytest.mark.parametrize("transpose", [False, True])
def test_wells_with_vectors_in_global_memory(transpose):
    need_gpu()
    from paper_2406_10862_gb300 import ocp as O

    dims = (9, 8, 40)
    grid0, v, b, *_ = _system(dims, 3)
    g, _ = W.tiny(*dims, wells=False)
    g.wells = [W.Well(kind=0, phase=0, p_bh=4600.0, cells=g.column(1, 1)),
               W.Well(kind=1, phase=2, p_bh=5100.0, cells=g.column(7, 6))]
    grid = O.Grid(g)
    rng = np.random.default_rng(3)
    T = lambda a: torch.as_tensor(np.ascontiguousarray(a).ravel(), device="cuda")
    wb, wc, wd, bw = T(rng.normal(size=240)), T(rng.normal(size=240)), T(np.array([40.0, -55.0])), T(rng.normal(size=2))
    for ctas in (0, 3):
        want = None
        for spill in range(8):
            grid.probe_solver_limits(spill=spill, ctas=ctas)
            x, xw = T(np.zeros(b.size)), T(np.zeros(2))
            assert grid.bicgstab_wells(T(v), wb, wc, wd, T(b), bw, x, xw, RTOL, 400, transpose=transpose)[0] == 0
            want = (x, xw) if want is None else want
            assert torch.equal(x, want[0]) and torch.equal(xw, want[1])
    assert grid.status() == 0


# unknowns a CTA of 152: 3x3 100 000 cells 1974; 2x2 1.44 M cells 18 950, whose
# shared memory holds one vector; scalar 600 000 cells 3948
@pytest.mark.parametrize("dims,nb,transpose", [((100, 100, 10), 3, False), ((100, 100, 10), 3, True),
                                               ((120, 120, 100), 2, False), ((120, 120, 100), 2, True),
                                               ((200, 100, 30), 1, False)])
def test_large_systems_against_another_product(dims, nb, transpose):
    need_gpu()
    grid, v, b, rp, ci, diag = _system(dims, nb)
    T = lambda a: torch.as_tensor(a.ravel(), device="cuda")
    x = torch.zeros(b.size, dtype=torch.float64, device="cuda")
    assert _solve(grid, nb, T(v), T(b), x, transpose)[0] == 0
    A = sp.bsr_matrix((v, ci, rp), shape=(b.size, b.size)).tocsr()
    z = b - (A.T if transpose else A) @ x.cpu().numpy()
    D = v[diag].transpose(0, 2, 1) if transpose else v[diag]
    y = np.linalg.solve(D, np.stack([z, b]).reshape(2, grid.N, nb, 1))
    assert np.linalg.norm(y[0]) < RES * np.linalg.norm(y[1])
    assert grid.status() == 0
