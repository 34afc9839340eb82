"""The persistent BiCGSTAB on the GPU against dense solves.

Sizes at the edges of its work split (an unknown per thread, 32-unknown
chunks, CTAs of at least 128 unknowns, ranges that do not divide evenly, the
largest system of the one-cluster launch and the smallest above it), grids
without one or two directions, both orientations, every block size,
and the path without the scaled copy of the matrix.
"""
import numpy as np
import pytest

from paper_2406_10862_gb300 import workloads as W

from _gpu_common import need_gpu

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# The solver stops at |D^-1 (b - A x)| <= rtol |D^-1 b|; a dense LU of the
# same matrix has an error of the order of eps cond.  x is compared through
# its scaled residual, so no condition number enters: rtol plus rounding.
RTOL = 1e-11
RES = 1e-10


def _dense(grid, val, nb):
    rp, ci = (t.cpu().numpy() for t in grid.pattern())
    v = val.cpu().numpy().reshape(-1, nb, nb)
    A = np.zeros((grid.N * nb, grid.N * nb))
    for r in range(grid.N):
        for s in range(rp[r], rp[r + 1]):
            A[r * nb:(r + 1) * nb, ci[s] * nb:(ci[s] + 1) * nb] = v[s]
    return A


def _matrix(n_blocks, rp, ci, nb, seed):
    """A random block matrix with a dominant diagonal."""
    rng = np.random.default_rng(seed)
    v = rng.normal(size=(n_blocks, nb, nb))
    for r in range(len(rp) - 1):
        for s in range(rp[r], rp[r + 1]):
            if ci[s] == r:
                v[s] += 8.0 * nb * np.eye(nb)
    return v


def _scaled_residual(A, x, b, nb):
    n = len(b) // nb
    z, y = (b - A @ x).reshape(n, nb), b.reshape(n, nb)
    D = np.stack([A[c * nb:(c + 1) * nb, c * nb:(c + 1) * nb] for c in range(n)])
    return np.linalg.norm(np.linalg.solve(D, z[:, :, None])) / np.linalg.norm(np.linalg.solve(D, y[:, :, None]))


@pytest.mark.parametrize("transpose", [False, True])
@pytest.mark.parametrize("nb", [1, 2, 3])
@pytest.mark.parametrize("dims", [(1, 1, 1), (5, 1, 1), (1, 3, 1), (1, 1, 11), (7, 6, 1), (1, 9, 5), (4, 1, 8),
                                  (8, 8, 2), (11, 4, 4), (9, 8, 7), (17, 13, 3), (16, 16, 8), (41, 5, 10)])
def test_solves_random_block_systems(dims, nb, transpose):
    need_gpu()
    from paper_2406_10862_gb300 import ocp as O

    if nb == 1 and transpose:
        pytest.skip("the scalar system has no transposed entry point")
    g, _ = W.tiny(*dims, nphase=max(nb, 2), wells=False)
    grid = O.Grid(g)
    rp, ci = (t.cpu().numpy() for t in grid.pattern())
    v = _matrix(grid.nnzb, rp, ci, nb, sum(dims) + nb)
    val = torch.as_tensor(v.ravel(), device="cuda")
    rng = np.random.default_rng(7)
    b = rng.normal(size=grid.N * nb)
    x = torch.as_tensor(rng.normal(size=grid.N * nb), device="cuda")
    A = _dense(grid, val, nb)
    if transpose:
        A = A.T
    tb = torch.as_tensor(b, device="cuda")
    if nb == 1:
        st, it, rr = grid.bicgstab_scalar(val, tb, x, RTOL, 200)
    else:
        st, it, rr = grid.bicgstab(val, tb, x, RTOL, 200, transpose=transpose)
    assert st == 0 and rr <= RTOL and it <= 200
    assert _scaled_residual(A, x.cpu().numpy(), b, nb) < RES
    assert grid.status() == 0
    # an exact guess needs no iteration, and the solve is repeatable bit for bit
    x2 = torch.as_tensor(np.random.default_rng(7).normal(size=2 * grid.N * nb)[grid.N * nb:], device="cuda")
    if nb == 1:
        grid.bicgstab_scalar(val, tb, x2, RTOL, 200)
        assert torch.equal(x, x2)
        assert grid.bicgstab_scalar(val, tb, x.clone(), 1e-8, 200)[1] == 0
    else:
        grid.bicgstab(val, tb, x2, RTOL, 200, transpose=transpose)
        assert torch.equal(x, x2)
        assert grid.bicgstab(val, tb, x.clone(), 1e-8, 200, transpose=transpose)[1] == 0


@pytest.mark.parametrize("transpose", [False, True])
def test_wells_over_many_warps(transpose):
    """A well of more than 32 perforations, cells of two wells in one warp."""
    need_gpu()
    from paper_2406_10862_gb300 import ocp as O

    g, _ = W.tiny(6, 4, 40, wells=False)
    g.wells = [W.Well(kind=0, phase=0, p_bh=4600.0, cells=g.column(1, 1)),
               W.Well(kind=1, phase=2, p_bh=5100.0, cells=g.column(2, 1)),
               W.Well(kind=0, phase=0, p_bh=4500.0, cells=np.array([3], dtype=np.int64))]
    grid = O.Grid(g)
    nb, n, npf = 3, 3 * grid.N, 81
    rp, ci = (t.cpu().numpy() for t in grid.pattern())
    v = _matrix(grid.nnzb, rp, ci, nb, 5)
    rng = np.random.default_rng(11)
    wb, wc, wd = rng.normal(size=npf * nb), rng.normal(size=npf * nb), np.array([40.0, -55.0, 3.0])
    b, bw = rng.normal(size=n), rng.normal(size=3)
    T = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")
    x, xw = torch.zeros(n, dtype=torch.float64, device="cuda"), torch.zeros(3, dtype=torch.float64, device="cuda")
    st, it, rr = grid.bicgstab_wells(T(v.ravel()), T(wb), T(wc), T(wd), T(b), T(bw), x, xw, RTOL, 300,
                                     transpose=transpose)
    A = _dense(grid, T(v.ravel()), nb)
    full = np.zeros((n + 3, n + 3))
    full[:n, :n] = A
    k = 0
    for w, well in enumerate(g.wells):
        for c in well.cells:
            full[c * nb:(c + 1) * nb, n + w] = wb[k * nb:(k + 1) * nb]
            full[n + w, c * nb:(c + 1) * nb] = wc[k * nb:(k + 1) * nb]
            k += 1
        full[n + w, n + w] = wd[w]
    if transpose:
        full = full.T
    z = full @ np.concatenate([x.cpu().numpy(), xw.cpu().numpy()]) - np.concatenate([b, bw])
    assert st == 0 and np.linalg.norm(z) < 1e-9 * np.linalg.norm(np.concatenate([b, bw]))


def test_without_room_for_the_scaled_matrix():
    """Device memory filled up to less than the scaled copy of the matrix: the
    solve runs from the matrix itself and agrees to the solver's tolerance."""
    need_gpu()
    from paper_2406_10862_gb300 import ocp as O

    g, s = W.layered_box(nx=100, ny=100, nz=24)              # the copy takes 104 MB
    grid = O.Grid(g)
    T = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")
    un, fn, uo, fo = T(s.u_new.ravel()), T(s.flag_new), T(s.u_old.ravel()), T(s.flag_old)
    r, val, _ = grid.linearize(un, fn, uo, fo, 0.1)
    work, b = grid.solver_work(), r / r.abs().max()
    xs = []
    other = O.Grid(W.tiny(4, 4, 4)[0])                       # loads the solver's kernels
    w2 = torch.zeros(3 * other.N, dtype=torch.float64, device="cuda")
    other.bicgstab(torch.ones(other.nnzb * 9, dtype=torch.float64, device="cuda"), w2, w2.clone(), 1e-8, 1, check=False)
    other.status()
    x = torch.zeros_like(b)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    fill = torch.empty(free - (80 << 20), dtype=torch.uint8, device="cuda")
    try:
        assert torch.cuda.mem_get_info()[0] < 100 << 20
        for transpose in (False, True):
            x.zero_()
            st, it, rr = grid.bicgstab(val, b, x, 1e-12, 2000, transpose=transpose, work=work)
            assert st == 0
            xs.append(x.cpu())
    finally:
        del fill
        torch.cuda.empty_cache()
    for transpose, got in zip((False, True), xs):
        x.zero_()
        grid.bicgstab(val, b, x, 1e-12, 2000, transpose=transpose, work=work)
        want = x.cpu()
        # both stop at 1e-12 of the scaled residual; the systems' condition is
        # below 1e5, which bounds the solutions' difference by 2e-7
        assert float((got - want).norm() / want.norm()) < 2e-7
    assert grid.status() == 0
