"""The device memory of a solve on the GPU: lent by the caller, none held by
the library after it, the path that runs without, and the C interface's own."""
import ctypes
import warnings

import numpy as np
import pytest

from paper_2406_10862_gb300 import workloads as W

from _gpu_common import need_gpu

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

RTOL, RES = 1e-11, 1e-10          # as in test_gpu_solver.py


def _system(dims, nphase=3):
    """A random block matrix with a dominant diagonal on the grid's pattern."""
    from paper_2406_10862_gb300 import ocp as O

    grid = O.Grid(W.tiny(*dims, nphase=nphase, wells=False)[0])
    rng = np.random.default_rng(sum(dims) + nphase)
    rp, ci = (t.cpu().numpy() for t in grid.pattern())
    v = rng.normal(size=(grid.nnzb, nphase, nphase))
    v[ci == np.repeat(np.arange(grid.N), np.diff(rp))] += 8.0 * nphase * np.eye(nphase)
    T = lambda a: torch.as_tensor(a.ravel(), device="cuda")
    return O, grid, T(v), T(rng.normal(size=grid.N * nphase))


def _scaled_residual(grid, val, b, x, transpose):
    """|D^-1 (b - A x)| / |D^-1 b| by the library's product, an independent kernel."""
    nb = grid.nb
    rp, ci = (t.cpu().numpy() for t in grid.pattern())
    diag = np.flatnonzero(ci == np.repeat(np.arange(grid.N), np.diff(rp)))
    D = val.view(-1, nb, nb)[torch.as_tensor(diag, device="cuda")]
    D = D.transpose(1, 2) if transpose else D
    y = torch.linalg.solve(D, torch.stack([b - grid.spmv(val, x, transpose=transpose), b]).view(2, grid.N, nb, 1))
    return float(y[0].norm() / y[1].norm())


def _refuse(monkeypatch, grid):
    """torch has no room for the solver's copy of the matrix."""
    empty = grid.empty

    def refuse(n, dtype=torch.float64):
        if n == 6 * grid.nb * grid.nb * grid.N:
            raise torch.OutOfMemoryError("none")
        return empty(n, dtype)

    monkeypatch.setattr(grid, "empty", refuse)
    monkeypatch.setattr(grid, "_free_bytes", lambda: 0)


@pytest.mark.parametrize("transpose", [False, True])
@pytest.mark.parametrize("dims,nphase", [((17, 19, 13), 3), ((31, 23, 19), 2), ((2, 3, 900), 3)])
def test_without_room_the_solve_runs_and_says_so(monkeypatch, dims, nphase, transpose):
    need_gpu()
    O, grid, val, b = _system(dims, nphase)
    x = torch.zeros_like(b)
    work = grid.solver_work()
    _refuse(monkeypatch, grid)
    with pytest.warns(RuntimeWarning, match="no room"):
        grid.bicgstab(val, b, x, RTOL, 2000, transpose=transpose, work=work)
    assert _scaled_residual(grid, val, b, x, transpose) < RES
    with warnings.catch_warnings():              # and only once while there is none
        warnings.simplefilter("error")
        x.zero_()
        grid.bicgstab(val, b, x, RTOL, 2000, transpose=transpose, work=work)
    assert _scaled_residual(grid, val, b, x, transpose) < RES
    assert grid.status() == 0


@pytest.mark.parametrize("dims,nphase,own", [((10, 10, 3), 3, True), ((1, 1, 2427), 3, True), ((4, 1, 607), 3, False),
                                             ((2, 2, 1365), 2, True), ((1, 1, 5462), 2, False)])
def test_a_small_copy_has_its_place_in_the_grid(dims, nphase, own):
    """Copies of up to 1 MiB: the same answer whether or not memory is lent."""
    need_gpu()
    O, grid, val, b = _system(dims, nphase)
    lib = O.load()
    n = lib.ocp_solver_matrix_doubles(grid._h, nphase)
    assert n == (0 if own else 6 * nphase * nphase * grid.N)
    x, y = torch.zeros_like(b), torch.zeros_like(b)
    grid.bicgstab(val, b, x, RTOL, 2000)
    assert _scaled_residual(grid, val, b, x, False) < RES
    assert lib.ocp_solver_lend(grid._h, None, 0) == 0
    st = lib.ocp_bicgstab(grid._h, val.data_ptr(), b.data_ptr(), y.data_ptr(), RTOL, 2000, 0,
                          grid.solver_work().data_ptr(), None, None, torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    assert st == 0 and (not own or torch.equal(x, y))
    assert _scaled_residual(grid, val, b, y, False) < RES


def test_a_solve_holds_no_device_memory_of_its_own():
    need_gpu()
    O, small, val, b = _system((4, 4, 4))
    small.bicgstab(val, b, torch.zeros_like(b), RTOL, 2000)      # loads the kernels
    O, grid, val, b = _system((100, 100, 12))                    # the copy takes 52 MB
    x, work = torch.zeros_like(b), grid.solver_work()
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0] + torch.cuda.memory_reserved()
    used = torch.cuda.memory_allocated()
    grid.bicgstab(val, b, x, RTOL, 2000, work=work)
    torch.cuda.synchronize()
    assert torch.cuda.memory_allocated() == used
    assert torch.cuda.mem_get_info()[0] + torch.cuda.memory_reserved() == before


def test_the_c_interface_lends_refuses_and_releases():
    need_gpu()
    O, grid, val, b = _system((100, 100, 12))
    lib, h = O.load(), grid._h
    n = lib.ocp_solver_matrix_doubles(h, 3)
    assert n == 54 * grid.N and lib.ocp_solver_matrix_doubles(h, 1) == 6 * grid.N
    assert lib.ocp_solver_matrix_doubles(h, 2) == 0 and lib.ocp_solver_matrix_doubles(None, 3) == 0
    work = grid.solver_work()
    guard = 3.5
    buf = torch.full((n + 2,), guard, dtype=torch.float64, device="cuda")

    def solve(b=b):
        x = torch.zeros_like(val[:3 * grid.N])
        st = lib.ocp_bicgstab(h, val.data_ptr(), b.data_ptr() if b is not None else None, x.data_ptr(), RTOL, 2000, 0,
                              work.data_ptr(), None, None, torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        return st, x

    def lend(t, m):
        return lib.ocp_solver_lend(h, t.data_ptr() if t is not None else None, ctypes.c_int64(m))

    free = lambda: torch.cuda.mem_get_info()[0] + torch.cuda.memory_reserved()
    solve()                                      # loads both forms' kernels
    assert lend(None, 0) == 0
    solve()
    _scaled_residual(grid, val, b, torch.zeros_like(b), False)
    assert lib.ocp_solver_release(h) == 0
    assert lend(buf[1:], n) == 0
    before = free()
    st, want = solve()
    assert st == 0 and free() == before
    assert buf[0] == guard and buf[-1] == guard and (buf[1:-1] != guard).any()
    buf.fill_(guard)
    assert lend(buf, n - 1) == 0                 # too small: from the matrix, the buffer untouched
    st, x = solve()
    assert st == 0 and (buf == guard).all() and free() == before
    assert _scaled_residual(grid, val, b, x, False) < RES
    assert lend(buf, n) == 0                     # a call that is refused gives it back too
    assert solve(None)[0] == O.OCP_ERR_INVALID_ARG
    st, x = solve()                              # nothing lent: the grid's own
    assert st == 0 and torch.equal(x, want) and (buf == guard).all() and free() < before
    assert lib.ocp_solver_release(h) == 0 and free() == before
    assert lend(None, 0) == 0
    st, x = solve()
    assert st == 0 and free() == before
    assert lend(None, 5) == O.OCP_ERR_INVALID_ARG and lend(buf, -1) == O.OCP_ERR_INVALID_ARG
    assert lib.ocp_solver_lend(None, None, 0) == O.OCP_ERR_INVALID_ARG
    assert lib.ocp_solver_release(None) == O.OCP_ERR_INVALID_ARG


@pytest.mark.parametrize("copy", [True, False])
@pytest.mark.parametrize("dims", [(5, 4, 3), (17, 19, 13)])
def test_the_work_buffer_is_not_overrun(monkeypatch, dims, copy):
    need_gpu()
    from paper_2406_10862_gb300 import ocp as O

    _, _, val, b = _system(dims)
    g, _ = W.tiny(*dims, wells=False)
    g.wells = [W.Well(kind=0, phase=0, p_bh=4600.0, cells=np.arange(g.N))]     # every cell perforated
    grid = O.Grid(g)
    n, guard = grid.solver_work().numel(), 3.5
    work = torch.full((n + 2,), guard, dtype=torch.float64, device="cuda")
    rng = np.random.default_rng(0)
    T = lambda a: torch.as_tensor(a, device="cuda")
    wb, wc = T(0.01 * rng.normal(size=b.numel())), T(0.01 * rng.normal(size=b.numel()))
    x, xw = torch.zeros_like(b), torch.zeros(1, dtype=torch.float64, device="cuda")
    if not copy:
        _refuse(monkeypatch, grid)
    with warnings.catch_warnings():
        warnings.simplefilter("ignore")
        grid.bicgstab_wells(val, wb, wc, T(np.array([30.0])), b, T(np.array([1.0])), x, xw, RTOL, 2000,
                            work=work[1:-1])
    assert work[0] == guard and work[-1] == guard
    z = grid.spmv(val, x) + wb * xw - b
    assert float(z.norm()) < 1e-9 * float(b.norm())
    assert abs(float(wc @ x + 30.0 * xw - 1.0)) < 1e-9
