"""A wait between the solver's CTAs that runs out on the GPU: the solve is
reported as failed, also where the other CTAs finished it, and the next solve
on the grid is untouched by it."""
import numpy as np
import pytest

from paper_2406_10862_gb300 import workloads as W

from _gpu_common import need_gpu

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

POLLS = 20000          # about 10 ms: the other CTAs' waits end soon


def _system(dims):
    from paper_2406_10862_gb300 import ocp as O

    g, s = W.tiny(*dims)
    grid = O.Grid(g)
    T = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")
    r, val, _ = grid.linearize(T(s.u_new.ravel()), T(s.flag_new), T(s.u_old.ravel()), T(s.flag_old), 0.1)
    return O, grid, val, r / r.abs().max()


# 12 597 unknowns: about a hundred CTAs of 128
@pytest.mark.parametrize("start", ["zero", "solved"])
@pytest.mark.parametrize("cta", [0, 1, 57])
def test_a_wait_that_runs_out_is_an_error(cta, start):
    need_gpu()
    O, grid, val, b = _system((17, 19, 13))
    want = torch.zeros_like(b)
    grid.bicgstab(val, b, want, 1e-12, 2000)
    # from the solution the loop's first test ends the solve at its first wait:
    # every CTA but one then finishes it
    x = want.clone() if start == "solved" else torch.zeros_like(b)
    grid.probe_solver_limits(polls=POLLS, short_cta=cta)
    st, _, _ = grid.bicgstab(val, b, x, 1e-8, 2000, check=False)
    assert st == O.OCP_ERR_TIMEOUT
    assert grid.status() == O.OCP_ERR_TIMEOUT
    grid.probe_solver_limits()
    x = torch.zeros_like(b)
    st, _, _ = grid.bicgstab(val, b, x, 1e-12, 2000)
    assert st == 0 and grid.status() == 0 and torch.equal(x, want)
