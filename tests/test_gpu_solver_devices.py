"""The solver where its launch cannot have a CTA on every SM of the device: a
bounded number of CTAs, and a stream of a green context."""
import contextlib
import ctypes

import numpy as np
import pytest

from paper_2406_10862_gb300 import workloads as W

from _gpu_common import need_gpu

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# As in test_gpu_solver.py: the solver stops at |D^-1 (b - A x)| <= rtol |D^-1 b|;
# the residual formed apart from it may add rounding.
RTOL, RES = 1e-11, 1e-10


def _system(dims, nphase=3):
    from paper_2406_10862_gb300 import ocp as O

    g, s = W.tiny(*dims, nphase=nphase)
    grid = O.Grid(g)
    T = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")
    r, val, _ = grid.linearize(T(s.u_new.ravel()), T(s.flag_new), T(s.u_old.ravel()), T(s.flag_old), 0.1)
    return grid, val, r / r.abs().max()


def _scaled_residual(grid, val, b, x):
    """|D^-1 (b - A x)| / |D^-1 b| by the library's product, an independent kernel."""
    nb = grid.nb
    rp, ci = (t.cpu().numpy() for t in grid.pattern())
    diag = np.flatnonzero(ci == np.repeat(np.arange(grid.N), np.diff(rp)))
    D = val.view(-1, nb, nb)[torch.as_tensor(diag, device="cuda")]
    z = torch.stack([b - grid.spmv(val, x), b]).view(2, grid.N, nb, 1)
    y = torch.linalg.solve(D, z)
    return float(y[0].norm() / y[1].norm())


@pytest.mark.parametrize("dims", [(1, 1, 1), (10, 10, 3), (17, 19, 13)])
@pytest.mark.parametrize("ctas", [1, 5, 33])
def test_fewer_ctas_solve_the_same_system(ctas, dims):
    need_gpu()
    grid, val, b = _system(dims)
    want, x = torch.zeros_like(b), torch.zeros_like(b)
    grid.bicgstab(val, b, want, RTOL, 2000)
    grid.probe_solver_limits(ctas=ctas)
    assert grid.bicgstab(val, b, x, RTOL, 2000)[0] == 0
    assert _scaled_residual(grid, val, b, x) < RES
    grid.probe_solver_limits()
    x.zero_()
    assert grid.bicgstab(val, b, x, RTOL, 2000)[0] == 0 and torch.equal(x, want)
    assert grid.status() == 0


class _Resource(ctypes.Structure):          # CUdevResource of cuda.h
    _fields_ = [("type", ctypes.c_int), ("pad", ctypes.c_ubyte * 92), ("sms", ctypes.c_uint),
                ("rest", ctypes.c_ubyte * 44)]


@contextlib.contextmanager
def _share_of_the_device(least):
    """A stream of a green context of at least so many SMs, and their number."""
    lib = ctypes.CDLL("libcuda.so.1")

    def call(name, *args):
        st = getattr(lib, name)(*args)
        if st == 801:                        # CUDA_ERROR_NOT_SUPPORTED
            pytest.skip("this device makes no green contexts")
        assert st == 0, (name, st)

    whole, part, rest, n = _Resource(), _Resource(), _Resource(), ctypes.c_uint(1)
    desc, green, stream = ctypes.c_void_p(), ctypes.c_void_p(), ctypes.c_void_p()
    ref = ctypes.byref
    call("cuDeviceGetDevResource", 0, ref(whole), 1)
    call("cuDevSmResourceSplitByCount", ref(part), ref(n), ref(whole), ref(rest), ctypes.c_uint(0), ctypes.c_uint(least))
    call("cuDevResourceGenerateDesc", ref(desc), ref(part), ctypes.c_uint(1))
    call("cuGreenCtxCreate", ref(green), desc, 0, ctypes.c_uint(1))
    try:
        call("cuGreenCtxStreamCreate", ref(stream), green, ctypes.c_uint(1), 0)
        try:
            assert least <= part.sms < whole.sms
            yield torch.cuda.ExternalStream(stream.value), part.sms
        finally:
            call("cuStreamDestroy_v2", stream)
    finally:
        call("cuGreenCtxDestroy", green)


@pytest.mark.parametrize("dims", [(10, 10, 3), (17, 19, 13)])
def test_a_stream_with_a_share_of_the_device(dims):
    """The solve takes a CTA on each of its stream's SMs: the bits of as many on
    the whole device."""
    need_gpu()
    grid, val, b = _system(dims)
    x, want, work = torch.zeros_like(b), torch.zeros_like(b), grid.solver_work()
    torch.cuda.synchronize()
    with _share_of_the_device(16) as (stream, sms):
        assert grid.bicgstab(val, b, x, RTOL, 2000, work=work, stream=stream)[0] == 0
    assert _scaled_residual(grid, val, b, x) < RES
    grid.probe_solver_limits(ctas=sms)
    grid.bicgstab(val, b, want, RTOL, 2000, work=work)
    assert torch.equal(x, want) and grid.status() == 0
