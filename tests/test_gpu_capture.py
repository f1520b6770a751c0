"""Calls recorded into a CUDA graph by the caller, on the caller's stream, and replayed: the one-launch steps
of 1D grids, and 2D grids in FP64, in pairs with what is left taken block by block, and with the grid's
list, give what the same calls give when issued directly, bit for bit, replay after replay."""
import ctypes

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2411_11229_gb300 import Solver  # noqa: E402
from paper_2411_11229_gb300 import _capi as C  # noqa: E402


def _state(dim, nx, ny):
    if dim == 1:
        S, dx = W.euler1d_random(nx, 3, "jumps")
        return S, dx, dx
    S, dx, dy = W.euler2d_random(nx, ny, 3, "smooth")
    S[:, :, : ny // 3, : nx // 3] *= 1.3
    return S, dx, dy


@pytest.mark.parametrize("dim,nx,ny", [(1, 130, 1), (1, 5000, 1), (1, 20011, 1), (2, 40, 33), (2, 150, 139), (2, 197, 167)])
def test_steps_and_operator_in_a_graph(dim, nx, ny):
    S, dx, dy = _state(dim, nx, ny)
    st = torch.cuda.Stream()
    a = Solver(dim, "euler", nx, ny, dx=dx, dy=dy, bc="transmissive", stream=st)
    b = Solver(dim, "euler", nx, ny, dx=dx, dy=dy, bc="transmissive", stream=st)
    p = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    out = []
    for s in (a, b):
        s.set_state(S)
        s.set_time(0.0, 0.0)
        out.append([torch.zeros_like(s.state) for _ in range(2)])
    torch.cuda.synchronize()

    def calls(s, o):
        C.check(s.lib.hweno_steps(s.h, 0.0, 2), "hweno_steps")
        C.check(s.lib.hweno_rhs(s.h, p(s.state), p(o[0]), p(o[1])), "hweno_rhs")

    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        calls(a, out[0])
    for _ in range(3):
        with torch.cuda.stream(st):
            g.replay()
        calls(b, out[1])
        torch.cuda.synchronize()
        assert torch.equal(a.state, b.state)
        for x, y in zip(out[0], out[1]):
            assert torch.equal(x, y)
    assert np.isfinite(a.state.cpu().numpy()).all()
    assert a.last_dt() == b.last_dt()
