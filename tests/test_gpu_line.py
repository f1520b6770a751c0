"""Steps of a small 1D grid in one cooperative launch (csrc/hweno_line.cu) against the same steps through
the stage kernels (taken while per-kernel timing is on): block edges, boundaries, ends of runs."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2411_11229_gb300 import Solver  # noqa: E402


def _pair(system, n, bc, S, dx):
    out = []
    for stage_kernels in (False, True):
        s = Solver(1, system, n, dx=dx, bc=bc)
        s.set_profiling(stage_kernels)
        s.set_state(S)
        out.append(s)
    return out


def _same(a, b):
    x, y = a.state.cpu().numpy(), b.state.cpu().numpy()
    scale = np.abs(y).reshape(y.shape[0] * y.shape[1], -1).max(axis=1)
    err = np.abs(x - y).reshape(scale.size, -1).max(axis=1)
    assert (err <= 1e-12 * np.maximum(scale, 1e-300)).all(), err / scale
    (dt, t), (dt2, t2) = a.last_dt(), b.last_dt()
    assert abs(dt - dt2) <= 1e-13 * dt2 and abs(t - t2) <= 1e-13 * t2


# one block's cells are 124: one block, its edge, two and three blocks of uneven sizes, the largest grid
@pytest.mark.parametrize("n", [5, 6, 17, 123, 124, 125, 247, 248, 249, 1000, 18848])
@pytest.mark.parametrize("bc", ["periodic", "transmissive", "reflective"])
def test_steps_euler(n, bc):
    S, dx = W.euler1d_random(n, seed=n, kind="smooth" if n % 2 else "jumps")
    if n <= 6:  # too coarse for the random modes: a mild wave
        S, dx = W.euler1d_smooth(n)
    a, b = _pair("euler", n, bc, S, dx)
    for s in (a, b):
        s.set_time(0.0, 0.0)
        s.step(0.0, 3)
        s.step(1e-4 * dx, 1)
        s.step(0.0, 2)
    _same(a, b)


# four warps to a block's cells: 28 of them at most, up to 152 blocks
@pytest.mark.parametrize("n", [27, 28, 29, 56, 57, 59, 4255, 4256, 4257])
@pytest.mark.parametrize("system,bc", [("advection", "periodic"), ("advection", "transmissive"),
                                       ("burgers", "periodic"), ("burgers", "transmissive"), ("euler", "periodic"),
                                       ("euler", "transmissive"), ("euler", "reflective")])
def test_steps_four_warps(system, n, bc):
    if system == "euler":
        S, dx = W.euler1d_random(n, seed=n, kind="smooth" if n % 2 else "jumps")
    else:
        S, dx, _ = W.scalar_random(1, n, 1, seed=n, kind="smooth" if n % 2 else "jumps")
    a, b = _pair(system, n, bc, S, dx)
    for s in (a, b):
        s.set_time(0.0, 0.0)
        s.step(0.0, 3)
        s.step(1e-4 * dx, 1)
        s.step(0.0, 2)
    _same(a, b)


@pytest.mark.parametrize("system", ["advection", "burgers"])
@pytest.mark.parametrize("n", [40, 124, 125, 161, 3001])
def test_steps_scalar(system, n):
    S, dx, _ = W.scalar_random(1, n, 1, seed=4, kind="smooth")
    a, b = _pair(system, n, "periodic", S, dx)
    for s in (a, b):
        s.set_time(0.0, 0.0)
        s.step(0.0, 5)
    _same(a, b)


@pytest.mark.parametrize("n,t_end,most", [(160, 0.31, 10 ** 9), (160, 1e-9, 10 ** 9), (300, 5.0, 37), (130, 0.2, 16)])
def test_run(n, t_end, most):
    """To the end time, past it in the first step, and to a step limit."""
    S, dx = W.advection_1d(n)
    a, b = _pair("advection", n, "periodic", S, dx)
    assert a.run(t_end, most) == b.run(t_end, most)
    _same(a, b)
    # steps at the end time change nothing
    x = a.state.clone()
    if most > 10 ** 6:
        a.step(0.0, 4)
        assert torch.equal(a.state, x)


def test_record_and_two_streams():
    """The recorded wavespeeds are those of the stage kernels; two handles on two streams at once."""
    S, dx, _ = W.euler1d_riemann(2048, seed=1001)
    a, b = _pair("euler", 2048, "transmissive", S, dx)
    recs = []
    for s in (a, b):
        s.step(0.0, 4)
        r = torch.zeros(7, dtype=torch.float64, device="cuda")
        s.record(r)
        recs.append(r.cpu().numpy())
    assert np.abs(recs[0] - recs[1]).max() <= 1e-13 * np.abs(recs[1]).max()
    st = [torch.cuda.Stream() for _ in range(2)]
    hs = [Solver(1, "euler", 2048, dx=dx, bc="transmissive", stream=q) for q in st]
    for s in hs:
        s.set_state(S)
    for _ in range(5):
        for s in hs:
            s.step(0.0, 2)
    torch.cuda.synchronize()
    assert torch.equal(hs[0].state, hs[1].state)


def test_non_physical_state_is_reported():
    S, dx = W.euler1d_smooth(300)
    S[0, 0, 0, 150] = -1.0
    s = Solver(1, "euler", 300, dx=dx)
    s.set_state(S)
    s.step(0.0, 2)
    with pytest.raises(Exception, match="non-physical"):
        s.sync()
