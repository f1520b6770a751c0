"""The nonlinear part of the interpolation in pairs of FP32 values (csrc/hweno_pair.cuh) against the
oracle's extended-precision evaluation: where the pairs take over from the FP64 weights, beside
fronts, at ragged sizes, and outside the range that FP32 holds (where the FP64 weights are used)."""
import numpy as np
import pytest

import oracle as O
import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2411_11229_gb300 import Solver  # noqa: E402


def _planes(a):
    return a.reshape(a.shape[0] * a.shape[1], -1)


def _check(got, ref, plain):
    """Per plane: no further from the extended evaluation than three times the FP64 oracle's distance
    plus 1e-14 (the bar of the extended-precision tests)."""
    scale = np.maximum(np.abs(_planes(ref)).max(axis=1), 1e-300)
    err = np.abs(_planes(got) - _planes(ref)).max(axis=1) / scale
    own = np.abs(_planes(plain) - _planes(ref)).max(axis=1) / scale
    assert (err <= 3.0 * own + 1e-14).all(), (err, own)


def _rhs(cfg, S, **kw):
    s = Solver(cfg.dim, kw.pop("system"), cfg.nx, cfg.ny, dx=cfg.dx, dy=cfg.dy, **kw)
    s.set_state(S)
    L, M = s.rhs()
    return L.cpu().numpy(), M.cpu().numpy()


@pytest.mark.parametrize("flags", [0, O.FLAG_R2 if hasattr(O, "FLAG_R2") else 4])
@pytest.mark.parametrize("amp", [1e-6, 1e-3, 1e-2, 3e-2, 0.1, 0.3])
def test_euler_amplitude_sweep(amp, flags):
    """Waves whose second differences run through the bound of the pairs (max t = 2^-14), with a jump
    in one corner, on a ragged grid."""
    nx, ny = 67, 41
    S, dx, dy = W.euler2d_random(nx, ny, seed=5, kind="smooth")
    mean = S[0].mean(axis=(1, 2), keepdims=True)
    S[0] = mean + amp * (S[0] - mean)
    S[1:] *= amp
    S[0, 0, :7, :9] *= 1.5
    S[0, 3, :7, :9] *= 1.5
    cfg = O.make_cfg(2, O.EULER, nx, ny, dx=dx, dy=dy, flags=flags)
    L, M = _rhs(cfg, S, system="euler", flags=flags)
    Le, Me = O.rhs_ext(cfg, S)[:2]
    Lo, Mo = O.rhs(cfg, S)
    _check(L, Le, Lo)
    _check(M, Me, Mo)


@pytest.mark.parametrize("n", [19456, 19457, 20001])
@pytest.mark.parametrize("kind", ["smooth", "jumps"])
def test_euler_1d_sides_of_the_size_rule(n, kind):
    S, dx = W.euler1d_random(n, seed=9, kind=kind)
    cfg = O.make_cfg(1, O.EULER, n, dx=dx, bc=O.BC_TRANSMISSIVE)
    L, M = _rhs(cfg, S, system="euler", bc="transmissive")
    Le, Me = O.rhs_ext(cfg, S)[:2]
    Lo, Mo = O.rhs(cfg, S)
    _check(L, Le, Lo)
    _check(M, Me, Mo)


@pytest.mark.parametrize("scale", [1e-45, 1e-20, 1e-8, 1.0, 1e8, 1e25, 1e30])
@pytest.mark.parametrize("system", ["advection", "burgers"])
def test_scalar_scales(system, scale):
    """Values below, inside and above the FP32 range."""
    nx, ny = 45, 33
    S, dx, dy = W.scalar_random(2, nx, ny, seed=3, kind="smooth")
    S = S * scale
    cfg = O.make_cfg(2, getattr(O, system.upper()), nx, ny, dx=dx, dy=dy)
    L, M = _rhs(cfg, S, system=system)
    Le, Me = O.rhs_ext(cfg, S)[:2]
    Lo, Mo = O.rhs(cfg, S)
    _check(L, Le, Lo)
    _check(M, Me, Mo)


@pytest.mark.parametrize("eps", [1e-40, 1e-20, 1e-6, 1.0])
def test_epsilon_range(eps):
    nx, ny = 40, 37
    S, dx, dy = W.euler2d_random(nx, ny, seed=8, kind="smooth")
    cfg = O.make_cfg(2, O.EULER, nx, ny, dx=dx, dy=dy, eps=eps)
    L, M = _rhs(cfg, S, system="euler", eps=eps)
    Le, Me = O.rhs_ext(cfg, S)[:2]
    Lo, Mo = O.rhs(cfg, S)
    _check(L, Le, Lo)
    _check(M, Me, Mo)


def test_constant_state_stays_constant():
    nx, ny = 130, 5
    S = np.zeros((3, 4, ny, nx))
    S[0] = np.array([1.3, 0.4, -0.2, 2.5]).reshape(4, 1, 1)
    cfg = O.make_cfg(2, O.EULER, nx, ny, dx=0.1, dy=0.3)
    L, M = _rhs(cfg, S, system="euler")
    assert np.array_equal(M, S)
    assert np.abs(L).max() <= 1e-13
