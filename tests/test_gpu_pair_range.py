"""The pair arithmetic (csrc/hweno_pair.cuh) on 2D Euler grids that take it (more than 19456 cells), in units
and on meshes that FP32 does not hold: those cells and faces have to take the FP64 weights and fluxes.
Reference: the oracle's extended-precision evaluation, at the bars of the extended-precision tests."""
import numpy as np
import pytest

import oracle as O
import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2411_11229_gb300 import Solver  # noqa: E402

# without and with the grid's list (2^15 cells) of what is left to the FP64 weights
SIZES = [(211, 97), (197, 167)]


def _planes(a):
    return a.reshape(12, -1)


def _check(cfg, S, where=None, **kw):
    """L and M (at the cells where): per plane no further from the extended evaluation than three times the
    FP64 oracle's distance plus 1e-14."""
    s = Solver(cfg.dim, "euler", cfg.nx, cfg.ny, dx=cfg.dx, dy=cfg.dy, **kw)
    s.set_state(S)
    got = [t.cpu().numpy() for t in s.rhs()]
    for g, e, o in zip(got, O.rhs_ext(cfg, S)[:2], O.rhs(cfg, S)):
        g, e, o = (_planes(a if where is None else a[..., where]) for a in (g, e, o))
        scale = np.maximum(np.abs(e).max(axis=1), 1e-300)
        err, own = np.abs(g - e).max(axis=1) / scale, np.abs(o - e).max(axis=1) / scale
        assert (err <= 3.0 * own + 1e-14).all(), (err, own)


def _flow(nx, ny, kind):
    """A weak smooth wave; shear: momenta that change sign from block to block where density and energy
    are (nearly) the same on both sides."""
    S, dx, dy = W.euler2d_random(nx, ny, seed=5, kind="smooth")
    amp = 1e-2 if kind == "smooth" else 1e-6
    mean = S[0].mean(axis=(1, 2), keepdims=True)
    S[0] = mean + amp * (S[0] - mean)
    S[1:] *= amp
    if kind == "shear":
        S[0, 1, : ny // 2, : nx // 3] *= -1.0
        S[0, 2, ny // 4:, nx // 2:] *= -1.0
    return S, dx, dy


@pytest.mark.parametrize("flags", [0, O.FLAG_R2])
@pytest.mark.parametrize("nx,ny", SIZES)
@pytest.mark.parametrize("kind", ["smooth", "shear"])
@pytest.mark.parametrize("rho,vel", [(1e-40, 1.0), (1e-30, 1.0), (1e-30, 1e7), (1e-24, 1e6), (1e-20, 1e-4), (1e-20, 1.0),
                                     (1e-14, 1e-10), (1e-8, 1e-3), (1.0, 1e-15), (1.0, 300.0), (1.0, 1e12), (1e10, 1e-12),
                                     (1e20, 1e10), (1e30, 1.0)])
def test_euler_units(rho, vel, kind, nx, ny, flags):
    """The same flow in units of density rho and velocity vel."""
    S, dx, dy = _flow(nx, ny, kind)
    S = S * (rho * np.array([1.0, vel, vel, vel * vel])).reshape(1, 4, 1, 1)
    _check(O.make_cfg(2, O.EULER, nx, ny, dx=dx, dy=dy, flags=flags), S, flags=flags)


@pytest.mark.parametrize("flags", [0, O.FLAG_R2])
@pytest.mark.parametrize("nx,ny", SIZES)
@pytest.mark.parametrize("length", [1e-36, 1e-30, 1e-20, 1e-9, 1e9, 1e20, 1e30, 1e36])
def test_mesh_sizes(length, nx, ny, flags):
    """The same flow on a domain scaled by length."""
    S, dx, dy = _flow(nx, ny, "smooth")
    S[1:] /= length
    cfg = O.make_cfg(2, O.EULER, nx, ny, dx=dx * length, dy=dy * length, flags=flags)
    _check(cfg, S, flags=flags)


@pytest.mark.parametrize("flags", [0, O.FLAG_R2])
@pytest.mark.parametrize("nx,ny", SIZES)
@pytest.mark.parametrize("energy", [1e30, 1e70, 1e80, 1e160])
def test_one_cell_of_any_wavespeed(energy, nx, ny, flags):
    """A smooth flow but for one cell whose wavespeed (the Lax-Friedrichs coefficient of every face) goes
    through the end of the FP32 range: the cells out of its reach, where the dissipation is that
    coefficient times the small jumps of a smooth flow."""
    S, dx, dy = _flow(nx, ny, "smooth")
    S[0, 3, ny // 2, nx // 2] = energy
    far = np.ones((ny, nx), bool)
    far[ny // 2 - 4: ny // 2 + 5, :] = False
    far[:, nx // 2 - 4: nx // 2 + 5] = False
    _check(O.make_cfg(2, O.EULER, nx, ny, dx=dx, dy=dy, flags=flags), S, far, flags=flags)
