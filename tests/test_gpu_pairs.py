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


@pytest.mark.parametrize("n", [18848, 18849, 20001])
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


@pytest.mark.parametrize("kind", ["smooth", "jumps"])
@pytest.mark.parametrize("nx,ny,bc", [(67, 41, "periodic"), (5, 130, "transmissive"), (40, 33, "reflective"),
                                      # both sides of the size from which the pairs are used (9728 cells)
                                      (97, 100, "periodic"), (128, 76, "periodic"), (101, 97, "reflective"),
                                      (13, 801, "transmissive"), (801, 13, "reflective")])
def test_adjoint_scales_with_its_seeds(nx, ny, bc, kind):
    """The stage VJP against the oracle's (1e-10, the bar of the adjoint tests), and exactly linear under
    powers of two of any size: the pairs take each thread's seeds relative to their largest."""
    import ctypes

    from paper_2411_11229_gb300 import capi as C

    S, dx, dy = W.euler2d_random(nx, ny, seed=nx, kind="smooth")
    if kind == "jumps":
        S[0, 0, : ny // 3, : nx // 2] *= 1.4
        S[0, 3, : ny // 3, : nx // 2] *= 1.4
    cfg = O.make_cfg(2, O.EULER, nx, ny, dx=dx, dy=dy, bc=getattr(O, "BC_" + bc.upper()))
    al = O.max_wavespeed(cfg, S)
    r = np.random.default_rng(1)
    mM, mL = r.normal(size=S.shape), 1e-3 * r.normal(size=S.shape)
    s = Solver(2, "euler", nx, ny, dx=dx, dy=dy, bc=bc)
    ws, out = s._adj_ws(), []
    p = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    Sd, ad = torch.as_tensor(S, device="cuda"), torch.tensor([al[0], al[1]], dtype=torch.float64, device="cuda")
    for e in (0, 300, -300, -850):
        a, b = (torch.as_tensor(np.ldexp(m, e), device="cuda") for m in (mM, mL))
        lam = torch.empty_like(Sd)
        C.check(s.lib.hweno_stage_vjp(s.h, p(Sd), p(ad), p(a), p(b), p(lam), p(ws)), "hweno_stage_vjp")
        out.append(np.ldexp(lam.cpu().numpy(), -e))
    ref = O.stage_vjp(cfg, S, al, mM, mL)
    for k in range(4):
        err = np.abs(_planes(out[k]) - _planes(ref)).max(axis=1) / np.abs(_planes(ref)).max(axis=1)
        assert (err <= 1e-10).all(), (k, err)
    assert np.array_equal(out[0], out[1]) and np.array_equal(out[0], out[2])


@pytest.mark.parametrize("kind", ["none", "corner", "all"])
@pytest.mark.parametrize("system,nx,ny,bc,flags", [
    ("euler", 181, 181, "periodic", 0), ("euler", 128, 256, "periodic", 0), ("euler", 1001, 33, "reflective", 0),
    ("euler", 33, 1001, "transmissive", 4), ("burgers", 256, 129, "periodic", 0)])
def test_left_to_the_fp64_weights(system, nx, ny, bc, flags, kind):
    """Grids on both sides of the size from which the cells and faces of the FP64 weights go through the
    grid's list (2^15 cells), with none, some and every one of them in it; again on a handle whose list
    has been used."""
    if system == "euler":
        S, dx, dy = W.euler2d_random(nx, ny, seed=2, kind="smooth")
        mean = S[0].mean(axis=(1, 2), keepdims=True)
    else:
        S, dx, dy = W.scalar_random(2, nx, ny, seed=2, kind="smooth")
        mean = 0.3 + 0 * S[0].mean(axis=(1, 2), keepdims=True)
    amp = 1e-3 if kind != "all" else 0.05
    S[0] = mean + amp * (S[0] - mean)
    S[1:] *= amp
    if kind == "corner":
        S[0, 0, : ny // 3, : nx // 4] *= 1.5
    if kind == "all":
        r = np.random.default_rng(7)
        S[0] *= 1.0 + 0.1 * r.uniform(-1.0, 1.0, size=S[0, :1].shape)
    cfg = O.make_cfg(2, getattr(O, system.upper()), nx, ny, dx=dx, dy=dy, bc=getattr(O, "BC_" + bc.upper()),
                     flags=flags)
    s = Solver(2, system, nx, ny, dx=dx, dy=dy, bc=bc, flags=flags)
    Le, Me = O.rhs_ext(cfg, S)[:2]
    Lo, Mo = O.rhs(cfg, S)
    for _ in range(2):
        s.set_state(S)
        L, M = s.rhs()
        _check(L.cpu().numpy(), Le, Lo)
        _check(M.cpu().numpy(), Me, Mo)
        s.set_time(0.0, 0.0)
        s.step(0.0, 2)
    s.sync()
