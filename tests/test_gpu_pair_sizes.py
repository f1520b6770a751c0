"""The pair arithmetic on grids large enough to take it, by both ways of taking what it leaves to the FP64
weights (block by block; in the grid's list from 2^15 cells): every variant, side and source, and the
amplitudes, scales and eps of its bounds.  Reference: the oracle's extended-precision evaluation, at the
bars of the extended-precision tests.  How a grid takes the nonlinear part shows in its workspace (the
list) and in the launches of an evaluation (k_left)."""
import numpy as np
import pytest

import oracle as O
import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2411_11229_gb300 import Solver  # noqa: E402

P, T, R, F = O.BC_PERIODIC, O.BC_TRANSMISSIVE, O.BC_REFLECTIVE, O.BC_FIXED
VW, CD2, R2, AST, ALOC = (O.FLAG_V_WEIGHTED, O.FLAG_CD2, O.FLAG_R2, O.FLAG_ALPHA_STEP, O.FLAG_ALPHA_LOCAL)


def _planes(a):
    return a.reshape(a.shape[0] * a.shape[1], -1)


def _bar(got, ext, own):
    """Per plane no further from the extended evaluation than three times the FP64 oracle plus 1e-14."""
    got, ext, own = _planes(got), _planes(ext), _planes(own)
    scale = np.maximum(np.abs(ext).max(axis=1), 1e-300)
    err, ref = np.abs(got - ext).max(axis=1) / scale, np.abs(own - ext).max(axis=1) / scale
    assert (err <= 3.0 * ref + 1e-14).all(), (err, ref)


def _data(nx, ny, seed=5, amp=1e-3):
    """A smooth flow of the given amplitude with a front about a third of the grid, in every field."""
    S, dx, dy = W.euler2d_random(nx, ny, seed=seed, kind="smooth")
    mean = S[0].mean(axis=(1, 2), keepdims=True)
    S[0] = mean + amp * (S[0] - mean)
    S[1:] *= amp
    S[0, :, : ny // 3, : nx // 4] *= 1.4
    S[1:, :, : ny // 3, : nx // 4] *= 1.4
    return S, dx, dy


def _fixed(S):
    U = S[0]
    return {0: U[:, :, 0].mean(axis=1) * 1.001, 1: U[:, :, -1].mean(axis=1) * 0.97,
            2: U[:, 0, :].mean(axis=1) * 1.02, 3: U[:, -1, :].mean(axis=1) * 0.9999}


@pytest.mark.parametrize("nx,ny", [(211, 97), (97, 211), (197, 167), (131, 257)])
@pytest.mark.parametrize("flags,sides,grav", [
    (0, (F, R, T, F), 0.0), (0, (R, R, F, F), 1.0), (CD2, (P, P, R, T), 0.0), (ALOC, (F, T, P, P), 0.0),
    (ALOC | CD2, (R, F, F, R), -0.7), (AST, (T, R, P, P), 0.0), (AST | ALOC, (P, P, F, T), 0.0), (VW, (R, F, T, R), 1.0),
    (VW | CD2, (P, P, P, P), 0.0), (R2, (F, R, R, F), 1.0), (R2 | ALOC, (P, P, T, F), 0.0), (R2 | VW, (R, T, F, R), 0.0),
    (R2 | VW | CD2 | AST, (T, F, R, R), 0.0)])
def test_variants(flags, sides, grav, nx, ny):
    """One stage and one clamped step (three stages: the held coefficient, the list used again)."""
    S, dx, dy = _data(nx, ny)
    fixed = _fixed(S) if F in sides else None
    cfg = O.make_cfg(2, O.EULER, nx, ny, dx=dx, dy=dy, flags=flags, sides=sides, fixed=fixed, grav=grav)
    s = Solver(2, "euler", nx, ny, dx=dx, dy=dy, flags=flags, sides=sides, fixed=fixed, grav=grav)
    s.set_state(S)
    n0 = s.launch_count()
    L, M = s.rhs()
    listed = nx * ny >= 2 ** 15 and not flags & VW
    assert s.launch_count() - n0 == 3 + listed + bool(flags & R2)
    for got, ext, own in zip((L, M), O.rhs_ext(cfg, S)[:2], O.rhs(cfg, S)):
        _bar(got.cpu().numpy(), ext, own)
    t_end = 0.9 * O.cfl_dt(cfg, S, 0.6)
    assert s.run(t_end) == 1
    ext, n, _ = O.run_ext(cfg, S, t_end)
    own, _, _ = O.run(cfg, S, t_end)
    assert n == 1
    _bar(s.state.cpu().numpy(), ext, own)


@pytest.mark.parametrize("flags", [0, R2])
@pytest.mark.parametrize("nx,ny", [(211, 97), (197, 167)])
@pytest.mark.parametrize("amp", [1e-6, 1e-3, 3e-2, 0.1, 0.3, 1.0])
def test_amplitudes(amp, nx, ny, flags):
    """Second differences through the bound of the pairs (max t = 2^-14)."""
    S, dx, dy = _data(nx, ny, seed=7, amp=amp)
    cfg = O.make_cfg(2, O.EULER, nx, ny, dx=dx, dy=dy, flags=flags)
    s = Solver(2, "euler", nx, ny, dx=dx, dy=dy, flags=flags)
    s.set_state(S)
    for got, ext, own in zip(s.rhs(), O.rhs_ext(cfg, S)[:2], O.rhs(cfg, S)):
        _bar(got.cpu().numpy(), ext, own)


@pytest.mark.parametrize("flags", [0, R2])
@pytest.mark.parametrize("par", [{"eps": 1e-40}, {"eps": 1e-20}, {"eps": 1e-6}, {"eps": 1.0}, {"gamma0": 0.5},
                                 {"gamma0": 0.02, "d0": 0.5}, {"d0": 0.02}])
def test_parameters(par, flags):
    nx, ny = 197, 167
    S, dx, dy = _data(nx, ny, seed=9, amp=0.1)
    cfg = O.make_cfg(2, O.EULER, nx, ny, dx=dx, dy=dy, flags=flags, **par)
    s = Solver(2, "euler", nx, ny, dx=dx, dy=dy, flags=flags, **par)
    s.set_state(S)
    for got, ext, own in zip(s.rhs(), O.rhs_ext(cfg, S)[:2], O.rhs(cfg, S)):
        _bar(got.cpu().numpy(), ext, own)


@pytest.mark.parametrize("system", ["advection", "burgers"])
@pytest.mark.parametrize("nx,ny,sides", [(211, 199, (P, P, P, P)), (199, 197, (T, F, F, T))])
@pytest.mark.parametrize("scale", [1e-45, 1e-20, 1e-8, 1.0, 1e8, 1e25, 1e30])
def test_scalar_scales(scale, nx, ny, sides, system):
    """Values below, inside and above the FP32 range, with a jump (from 38912 cells)."""
    S, dx, dy = W.scalar_random(2, nx, ny, seed=3, kind="smooth")
    S[0, 0, : ny // 3, : nx // 4] += 0.4
    S = S * scale
    fixed = {k: S[0].mean(axis=(1, 2)) for k in range(4)} if F in sides else None
    kw = dict(dx=dx, dy=dy, sides=sides, fixed=fixed, ax=0.8, ay=-0.6)
    cfg = O.make_cfg(2, getattr(O, system.upper()), nx, ny, **kw)
    s = Solver(2, system, nx, ny, **kw)
    s.set_state(S)
    for got, ext, own in zip(s.rhs(), O.rhs_ext(cfg, S)[:2], O.rhs(cfg, S)):
        _bar(got.cpu().numpy(), ext, own)


@pytest.mark.parametrize("system,nx,ny,bc,listed", [("burgers", 256, 153, "periodic", True),
                                                    ("burgers", 256, 151, "transmissive", False)])
@pytest.mark.parametrize("kind", ["none", "all"])
def test_scalar_list(system, nx, ny, bc, listed, kind):
    """A scalar grid with none and with every cell and face left to the FP64 weights, twice."""
    S, dx, dy = W.scalar_random(2, nx, ny, seed=2, kind="smooth")
    if kind == "none":
        S[0] = 0.3 + 1e-3 * (S[0] - 0.3)
        S[1:] *= 1e-3
    else:
        S[0] *= 1.0 + 0.1 * np.random.default_rng(7).uniform(-1.0, 1.0, size=S[0].shape)
    cfg = O.make_cfg(2, O.BURGERS, nx, ny, dx=dx, dy=dy, bc=getattr(O, "BC_" + bc.upper()))
    s = Solver(2, system, nx, ny, dx=dx, dy=dy, bc=bc)
    ext, own = O.rhs_ext(cfg, S)[:2], O.rhs(cfg, S)
    for _ in range(2):
        s.set_state(S)
        n0 = s.launch_count()
        out = s.rhs()
        assert s.launch_count() - n0 == 3 + listed
        for g, e, o in zip(out, ext, own):
            _bar(g.cpu().numpy(), e, o)
        s.step(0.0, 1)
    s.sync()


@pytest.mark.parametrize("flags", [0, R2])
@pytest.mark.parametrize("nx,ny", [(4001, 5), (211, 97), (197, 167)])
def test_constant_state_stays_constant(nx, ny, flags):
    S = np.zeros((3, 4, ny, nx))
    S[0] = np.array([1.3, 0.4, -0.2, 2.5]).reshape(4, 1, 1)
    s = Solver(2, "euler", nx, ny, dx=0.1, dy=0.3, flags=flags)
    s.set_state(S)
    L, M = (t.cpu().numpy() for t in s.rhs())
    assert np.array_equal(M, S)
    assert np.abs(L).max() <= 1e-13


@pytest.mark.parametrize("kind", ["smooth", "jumps"])
@pytest.mark.parametrize("n,kernels", [(18848, "line"), (18849, "stages"), (19455, "stages"), (19456, "stages"), (30011, "stages")])
def test_sides_of_the_1d_rules(n, kernels, kind):
    """Steps in one launch up to 18848 cells, pairs from 19456 (a second warp of faces to a scheduler)."""
    S, dx = W.euler1d_random(n, seed=9, kind=kind)
    cfg = O.make_cfg(1, O.EULER, n, dx=dx, bc=T)
    s = Solver(1, "euler", n, dx=dx, bc="transmissive")
    s.set_state(S)
    for got, ext, own in zip(s.rhs(), O.rhs_ext(cfg, S)[:2], O.rhs(cfg, S)):
        _bar(got.cpu().numpy(), ext, own)
    s.set_time(0.0, 0.0)
    n0 = s.launch_count()
    s.step(0.0, 2)
    assert s.launch_count() - n0 == (1 if kernels == "line" else 18)
    s.sync()
