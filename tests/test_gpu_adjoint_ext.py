"""The stage VJP against the exact value of the adjoint formulas (the oracle's reverse mode in long double),
on both sides of the size from which a 2D VJP takes the nonlinear part in pairs (9728 cells): per plane no
further from it than three times the FP64 oracle plus 1e-14, the bars of the extended-precision tests.
Also the number of kernels that a VJP launches, and gradients of 1D rollouts from checkpoints and from
kept stage inputs."""
import ctypes

import numpy as np
import pytest

import oracle as O
import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2411_11229_gb300 import Solver  # noqa: E402
from paper_2411_11229_gb300 import _capi as C  # noqa: E402
from paper_2411_11229_gb300.adjoint import rollout  # noqa: E402


def _ptr(t):
    return ctypes.c_void_p(t.data_ptr())


def _vjp(s, S, al, mM, mL):
    Sd, a, b = (torch.as_tensor(np.ascontiguousarray(x), device="cuda") for x in (S, mM, mL))
    ad = torch.tensor([al[0], al[1]], dtype=torch.float64, device="cuda")
    lam, ws = torch.empty_like(Sd), s._adj_ws()
    C.check(s.lib.hweno_stage_vjp(s.h, _ptr(Sd), _ptr(ad), _ptr(a), _ptr(b), _ptr(lam), _ptr(ws)), "hweno_stage_vjp")
    return lam.cpu().numpy()


@pytest.mark.parametrize("nx,ny,amp,units,par", [
    (67, 41, 0.3, (1.0, 1.0), {}), (101, 97, 1e-3, (1.0, 1.0), {}), (101, 97, 1e-2, (1.0, 1.0), {}),
    (101, 97, 0.1, (1.0, 1.0), {}), (101, 97, 1e-2, (1.0, 1.0), {"gamma0": 0.5}),
    (101, 97, 3e-2, (1.0, 1.0), {"gamma0": 0.02, "d0": 0.5}), (101, 97, 1e-2, (1.0, 1.0), {"gamma0": 0.985, "d0": 0.02}),
    (101, 97, 1e-2, (1e-30, 1e7), {}), (101, 97, 1e-2, (1e-20, 1e-4), {}), (101, 97, 1e-2, (1e-14, 1e-10), {}),
    (101, 97, 1e-2, (1.0, 1e-15), {}), (101, 97, 1e-2, (1.0, 1e-17), {}), (101, 97, 1e-2, (1e10, 1e-12), {}),
    (101, 97, 1e-2, (1.0, 1e6), {})])
def test_stage_vjp(nx, ny, amp, units, par):
    S, dx, dy = W.euler2d_random(nx, ny, seed=11, kind="smooth")
    mean = S[0].mean(axis=(1, 2), keepdims=True)
    S[0] = mean + amp * (S[0] - mean)
    S[1:] *= amp
    rho, vel = units
    unit = (rho * np.array([1.0, vel, vel, vel * vel])).reshape(1, 4, 1, 1)
    S = S * unit
    cfg = O.make_cfg(2, O.EULER, nx, ny, dx=dx, dy=dy, **par)
    al = O.max_wavespeed(cfg, S)
    dt = O.cfl_dt(cfg, S, 0.6)
    r = np.random.default_rng(3)
    lam = r.normal(size=S.shape) / unit
    lam[1] *= dx
    lam[2] *= dy
    mM, mL = 2.0 / 3.0 * lam, 2.0 / 3.0 * dt * lam
    s = Solver(2, "euler", nx, ny, dx=dx, dy=dy, **par)
    got, ref, own = (a.reshape(12, -1) for a in (_vjp(s, S, al, mM, mL), O.stage_vjp_ext(cfg, S, al, mM, mL),
                                                 O.stage_vjp(cfg, S, al, mM, mL)))
    scale = np.abs(ref).max(axis=1)
    err, own = np.abs(got - ref).max(axis=1) / scale, np.abs(own - ref).max(axis=1) / scale
    assert (err <= 3.0 * own + 1e-14).all(), (err, own)


@pytest.mark.parametrize("dim,nx,ny,kernels", [(1, 300, 1, 3), (2, 40, 33, 3), (2, 97, 100, 3), (2, 128, 76, 5),
                                               (2, 101, 97, 5)])
def test_launch_counts(dim, nx, ny, kernels):
    """Three kernels a VJP; five where the pairs' kernels come before those of their lists (from 9728
    cells).  A step's adjoint is three VJPs and three passes over the state."""
    if dim == 2:
        S, dx, dy = W.euler2d_random(nx, ny, seed=1, kind="smooth")
    else:
        S, dx = W.euler1d_random(nx, seed=1, kind="smooth")
        dy = dx
    s = Solver(dim, "euler", nx, ny, dx=dx, dy=dy)
    s.set_state(S)
    r = np.random.default_rng(0)
    n0 = s.launch_count()
    _vjp(s, S, (2.0, 2.0), r.normal(size=S.shape), r.normal(size=S.shape))
    n1 = s.launch_count()
    assert n1 - n0 == kernels
    Sd = s.state.clone()
    al = torch.full((6,), 2.0, dtype=torch.float64, device="cuda")
    s.adjoint_step_stages(Sd, Sd, Sd, 1e-4, al, torch.ones_like(Sd))
    assert s.launch_count() - n1 == 3 * kernels + 3
    torch.cuda.synchronize()


# four warps to a block's cells, one block; 152 blocks; a thread to a cell; stage kernels
@pytest.mark.parametrize("n", [21, 300, 4256, 5000, 18849])
@pytest.mark.parametrize("bc,kind", [("periodic", "smooth"), ("transmissive", "jumps"), ("reflective", "smooth")])
def test_rollout_1d_same_gradient_from_checkpoints(n, bc, kind):
    S, dx = W.euler1d_random(n, seed=n, kind=kind)
    grads, ends = [], []
    for keep in (False, True):
        s = Solver(1, "euler", n, dx=dx, bc=bc)
        S0 = torch.as_tensor(S, device="cuda").requires_grad_(True)
        ST = rollout(S0, s, 5, every=2, keep_stages=keep)
        (0.5 * (ST[0, 0] ** 2).sum() * dx).backward()
        grads.append(S0.grad.clone())
        ends.append(ST.detach().clone())
    assert torch.equal(ends[0], ends[1])
    assert torch.equal(grads[0], grads[1])
