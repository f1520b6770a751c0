"""The library's square root and reciprocal square root (hardware approximation and one third-order step)
against the correctly rounded ones: at most one unit in the last place, over the range of double, at its
ends, beside powers of four (where the unit changes) and for denormals; and a state whose squared sound
speed is a denormal."""
import ctypes
from decimal import Decimal, localcontext

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2411_11229_gb300 import Solver  # noqa: E402
from paper_2411_11229_gb300 import _capi as C  # noqa: E402


def _eval(x):
    xd = torch.as_tensor(x, device="cuda")
    s, r = torch.empty_like(xd), torch.empty_like(xd)
    p = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    C.check(C.load().hweno_selftest_sqrt(p(xd), p(s), p(r), x.size,
                                         ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)), "hweno_selftest_sqrt")
    return s.cpu().numpy(), r.cpu().numpy()


def test_against_the_correctly_rounded_ones():
    rng = np.random.default_rng(23)
    f = np.finfo(np.float64)
    near = np.ldexp(1.0, 2 * rng.integers(-500, 500, 2000)) * (1.0 + f.eps * rng.integers(-8, 9, 2000))
    x = np.concatenate([rng.uniform(1.0, 4.0, 200000) * 4.0 ** rng.integers(-510, 510, 200000), near,
                        [f.tiny, f.max, np.nextafter(f.tiny, 1.0), 1.0, 2.0, 4.0, np.nextafter(1.0, 0.0)],
                        np.ldexp(rng.uniform(0.5, 1.0, 200), -1022 - rng.integers(0, 51, 200)), [5e-324, 1e-323]])
    s, r = _eval(x)
    exact = np.sqrt(x)
    assert (np.abs(s - exact) <= np.spacing(exact)).all()
    # 1/sqrt(x) to 40 digits, for a part of them
    pick = np.concatenate([np.arange(0, 200000, 40), np.arange(200000, x.size)])
    with localcontext() as ctx:
        ctx.prec = 40
        for i in pick:
            e = 1 / Decimal(float(x[i])).sqrt()
            assert abs(Decimal(float(r[i])) - e) <= Decimal(float(np.spacing(float(e)))), (x[i], r[i])


def test_what_has_no_root():
    s, r = _eval(np.array([0.0, -1.0, -5e-324, np.inf, np.nan, -np.inf]))
    assert np.isnan(s).all() and np.isnan(r).all()


@pytest.mark.parametrize("dim", [1, 2])
def test_denormal_sound_speed_squared(dim):
    """A gas at rest whose squared sound speed is below the normal range is a physical state."""
    n = 16
    s = Solver(dim, "euler", n, n if dim == 2 else 1, dx=0.1)
    S = torch.zeros_like(s.state)
    S[0, 0] = 1.0
    S[0, -1] = 1e-309
    s.set_state(S)
    s.rhs()
    s.sync()
    a = s.max_wavespeed()[0]
    assert abs(a - np.sqrt(1.4 * 0.4 * 1e-309)) <= 1e-13 * a
