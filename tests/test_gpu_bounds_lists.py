"""The bounds-checked build (libhweno_bounds.so) on grids large enough for the pair arithmetic and its lists:
tests/bounds_sweep_lists.py on each library, in child processes.  The checked build, which checks the
entries and the places of the lists as well, must record no out-of-range index, and both builds must give
the same results bit for bit."""
import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

HERE = os.path.dirname(os.path.abspath(__file__))
SWEEP = os.path.join(HERE, "bounds_sweep_lists.py")


def _sweep(out, checked):
    env = dict(os.environ)
    env.pop("HWENO_BOUNDS_CHECK", None)
    if checked:
        env["HWENO_BOUNDS_CHECK"] = "1"
    r = subprocess.run([sys.executable, SWEEP, str(out)], env=env, capture_output=True, text=True, timeout=600,
                       cwd=os.path.dirname(HERE))
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-3000:]
    return r.stdout


def test_bounds_checked_build_sweep_of_lists(tmp_path):
    log = _sweep(tmp_path / "checked.npz", True)
    assert "bounds: out-of-range 0 " in log, log
    _sweep(tmp_path / "plain.npz", False)
    a, b = np.load(tmp_path / "checked.npz"), np.load(tmp_path / "plain.npz")
    assert sorted(a.files) == sorted(b.files) and len(a.files) > 150
    differ = [k for k in a.files if not np.array_equal(a[k], b[k], equal_nan=True)]
    assert not differ, differ[:10]
