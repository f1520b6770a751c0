"""Batches on both sides of the size from which their lines and their grids take the nonlinear part in pairs
(19456 faces of either): every member's step against the oracle's extended-precision evaluation, at the
bars of the extended-precision tests, and the same step again after the autotuner."""
import numpy as np
import pytest

import oracle as O
import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2411_11229_gb300 import Batch  # noqa: E402

BCS = ("periodic", "transmissive", "reflective")


def _bar(got, ext, own):
    got, ext, own = (a.reshape(a.shape[0] * a.shape[1], -1) for a in (got, ext, own))
    scale = np.maximum(np.abs(ext).max(axis=1), 1e-300)
    err, ref = np.abs(got - ext).max(axis=1) / scale, np.abs(own - ext).max(axis=1) / scale
    assert (err <= 3.0 * ref + 1e-14).all(), (err, ref)


@pytest.mark.parametrize("lines,grids", [
    ([128], []), ([300, 7001, 9000], []),                # FP64 lines
    ([9700, 9753], []), ([9700, 9754], []),              # 19455 and 19456 faces
    ([9700, 9755], []), ([12001, 128, 9003], []),        # 19457: pairs
    ([], [(40, 33)]), ([], [(98, 98)]), ([], [(99, 98)]), ([], [(101, 97), (5, 40)]),
    ([200, 4000], [(128, 97)]), ([20011], [(33, 21)]), ([20011, 130], [(128, 97), (64, 64)])])
def test_members_of_batches(lines, grids):
    items = []
    for k, n in enumerate(lines):
        S, dx = W.euler1d_random(n, 3 + k, ("jumps", "smooth")[k % 2])
        items.append(({"dim": 1, "nx": n, "dx": dx, "bc": BCS[k % 3]}, S, O.make_cfg(1, O.EULER, n, dx=dx, bc=k % 3)))
    for k, (nx, ny) in enumerate(grids):
        S, dx, dy = W.euler2d_random(nx, ny, 5 + k, "smooth")
        mean = S[0].mean(axis=(1, 2), keepdims=True)
        S[0] = mean + 1e-2 * (S[0] - mean)
        S[1:] *= 1e-2
        S[:, :, : ny // 3, : nx // 3] *= 1.3
        items.append(({"dim": 2, "nx": nx, "ny": ny, "dx": dx, "dy": dy, "bc": BCS[k % 3]}, S,
                      O.make_cfg(2, O.EULER, nx, ny, dx=dx, dy=dy, bc=k % 3)))
    t_end = 0.9 * min(O.cfl_dt(c, S, 0.6) for _, S, c in items)
    b = Batch([d for d, _, _ in items])
    first = []
    for again in range(2):
        for i, (_, S, _) in enumerate(items):
            b.set_state(i, S)
        b.set_time(t_end)
        b.step(1)
        b.sync()
        out = [b.view(i).cpu().numpy() for i in range(len(items))]
        if again:
            assert all(np.array_equal(x, y) for x, y in zip(first, out))
            break
        first = out
        for got, (_, S, c) in zip(out, items):
            ext, n, _ = O.run_ext(c, S, t_end)
            assert n == 1
            _bar(got, ext, O.run(c, S, t_end)[0])
        b.tune()
    b.close()
