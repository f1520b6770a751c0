"""Grids large enough for the pair arithmetic and its lists (forward from 19456 and 2^15 cells of 2D Euler,
38912 of a scalar law; the adjoint from 9728), the batches that take it, and the one-launch steps of 1D
grids at the edges of their blocks, with data that leave none, some and all of the cells and faces to the
FP64 weights, on the library the environment selects (HWENO_BOUNDS_CHECK=1: the bounds-checked build),
with the results saved to the .npz file named on the command line.  Run by
tests/test_gpu_bounds_lists.py as a child process, once per library.
"""
import ctypes
import os
import sys

import numpy as np
import torch

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))

import workloads as W  # noqa: E402
from paper_2411_11229_gb300 import Batch, Solver  # noqa: E402
from paper_2411_11229_gb300 import _capi as C  # noqa: E402

P, T, R, F = C.HWENO_BC_PERIODIC, C.HWENO_BC_TRANSMISSIVE, C.HWENO_BC_REFLECTIVE, C.HWENO_BC_FIXED
VW, CD2, R2, ALOC = (C.HWENO_FLAG_V_WEIGHTED, C.HWENO_FLAG_CD2, C.HWENO_FLAG_R2, C.HWENO_FLAG_ALPHA_LOCAL)


def _ptr(t):
    return ctypes.c_void_p(t.data_ptr())


def _flow(nx, ny, kind, seed=3):
    """none, some or all of the cells and faces left to the FP64 weights"""
    S, dx, dy = W.euler2d_random(nx, ny, seed=seed, kind="smooth")
    mean = S[0].mean(axis=(1, 2), keepdims=True)
    amp = 1e-3 if kind != "all" else 0.05
    S[0] = mean + amp * (S[0] - mean)
    S[1:] *= amp
    if kind == "some":
        S[0, :, : ny // 3, : nx // 2] *= 1.4
    if kind == "all":
        S[0] *= 1.0 + 0.05 * np.random.default_rng(7).uniform(-1.0, 1.0, size=S[0, :1].shape)
    return S, dx, dy


def forward(res):
    plain = (P, P, P, P)
    cases = [(140, 139, 0, plain), (141, 139, 0, (T,) * 4), (5, 3907, 0, (R,) * 4), (181, 181, 0, plain),
             (182, 181, 0, (R,) * 4), (257, 128, 0, (T,) * 4), (6, 5501, 0, (R,) * 4), (5501, 6, 0, (T,) * 4),
             (181, 183, CD2, (F, T, R, F)), (181, 183, ALOC, (F, R, P, P)), (150, 139, R2, (R, F, T, R)),
             (181, 183, R2, (F, R, R, F)), (181, 183, R2 | VW, (R, R, F, F)), (181, 183, VW, (T, F, P, P))]
    for nx, ny, flags, sides in cases:
        for kind in ("none", "some", "all"):
            S, dx, dy = _flow(nx, ny, kind)
            fixed = {k: S[0].mean(axis=(1, 2)) * (1.0 + 0.01 * k) for k in range(4)} if F in sides else None
            s = Solver(2, "euler", nx, ny, dx=dx, dy=dy, flags=flags, sides=sides, fixed=fixed)
            s.set_state(S)
            key = f"fwd_{nx}_{ny}_{flags}_{'_'.join(map(str, sides))}_{kind}"
            L, M = s.rhs()
            res[key + "_L"], res[key + "_M"] = L.cpu().numpy(), M.cpu().numpy()
            s.set_time(0.0, 0.0)
            s.step(0.0, 1)
            res[key + "_S1"] = s.state.cpu().numpy()
            s.close()
    for nx, ny, bc in ((199, 197, "periodic"), (7, 5601, "transmissive")):
        for kind in ("smooth", "jumps"):
            S, dx, dy = W.scalar_random(2, nx, ny, 5, kind)
            s = Solver(2, "burgers", nx, ny, dx=dx, dy=dy, bc=bc)
            s.set_state(S)
            L, M = s.rhs()
            key = f"scalar_{nx}_{ny}_{kind}"
            res[key + "_L"], res[key + "_M"] = L.cpu().numpy(), M.cpu().numpy()
            s.close()
    S, dx = W.euler1d_random(18851, 5, "jumps")
    s = Solver(1, "euler", 18851, dx=dx, bc="reflective")
    s.set_state(S)
    L, M = s.rhs()
    res["fwd1d_L"], res["fwd1d_M"] = L.cpu().numpy(), M.cpu().numpy()
    s.close()


def line(res):
    for n, system, bc in ((5, "euler", "periodic"), (28, "euler", "reflective"), (29, "burgers", "transmissive"),
                          (4256, "euler", "transmissive"), (4257, "euler", "periodic"), (18848, "euler", "reflective")):
        if system == "euler":
            S, dx = W.euler1d_smooth(n) if n < 10 else W.euler1d_random(n, 4, "jumps")
        else:
            S, dx, _ = W.scalar_random(1, n, 1, 4, "jumps")
        s = Solver(1, system, n, dx=dx, bc=bc)
        s.set_state(S)
        s.set_time(0.0, 0.0)
        s.step(0.0, 3)
        res[f"line_{n}_{system}_{bc}"] = s.state.cpu().numpy()
        s.close()


def adjoint(res):
    for nx, ny, bc in ((97, 101, "periodic"), (99, 99, "reflective"), (5, 1951, "transmissive"), (1951, 5, "reflective")):
        for kind in ("none", "some", "all"):
            S, dx, dy = _flow(nx, ny, kind, seed=nx)
            s = Solver(2, "euler", nx, ny, dx=dx, dy=dy, bc=bc)
            s.set_state(S)
            rng = np.random.default_rng(nx * 3 + ny)
            dev = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")
            Sd, lam_in = dev(S), dev(rng.normal(size=S.shape))
            rec = torch.empty(7, dtype=torch.float64, device="cuda")
            S1, S2 = torch.empty_like(Sd), torch.empty_like(Sd)
            s.set_time(0.0, 0.0)
            s.step_stages(S1, S2)
            s.record(rec)
            dt, a6 = float(rec[0].item()), rec[1:].contiguous()
            key = f"adj_{nx}_{ny}_{kind}"
            res[key + "_step"] = s.adjoint_step(Sd, dt, a6, lam_in).cpu().numpy()
            res[key + "_stages"] = s.adjoint_step_stages(Sd, S1, S2, dt, a6, lam_in).cpu().numpy()
            s.close()


def batch(res):
    for name, lines, grids in (("lines", [4001, 9001, 7003], []), ("grids", [], [(101, 103), (5, 130)]),
                               ("both", [12001, 8003, 6], [(128, 97)])):
        items = []
        for k, n in enumerate(lines):
            S, dx = W.euler1d_random(n, 1 + k, "jumps") if n > 9 else W.euler1d_smooth(n)
            items.append(({"dim": 1, "nx": n, "dx": dx, "bc": ("periodic", "transmissive", "reflective")[k % 3]}, S))
        for k, (nx, ny) in enumerate(grids):
            S, dx, dy = _flow(nx, ny, ("some", "all")[k % 2])
            items.append(({"dim": 2, "nx": nx, "ny": ny, "dx": dx, "dy": dy, "bc": ("reflective", "periodic")[k % 2]}, S))
        b = Batch([d for d, _ in items])
        for i, (_, S) in enumerate(items):
            b.set_state(i, S)
        b.set_time(0.0)
        b.step(1)
        b.tune()
        b.step(1)
        b.sync()
        for i in range(len(items)):
            res[f"batch_{name}_{i}"] = b.view(i).cpu().numpy()
        b.close()


def main(out):
    lib = C.load()
    checked = C.bounds_checked()
    res = {}
    for part in (forward, line, adjoint, batch):
        part(res)
    torch.cuda.synchronize()
    np.savez(out, **res)
    if checked:
        where = ctypes.c_int()
        n = int(lib.hweno_bounds_status(ctypes.byref(where)))
        print(f"bounds: out-of-range {n} first at {where.value}")
    print(f"arrays {len(res)}")


if __name__ == "__main__":
    main(sys.argv[1])
