"""The adjoint's entry points on a handle without a bound workspace: refused on the host (their kernels
read the workspace's scalars)."""
import ctypes

from paper_2411_11229_gb300 import _capi as C


def test_adjoint_of_an_unbound_handle_is_refused():
    lib = C.load()
    h = ctypes.c_void_p()
    assert lib.hweno_create(2, C.HWENO_EULER, 40, 30, 0.05, 0.05, 1.4, C.HWENO_BC_PERIODIC, ctypes.byref(h)) == 0
    try:
        p = [ctypes.c_void_p(k << 20) for k in range(1, 8)]  # never dereferenced
        assert lib.hweno_stage_vjp(h, p[0], p[1], p[2], p[3], p[4], p[5]) == C.HWENO_ESTATE
        assert lib.hweno_adjoint_step_stages(h, p[0], p[1], p[2], 0.1, p[3], p[4], p[5], p[6]) == C.HWENO_ESTATE
        assert lib.hweno_adjoint_step(h, p[0], 0.1, p[1], p[2], p[3], p[4]) == C.HWENO_ESTATE
    finally:
        lib.hweno_destroy(h)
