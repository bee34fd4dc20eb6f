"""A sliced residual that gives up waiting ends the adjoint there: its result is
not used for another correction.  Counted in launches: no more than those of an
adjoint that stops after its first residual (the stalled products are launched as
usual and return by themselves after the wait limit)."""
import ctypes

import pytest
import torch

from paper_2312_09376_gb300 import _lib, inputs

pytestmark = pytest.mark.gpu


def test_adjoint_stops_at_the_residual_that_timed_out():
    n, nrhs = 800, 16
    A, B = _lib.to_device(inputs.gaussian(n, seed=3)), _lib.to_device(inputs.rhs(n, nrhs, seed=4))
    X, Y = _lib.colmajor(n, nrhs), _lib.colmajor(n, nrhs)
    opts = _lib.make_opts(2, 1, "f64", 30, 1e-15, True)
    work = torch.empty(_lib.rbt_solve_workspace(opts, n, nrhs), dtype=torch.uint8, device="cuda")
    lib = _lib.load()
    fwd, adj = _lib.rbt_info(), _lib.rbt_info()
    p = lambda t: ctypes.c_void_p(t.data_ptr())
    s = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    assert lib.rbt_solve(ctypes.byref(opts), n, nrhs, p(A), n, p(B), n, p(X), n, p(work), work.numel(),
                         ctypes.byref(fwd), s) == 0

    def adjoint(refine_max):
        o = _lib.make_opts(2, 1, "f64", refine_max, 1e-15, True)
        before = _lib.rbt_kernel_launches()
        code = lib.rbt_solve_adjoint(ctypes.byref(o), ctypes.byref(fwd), n, nrhs, p(A), n, p(B), n, p(Y), n, p(work),
                                     work.numel(), ctypes.byref(adj), s)
        return code, _lib.rbt_kernel_launches() - before

    _, once = adjoint(0)
    code, whole = adjoint(30)
    assert code == _lib.RBT_OK and whole > once
    _lib.rbt_debug_wait_limit(2_000_000)
    _lib.rbt_debug_stall("oz_copy")
    try:
        code, stalled = adjoint(30)
    finally:
        _lib.rbt_debug_stall("none")
        _lib.rbt_debug_wait_limit(0)
    assert code == -4 and stalled <= once        # RBT_ERR_TIMEOUT
    code, again = adjoint(30)
    assert code == _lib.RBT_OK and again == whole
