"""Workspaces that start on an element's boundary only, not on a vector load's:
the same bits as with an aligned one.  (Orders and columns of one, two and four
right-hand sides a task; a double solve with sliced updates and residuals.)"""
import ctypes

import pytest
import torch

from paper_2312_09376_gb300 import _lib, inputs
from tests._df64 import to_df64

pytestmark = pytest.mark.gpu


def _buffer(nbytes, shift):
    return torch.empty(nbytes + shift, dtype=torch.uint8, device="cuda")[shift:]


@pytest.mark.parametrize("prec,shift", [("f64", 8), ("df64", 8), ("f32", 4), ("f32", 12)])
@pytest.mark.parametrize("n,nrhs", [(65, 1), (130, 3), (65, 3500)])
@pytest.mark.parametrize("trans", [0, 1])
def test_triangular_solve(prec, shift, n, nrhs, trans):
    A = inputs.gaussian(n, seed=1)
    A[range(n), range(n)] += 3 * n ** 0.5
    LU = to_df64(A)[0] if prec == "df64" else _lib.to_device(A)
    LU = LU.to(torch.float32) if prec == "f32" else LU
    B = _lib.to_device(inputs.rhs(n, nrhs, seed=2))
    out = []
    for k in (0, shift):
        X = B.clone()
        _lib.genp_solve(n, prec, LU, trans, X, _buffer(_lib.genp_solve_workspace(n, nrhs, prec), k))
        out.append(X)
    assert torch.equal(*out) and bool(torch.isfinite(out[0]).all())


@pytest.mark.parametrize("prec", ["f32", "df64"])
def test_triangular_solve_in_double(prec):
    n, nrhs = 130, 3
    A = inputs.gaussian(n, seed=1)
    A[range(n), range(n)] += 3 * n ** 0.5
    LU = to_df64(A)[0] if prec == "df64" else _lib.to_device(A).to(torch.float32)
    B = _lib.to_device(inputs.rhs(n, nrhs, seed=2))
    out = []
    for k in (0, 8):
        X = B.clone()
        _lib.genp_solve_wp(n, prec, LU, 0, X, _buffer(_lib.genp_solve_wp_workspace(n, nrhs), k))
        out.append(X)
    assert torch.equal(*out) and bool(torch.isfinite(out[0]).all())


@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("n,nrhs", [(500, 1), (800, 17)])
def test_solve_and_adjoint(prec, n, nrhs):
    A, B = _lib.to_device(inputs.gaussian(n, seed=3)), _lib.to_device(inputs.rhs(n, nrhs, seed=4))
    G = _lib.to_device(inputs.rhs(n, nrhs, seed=5))
    opts = _lib.make_opts(2, 1, prec, 30, 1e-14, True)
    lib = _lib.load()
    out = []
    for k in (0, 8):
        work = _buffer(_lib.rbt_solve_workspace(opts, n, nrhs), k)
        X, Y = _lib.colmajor(n, nrhs), _lib.colmajor(n, nrhs)
        fwd, adj = _lib.rbt_info(), _lib.rbt_info()
        p = lambda t: ctypes.c_void_p(t.data_ptr())
        s = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
        assert lib.rbt_solve(ctypes.byref(opts), n, nrhs, p(A), n, p(B), n, p(X), n, p(work), work.numel(),
                             ctypes.byref(fwd), s) == 0
        assert lib.rbt_solve_adjoint(ctypes.byref(opts), ctypes.byref(fwd), n, nrhs, p(A), n, p(G), n, p(Y), n,
                                     p(work), work.numel(), ctypes.byref(adj), s) == 0
        out.append((X, Y))
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
