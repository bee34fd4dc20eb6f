"""Solves and adjoints with many right-hand sides, whose residuals go through
the nine-digit sliced products (rbt_solve from 16 columns and n = 768 on,
A's entries of like size): sizes off the 448-row pieces and the 48-column
tiles.  The reported backward error must be that of the returned X, and small:
the sliced residual carries 62 bits of |A| |X|, so the two evaluations differ
by the double rounding of this one, gamma_{n+1} of (|A| |X| + |B|)_ij over
||A|| ||x|| + ||b||, at most about (n + 1) 2^-53."""
import numpy as np
import pytest
import torch

from paper_2312_09376_gb300 import _lib, inputs
from paper_2312_09376_gb300 import autograd as ag
from tests import _bounds

pytestmark = pytest.mark.gpu


def _berr(A, X, B):
    R = np.abs(B - A @ X).max(axis=0)
    return float((R / (np.abs(A).sum(axis=1).max() * np.abs(X).max(axis=0) + np.abs(B).max(axis=0))).max())


@pytest.mark.parametrize("n,nrhs", [(800, 16), (1345, 49)])
@pytest.mark.parametrize("prec", ["f64", "df64tc7", "f32"])
@pytest.mark.parametrize("sparse", [False, True])
def test_reported_backward_errors_with_many_right_hand_sides(n, nrhs, prec, sparse):
    A = inputs.gaussian(n, seed=21)
    if sparse:                                   # stays on the FP64 residual
        A *= np.random.default_rng(2).random((n, n)) < 0.1
        A[np.arange(n), np.arange(n)] += 4.0
    B, W = inputs.rhs(n, nrhs, seed=22), inputs.rhs(n, nrhs, seed=23)
    opts = _lib.make_opts(2, 1, prec, 30, 1e-14, True)
    X = _lib.colmajor(n, nrhs)
    work = torch.empty(_lib.rbt_solve_workspace(opts, n, nrhs), dtype=torch.uint8, device="cuda")
    code, info = _lib.rbt_solve(opts, n, _lib.to_device(A), _lib.to_device(B), X, work)
    slack = _bounds.gamma(n + 1, _bounds.U64)
    assert code == _lib.RBT_OK
    assert abs(_berr(A, _lib.to_host(X), B) - info["berr"]) <= slack
    At = _lib.to_device(A).requires_grad_(True)
    Bt = _lib.to_device(B).requires_grad_(True)
    Xt = ag.solve(At, Bt, depth=2, seed=1, prec=prec, tol=1e-14)
    gA, gB = torch.autograd.grad(Xt, (At, Bt), _lib.to_device(W))
    assert _berr(A.T, _lib.to_host(gB), W) <= 1e-14 + slack
    assert torch.allclose(gA, -gB @ Xt.detach().T, rtol=1e-13, atol=1e-13 * float(gA.abs().max()))
