"""Sliced residuals of right-hand sides that have little in common: one column
of the solution holds an isolated entry 2^p, the others are N(0, 1).  A column's
residual must not depend on the other columns.

Evaluated in extended precision here, the returned X's backward error may
differ from the reported one by the sliced residual's own error.  That is one
rounding of R (2^-53 of |A| |X| + |B|) per piece of 448 rows, three at n = 1024,
and the digits: 2^-57 n max|A_ik| 2^-E_k max 2^E_k |X_kj| <= 2^-57 n max|A| ||x||,
for a Gaussian A (||A||_inf > n / 2, max|A| < 6) below 2^-53 ||A|| ||x||.  Twice
that sum: 8 2^-53."""
import numpy as np
import pytest
import torch

from paper_2312_09376_gb300 import _lib, inputs
from paper_2312_09376_gb300 import autograd as ag

pytestmark = pytest.mark.gpu

TOL, SLACK = 1e-15, 8 * 2.0 ** -53


def _berr(A, X, B):
    A, X, B = (M.astype(np.longdouble) for M in (A, X, B))
    R = np.abs(B - A @ X).max(axis=0)
    return (R / (np.abs(A).sum(axis=1).max() * np.abs(X).max(axis=0) + np.abs(B).max(axis=0))).astype(float)


def _solution(n, nrhs, p, seed):
    X = inputs.rhs(n, nrhs, seed=seed)
    X[5, 0] = 2.0 ** p
    return X


@pytest.mark.parametrize("prec", ["f64", "df64tc7"])
@pytest.mark.parametrize("p", [0, 40, 60, 200])
def test_an_isolated_entry_leaves_the_other_columns_alone(prec, p):
    n, nrhs = 1024, 16
    A = inputs.gaussian(n, seed=31)
    B = A @ _solution(n, nrhs, p, 32)
    opts = _lib.make_opts(2, 1, prec, 30, TOL, True)
    X = _lib.colmajor(n, nrhs)
    work = torch.empty(_lib.rbt_solve_workspace(opts, n, nrhs), dtype=torch.uint8, device="cuda")
    code, info = _lib.rbt_solve(opts, n, _lib.to_device(A), _lib.to_device(B), X, work)
    berr = _berr(A, _lib.to_host(X), B).max()
    assert code == _lib.RBT_OK
    assert abs(berr - info["berr"]) <= SLACK
    assert berr <= TOL + SLACK


@pytest.mark.parametrize("p", [0, 40, 60, 200])
def test_an_isolated_entry_leaves_the_other_columns_of_the_adjoint_alone(p):
    n, nrhs = 1024, 16
    A = inputs.gaussian(n, seed=33)
    G = A.T @ _solution(n, nrhs, p, 34)
    At = _lib.to_device(A).requires_grad_(True)
    Bt = _lib.to_device(inputs.rhs(n, nrhs, seed=35)).requires_grad_(True)
    Xt = ag.solve(At, Bt, depth=2, seed=1, prec="f64", tol=TOL)
    (gB,) = torch.autograd.grad(Xt, (Bt,), _lib.to_device(G))
    assert _berr(A.T, _lib.to_host(gB), G).max() <= TOL + SLACK
