"""Matrices that the sliced double factorization must leave to the FP64 pipe:
one entry far above all others, and entries that alternate between two sizes
(i + j even or odd), where a row of L and a column of U have no large factor in
common; and matrices that it may take, however their rows and columns are
scaled.  Depth 0: the factors of A itself, against the bound of Gaussian
elimination in double arithmetic |A - L U| <= gamma_n |L| |U| (Higham, Thm.
9.3), evaluated here with an error of the same size.  The route shows in the
factors: those of the FP64 pipe are the ones of an explicit block size, bit for
bit."""
import numpy as np
import pytest
import torch

from paper_2312_09376_gb300 import _lib
from tests import _bounds

pytestmark = pytest.mark.gpu


def _factor(A, nb):
    n = A.shape[0]
    ldt = (n + 31) // 32 * 32
    opts = _lib.make_opts(0, 1, "f64", 0, 1e-13, False, nb=nb)
    work = torch.empty(_lib.rbt_solve_workspace(opts, n, 1), dtype=torch.uint8, device="cuda")
    B = torch.ones(n, dtype=torch.float64, device="cuda")
    _, info = _lib.rbt_solve(opts, n, _lib.to_device(A), B, torch.empty_like(B), work)
    assert info["zero_pivot"] == -1
    return work[:8 * ldt * n].view(torch.float64).reshape(n, ldt)[:, :n].T


def _matrix(n, kind, p):
    rng = np.random.default_rng(n + p)
    if kind == "alternating":                    # no entry below 1 before: exactly half become small
        A = rng.choice([-1.0, 1.0], (n, n)) * rng.uniform(1, 2, (n, n))
        i, j = np.indices((n, n))
        A[(i + j) % 2 == 1] *= 2.0 ** -p
    else:
        A = rng.standard_normal((n, n))
    A += 2 * np.sqrt(n) * np.eye(n)
    if kind == "one":
        A[5, n - 100] = 2.0 ** p
    elif kind == "column":                       # a scaling, not an outlier
        A[:, n - 100] *= 2.0 ** p
    elif kind == "zeros":
        A *= rng.random((n, n)) >= 0.1
        A[np.arange(n), np.arange(n)] = 2 * np.sqrt(n)
    return A


@pytest.mark.parametrize("n,kind,p,sliced", [
    (767, "plain", 0, False), (768, "plain", 0, True), (800, "plain", 0, True), (1000, "one", 60, False),
    (1000, "one", 100, False), (1000, "one", 300, False), (1000, "column", 100, True), (1000, "zeros", 0, True),
    (1000, "alternating", 30, False), (1000, "alternating", 14, False), (1000, "alternating", 8, True)])
def test_route_and_bound(n, kind, p, sliced):
    A = _matrix(n, kind, p)
    F, G = _factor(A, 0), _factor(A, 64)
    Ad = torch.from_numpy(A).cuda()
    errs = []
    for T in (F, G):
        L = torch.tril(T, -1) + torch.eye(n, dtype=torch.float64, device="cuda")
        U = torch.triu(T)
        R, S = (Ad - L @ U).abs(), L.abs() @ U.abs()
        assert bool((R <= 2 * _bounds.gamma(n, _bounds.U64) * S).all())
        errs.append(float(((R / S.clamp(min=1e-300)).square().mean()).sqrt()))
    assert errs[0] <= 1.5 * errs[1]
    assert torch.equal(F, G) != sliced
