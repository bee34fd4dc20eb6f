"""The double factorization's sliced tensor-core updates (RBT_F64 in rbt_solve
from n = 1024): panel edges, rows and columns scaled by powers of two far
apart, a sparse matrix (which stays on the FP64 pipe), and entries that are
not finite, against the bound of Gaussian elimination in double arithmetic
|A - L U| <= gamma_n |L| |U| (Higham, Thm. 9.3) and against the FP64-pipe
factorization of the same matrix (an explicit block size).  Depth 0: the
factors of A itself, read from the front of the workspace (columns of n
rounded up to 32 rows)."""
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
    return work[:8 * ldt * n].view(torch.float64).reshape(n, ldt)[:, :n].T, info["zero_pivot"]


def _matrix(n, kind):
    rng = np.random.default_rng(n)
    A = rng.standard_normal((n, n))
    if kind == "scaled":
        A = A + 2 * np.sqrt(n) * np.eye(n)
        e = rng.integers(-200, 200, n)
        A = np.ldexp(np.ldexp(A, e[:, None]), -e[::-1][None, :])
        A[np.arange(n), np.arange(n)] *= 4
    elif kind == "sparse":
        A *= rng.random((n, n)) < 0.02
        A[np.arange(n), np.arange(n)] += 40.0
    else:
        A += 2 * np.sqrt(n) * np.eye(n)
    return A


@pytest.mark.parametrize("n,kind", [(1024, "plain"), (1087, "plain"), (1344, "plain"), (1345, "plain"),
                                    (1857, "plain"), (1100, "scaled"), (1100, "sparse")])
def test_sliced_double_factors_meet_the_double_bound(n, kind):
    A = _matrix(n, kind)
    F, info = _factor(A, 0)
    assert info == -1
    G, _ = _factor(A, 64)
    assert torch.equal(F, G) == (kind == "sparse")   # other roundings where the sliced updates ran
    Ad = torch.from_numpy(A).cuda()
    errs = []
    for T in (F, G):
        L = torch.tril(T, -1) + torch.eye(n, dtype=torch.float64, device="cuda")
        U = torch.triu(T)
        R, S = (Ad - L @ U).abs(), L.abs() @ U.abs()
        # L @ U here is itself a double product of n terms: twice the bound
        assert bool((R <= 2 * _bounds.gamma(n, _bounds.U64) * S).all())
        errs.append(float(((R / S.clamp(min=1e-300)).square().mean()).sqrt()))
    assert errs[0] <= 1.5 * errs[1]              # and no less accurate than the FP64 pipe


@pytest.mark.parametrize("val", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("at", [(700, 300), (300, 700), (1000, 1000)])
def test_entries_that_are_not_finite_stop_at_the_same_pivot(val, at):
    A = _matrix(1100, "plain")
    A[at] = val
    _, a = _factor(A, 0)
    _, b = _factor(A, 64)
    assert a == b and a >= 0
