"""The chained triangular solve at its branch edges: one, two and four
right-hand sides per task (chosen by n nrhs), orders at the edges of the
64-row blocks, a last task that is not full, a padded odd leading dimension,
both orientations; each against the substitution bound |B - op(L U) X| <=
c gamma_3n op(|L| |U|) |X| in the solve's precision (Higham, Thm. 8.5)."""
import numpy as np
import pytest
import torch

from paper_2312_09376_gb300 import _lib
from tests import _bounds, _df64

pytestmark = pytest.mark.gpu

U_DF64 = 2.0 ** -44


@pytest.mark.parametrize("prec,n,nrhs", [
    ("f64", 64, 5), ("f64", 65, 2), ("f64", 191, 33),
    ("df64", 63, 3), ("df64", 128, 2), ("df64", 65, 3079), ("df64", 192, 1043),
    ("f32", 64, 3), ("f32", 65, 925), ("f32", 192, 315), ("f32", 129, 1553), ("f32", 64, 3127)])
@pytest.mark.parametrize("trans", [False, True])
def test_solve_at_the_edges_of_blocks_and_groups(prec, n, nrhs, trans):
    rng = np.random.default_rng(n + nrhs)
    LU = 0.1 * rng.standard_normal((n, n))
    LU[np.arange(n), np.arange(n)] = 1.0 + np.abs(rng.standard_normal(n))
    pad = np.full((n + 3, n), np.nan)            # rows past the matrix are never read
    pad[:n] = LU
    if prec == "f32":
        pad = pad.astype(np.float32).astype(np.float64)
        LUd = _lib.to_device(pad).to(torch.float32)[:n]
        LU = pad[:n]
    elif prec == "df64":
        LUd, pad = _df64.to_df64(pad)
        LUd, LU = LUd[:n], pad[:n]
    else:
        LUd = _lib.to_device(pad)[:n]
    B = rng.standard_normal((n, nrhs))
    Bd = _lib.to_device(B)
    work = torch.empty(_lib.genp_solve_workspace(n, nrhs, prec), dtype=torch.uint8, device="cuda")
    _lib.genp_solve(n, prec, LUd, trans, Bd, work)
    torch.cuda.synchronize()
    assert int(work[:4].view(torch.int32).item()) == 0
    X = _lib.to_host(Bd)
    L, Uu = np.tril(LU, -1) + np.eye(n), np.triu(LU)
    M, absM = L @ Uu, np.abs(L) @ np.abs(Uu)
    if trans:
        M, absM = M.T, absM.T
    u = {"f64": _bounds.U64, "df64": U_DF64, "f32": _bounds.U32}[prec]
    assert np.all(np.abs(B - M @ X) <= 8 * _bounds.gamma(3 * n, u) * (absM @ np.abs(X)))
