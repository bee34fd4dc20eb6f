"""Explicit block sizes at the edges between the narrow and the 64-column panel
kernels, with a last step that is not full, against the bound of Gaussian
elimination |A - L U| <= gamma_n |L| |U| (Higham, Thm. 9.3) in the working
precision, evaluated here in double; the pairs' unit as in their other tests."""
import numpy as np
import pytest
import torch

from paper_2312_09376_gb300 import _lib, inputs
from tests import _bounds
from tests._df64 import from_df64, to_df64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,u", [("f64", 2.0 ** -53), ("f32", 2.0 ** -24), ("df64", 2.0 ** -44)])
@pytest.mark.parametrize("nb", [1, 15, 16, 17, 32, 33, 64, 65])
def test_factors_meet_the_bound(prec, u, nb):
    n = 203
    A = inputs.gaussian(n, seed=11)
    A[range(n), range(n)] += 2 * n ** 0.5
    if prec == "df64":
        LU, A = to_df64(A)
    else:
        LU = _lib.to_device(A).to(torch.float64 if prec == "f64" else torch.float32)
        A = _lib.to_host(LU).astype(np.float64)
    info = torch.empty(1, dtype=torch.int64, device="cuda")
    work = torch.empty(max(_lib.genp_factor_workspace(n, prec, nb), 1), dtype=torch.uint8, device="cuda")
    _lib.genp_factor(n, prec, LU, info, work, nb)
    torch.cuda.synchronize()
    assert int(info.item()) == -1
    F = from_df64(LU) if prec == "df64" else _lib.to_host(LU).astype(np.float64)
    L, U = np.tril(F, -1) + np.eye(n), np.triu(F)
    assert np.all(np.abs(A - L @ U) <= (_bounds.gamma(n, u) + _bounds.gamma(n, _bounds.U64)) * (np.abs(L) @ np.abs(U)))
