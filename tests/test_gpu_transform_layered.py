"""The layer-by-layer transform is an FP64 computation at every order, also where
the fused one works in fixed point: each layer is a sum or difference and two
products in double, in the order of the kernel (rows, then columns, then the row
and the column factor, each with 1/sqrt(2)), so plain float64 arithmetic gives
the same bits."""
import math

import numpy as np
import pytest

from paper_2312_09376_gb300 import _lib

pytestmark = pytest.mark.gpu


def _layers(A, U, V, d):
    n, s2 = A.shape[0], math.sqrt(0.5)
    X = A.copy()
    for k in range(d, 0, -1):
        h = n >> k
        Y = X.reshape(-1, 2, h, n)
        X = np.concatenate((Y[:, :1] + Y[:, 1:], Y[:, :1] - Y[:, 1:]), axis=1).reshape(n, n)
        Y = X.reshape(n, -1, 2, h)
        X = np.concatenate((Y[:, :, :1] + Y[:, :, 1:], Y[:, :, :1] - Y[:, :, 1:]), axis=2).reshape(n, n)
        X = X * (U[:, k - 1] * s2)[:, None]
        X = X * (V[:, k - 1] * s2)[None, :]
    return X


@pytest.mark.parametrize("n", [512, 2048, 2056])
@pytest.mark.parametrize("d", [1, 2])
def test_layers_in_double(n, d):
    A = np.random.default_rng(n).standard_normal((n, n))
    U, V = _lib.colmajor(n, d), _lib.colmajor(n, d)
    _lib.rbt_generate(n, d, 3, U, V)
    lay = _lib.to_device(A)
    _lib.rbt_apply_2sided_layered(n, d, U, V, lay)
    want = _layers(A, _lib.to_host(U), _lib.to_host(V), d)
    assert np.array_equal(_lib.to_host(lay), want)
