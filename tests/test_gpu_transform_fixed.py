"""The double transform's 64-bit fixed-point groups and the groups that leave
them for the FP64 form: orders around multiples of 2^d (nu rows; from n = 2048, below it the FP64 form), rows scaled
far apart, entries near the ends of the exponent range, factors outside the
fixed-point range, zero groups, and entries that are not finite, against the
layer-by-layer transform of the same data.

Both forms' errors are relative to the largest entry of the 2^d x 2^d group an
entry belongs to, gm: partial sums stay below 16 gm / 4 times the factors' e^0.2
(below 5 gm), the layered form rounds at most six times a layer and side, the
fixed form by a few units of 2^-58 gm: 2^-47 gm covers both at d <= 2."""
import numpy as np
import pytest
import torch

from paper_2312_09376_gb300 import _lib

pytestmark = pytest.mark.gpu


def _both(A, d, scale=1.0):
    n = A.shape[0]
    U, V = _lib.colmajor(n, d), _lib.colmajor(n, d)
    _lib.rbt_generate(n, d, 3, U, V)
    U.mul_(scale)
    pad = np.full((n + 3, n), np.nan)            # rows past the matrix are never read
    pad[:n] = A
    Ad = _lib.to_device(pad)[:n]
    out, lay = _lib.colmajor(n, n, ld=n + 1), _lib.to_device(A)
    _lib.rbt_apply_2sided(n, d, U, V, Ad, out)
    _lib.rbt_apply_2sided_layered(n, d, U, V, lay)
    _lib.rbt_apply_2sided(n, d, U, V, Ad)        # in place
    torch.cuda.synchronize()
    assert torch.equal(Ad.nan_to_num(7.0), out.nan_to_num(7.0))
    return _lib.to_host(out), _lib.to_host(lay)


def _group_max(A, d):
    n, p = A.shape[0], 2 ** d
    h = -(-n // p)
    full = np.zeros((p * h, p * h))
    full[:n, :n] = np.abs(A)
    gm = full.reshape(p, h, p, h).max(axis=(0, 2))
    return np.tile(gm, (p, p))[:n, :n]


@pytest.mark.parametrize("n", [66, 2048, 2049, 2051])
@pytest.mark.parametrize("d", [1, 2])
@pytest.mark.parametrize("kind", ["plain", "spread", "tiny", "huge", "zeros", "factors"])
def test_fixed_point_groups_match_the_layered_transform(n, d, kind):
    rng = np.random.default_rng(n + d)
    A = rng.standard_normal((n, n))
    if kind == "spread":
        A = np.ldexp(A, rng.integers(-250, 250, (n, 1)))
    elif kind == "tiny":
        A *= 1e-290
    elif kind == "huge":
        A *= 1e299
    elif kind == "zeros":
        A[rng.random((n, n)) < 0.7] = 0.0
    out, lay = _both(A, d, 8.0 if kind == "factors" else 1.0)
    grow = 8.0 ** d if kind == "factors" else 1.0
    assert np.all(np.abs(out - lay) <= 2.0 ** -47 * grow * _group_max(A, d))


def test_entries_that_are_not_finite_reach_the_same_outputs():
    A = np.random.default_rng(1).standard_normal((2100, 2100))
    A[3, 5], A[70, 1500], A[1999, 0] = np.inf, np.nan, -np.inf
    out, lay = _both(A, 2)
    assert np.array_equal(np.isfinite(out), np.isfinite(lay))
    assert np.array_equal(np.isnan(out), np.isnan(lay))
