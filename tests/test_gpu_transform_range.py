"""Columns of one large value among N(0, 1) entries: the row butterflies cancel it
exactly, and the rows where they do keep their small entries to rounding, however
large the value.  Against the layer-by-layer FP64 transform, entrywise relative to
what is left: with the column taken out of A the same rows come out of the same
sums, so |U|^T |A'| |V| (A' without the column) scales the error; each form rounds
at most seven times a layer, the products of two sides in a layer three: 32 2^-53
of it covers both at d <= 2."""
import numpy as np
import pytest

from paper_2312_09376_gb300 import _lib
from tests import _bounds

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2048, 2052])
@pytest.mark.parametrize("d", [1, 2])
@pytest.mark.parametrize("p", [18, 40, 60, 200])
def test_a_cancelling_column_leaves_the_small_entries(n, d, p):
    A = np.random.default_rng(n + p).standard_normal((n, n))
    A[:, 77] = 0.0
    small = A.copy()
    A[:, 77] = 2.0 ** p
    U, V = _lib.colmajor(n, d), _lib.colmajor(n, d)
    _lib.rbt_generate(n, d, 3, U, V)
    out, lay = _lib.colmajor(n, n), _lib.to_device(A)
    _lib.rbt_apply_2sided(n, d, U, V, _lib.to_device(A), out)
    _lib.rbt_apply_2sided_layered(n, d, U, V, lay)
    out, lay = _lib.to_host(out), _lib.to_host(lay)
    bound = 32 * 2.0 ** -53 * _bounds.group_bound(small, d)
    h = n // 2 ** d
    rows = np.arange(n) // h % 2 == 1            # differences of the first layer's pairs
    # at p = 18 the group stays in fixed point: a few units of 2^-57 of the column's value
    slack = 24 * 2.0 ** (p - 57) if p <= 20 else 0.0
    assert np.all(np.abs(out - lay)[rows] <= bound[rows] + slack)
