"""The fixed-point transform's rounding is not one-sided.  The mean of its error
over the entries of one of the 2^d x 2^d blocks (sum and difference parts) is
compared with the layered FP64 transform of the same data, whose rounding to
nearest has mean zero: the difference of the two is a mean of N errors of
standard deviation s (measured), zero within 6 s / sqrt(N).  (Off by 1.3 units
of 2^-57 of the group's largest binade, as truncation leaves it, the mean lies
more than ten times outside.)

Sampled groups are also compared with rational arithmetic: within 5 2^-53 |U|^T
|A| |V| (four factors times 1/sqrt(2), each rounded to a double, and the result's
rounding) plus 24 units: 16 inputs below a unit each, weighted 0.31, make 5; a
layer's two products, a unit each and one for the factor's 62 bits, make 3.5,
those of the first layer 2.2 times that in the sums of the second: 17 in all."""
import math
from fractions import Fraction

import numpy as np
import pytest
import torch

from paper_2312_09376_gb300 import _lib

pytestmark = pytest.mark.gpu


def _transform(n, d, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    A = torch.randn((n, n), generator=g, device="cuda", dtype=torch.float64).T
    U, V = _lib.colmajor(n, d), _lib.colmajor(n, d)
    _lib.rbt_generate(n, d, 3, U, V)
    out, lay = _lib.colmajor(n, n), A.T.clone().T
    _lib.rbt_apply_2sided(n, d, U, V, A, out)
    _lib.rbt_apply_2sided_layered(n, d, U, V, lay)
    return A, U, V, out, lay


@pytest.mark.parametrize("n", [2048, 4096])
@pytest.mark.parametrize("d", [1, 2])
def test_errors_have_mean_zero(n, d):
    _, _, _, out, lay = _transform(n, d, n + d)
    p = 2 ** d
    E = (out - lay).reshape(p, n // p, p, n // p)
    for s in range(p):
        for t in range(p):
            e = E[s, :, t, :]
            assert abs(float(e.mean())) <= 6 * float(e.std()) / math.sqrt(e.numel()), (s, t)


def test_sampled_groups_against_rational_arithmetic():
    n, d = 2048, 2
    p, h = 4, n // 4
    A, U, V, out, _ = (_lib.to_host(t) for t in _transform(n, d, 9))
    s2 = Fraction(math.sqrt(0.5))
    rng = np.random.default_rng(5)
    for r, c in rng.integers(0, h, (64, 2)):
        x = [[Fraction(float(A[r + s * h, c + t * h])) for t in range(p)] for s in range(p)]
        big = max(abs(v) for row in x for v in row)
        amp = sum(abs(v) for row in x for v in row)
        unit = Fraction(2) ** (math.frexp(float(big))[1] - 1 - 57)
        for l in range(d):
            st, k = 1 << l, d - 1 - l
            for s in range(p):
                if not s & st:
                    for t in range(p):
                        x[s][t], x[s | st][t] = x[s][t] + x[s | st][t], x[s][t] - x[s | st][t]
            for t in range(p):
                if not t & st:
                    for s in range(p):
                        x[s][t], x[s][t | st] = x[s][t] + x[s][t | st], x[s][t] - x[s][t | st]
            for s in range(p):
                for t in range(p):
                    fu, fv = (Fraction(float(W[i + q * h, k])) * s2 for W, i, q in ((U, r, s), (V, c, t)))
                    x[s][t] *= fu * fv
            amp *= Fraction(math.exp(0.1)) / 2   # factors at most e^0.05 a side and layer, 1/2 a layer
        for s in range(p):
            for t in range(p):
                bound = 5 * Fraction(2) ** -53 * amp + 24 * unit
                assert abs(Fraction(float(out[r + s * h, c + t * h])) - x[s][t]) <= bound
