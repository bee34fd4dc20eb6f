"""A launch is timed in one class: the products of a sliced residual belong to the
residual, so a solve with many right-hand sides counts as many updates and slicings
as one with a single one."""
import pytest
import torch

from paper_2312_09376_gb300 import _lib, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["f64", "df64tc7"])
def test_sliced_residuals_are_not_counted_as_updates(prec):
    n, counts = 800, []
    A = _lib.to_device(inputs.gaussian(n, seed=3))
    for nrhs in (1, 16):
        B, X = _lib.to_device(inputs.rhs(n, nrhs, seed=4)), _lib.colmajor(n, nrhs)
        opts = _lib.make_opts(2, 1, prec, 30, 1e-14, False)
        work = torch.empty(_lib.rbt_solve_workspace(opts, n, nrhs), dtype=torch.uint8, device="cuda")
        _lib.rbt_prof_reset()
        _lib.rbt_prof_enable(True)
        try:
            _, info = _lib.rbt_solve(opts, n, A, B, X, work)
        finally:
            _lib.rbt_prof_enable(False)
        counts.append([_lib.rbt_prof_read(c)[1] for c in ("update", "slice")])
        # one for ||A||, one residual a step
        assert _lib.rbt_prof_read("residual")[1] == info["iters"] + 2
    assert counts[0] == counts[1] and counts[0][0] > 0
