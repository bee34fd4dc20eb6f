"""The batched float solver takes right-hand sides by eights from order 384 on and
one by one otherwise, with the same sums: unrefined, a column's solution does not
depend, bit for bit, on how many others it is solved with."""
import pytest
import torch

from paper_2312_09376_gb300 import _lib, inputs

pytestmark = pytest.mark.gpu


def _solve(As, Bs):
    Xs = [_lib.colmajor(*b.shape) for b in Bs]
    opts = _lib.make_opts(2, 1, "f32", 0, 1e-13, False)
    plan = _lib.rbt_solve_batched_plan(opts, As, Bs, Xs, seeds=[5] * len(As))
    _lib.rbt_solve_batched_run(plan)
    torch.cuda.synchronize()
    return Xs


@pytest.mark.parametrize("n", [383, 384, 401])
def test_columns_do_not_depend_on_their_number(n):
    A = _lib.to_device(inputs.gaussian(n, seed=7))
    B = _lib.to_device(inputs.rhs(n, 17, seed=8))
    alone = torch.cat(_solve([A] * 17, [B[:, c:c + 1] for c in range(17)]), dim=1)
    assert bool(torch.isfinite(alone).all())
    for k, X in zip((7, 8, 9, 16, 17), _solve([A] * 5, [B[:, :k] for k in (7, 8, 9, 16, 17)])):
        assert torch.equal(X, alone[:, :k]), k
