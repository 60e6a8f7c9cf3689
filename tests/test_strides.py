"""Right-hand sides and outputs of different leading dimensions: the library
takes one for both, so the binding hands it a block of the output's.  Padded
and sliced right-hand sides without an output, padded outputs, every
single-system call, against the calls on contiguous blocks."""
import numpy as np
import pytest
import torch

import synthetic as S


def test_right_hand_side_takes_the_outputs_leading_dimension():
    from paper_2609_40159_gb300.api import Plan
    wide, x = torch.arange(30.0).view(5, 6), torch.zeros(5, 3)
    b = wide[:, 1:4]
    y, ld = Plan._like(b, x)
    assert y.stride(0) == ld == 3 and torch.equal(y, b)
    assert Plan._like(b, wide[:, :3])[0] is b and Plan._like(x, x)[0] is x
    y, ld = Plan._like(x, wide[:, 2:5])
    assert y.stride() == (6, 1) and ld == 6 and y.shape == x.shape
    one = wide[:1, :3]
    assert Plan._like(one, x[:1])[0] is one
    with pytest.raises(ValueError):
        Plan._like(b, x[:, :2])
    with pytest.raises(ValueError):
        Plan._like(b, torch.zeros(1, 3).expand(5, 3))


@pytest.mark.gpu
@pytest.mark.parametrize("mode", ["level_launch", "level", "syncfree", "block", "hybrid"])
def test_padded_blocks(mode):
    import paper_2609_40159_gb300 as P
    A_h = S.lap2d(40)
    n, k = A_h.n, 3
    plan = P.Plan(P.Matrix.from_host(A_h), mode=mode, transpose=True)
    wide = torch.as_tensor(np.ascontiguousarray(S.rhs(n, k + 4, seed=1))).cuda()
    b = wide[:, 1:1 + k]
    other = torch.as_tensor(S.rhs(n, k, seed=2)).cuda()
    calls = [lambda v, out: plan.solve(v, out=out), lambda v, out: plan.solve_transpose(v, out=out),
             lambda v, out: plan.tt_apply(v, out=out)]
    for call in calls:
        want = call(b.contiguous(), None)
        assert torch.equal(call(b, None), want)
        room = torch.full((n, k + 2), 7.0, dtype=wide.dtype, device="cuda")
        call(b, room[:, 2:])
        assert torch.equal(room[:, 2:], want) and bool((room[:, :2] == 7.0).all())
        room = torch.full((n, k), 7.0, dtype=wide.dtype, device="cuda")
        call(b, room)
        assert torch.equal(room, want)
    want = plan.grad_vals(b.contiguous(), other)
    assert torch.equal(plan.grad_vals(b, other), want)
    assert torch.equal(plan.grad_vals(b.contiguous(), wide[:, 2:2 + k]), plan.grad_vals(b, wide[:, 2:2 + k]))
    assert P.handle().status() == 0
