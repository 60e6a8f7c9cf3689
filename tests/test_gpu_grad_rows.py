"""Value gradients where the loads of a row change width: every number of
columns from one to nine and the multiples above, contiguous, padded and
shifted blocks, rows of no to many entries and a last partial chunk of rows,
single and batched, against FP64 sums.  Tolerance: k + 1 roundings of the sum
of magnitudes, element by element."""
import numpy as np
import pytest
import torch

import synthetic as S

pytestmark = pytest.mark.gpu


def _check(gv, A_h, gb, x, dt):
    rows = np.repeat(np.arange(A_h.n), np.diff(A_h.row_ptr))
    a, b = gb.astype(np.float64)[rows], x.astype(np.float64)[A_h.col_idx]
    bound = (gb.shape[1] + 1) * np.finfo(dt).eps * np.abs(a * b).sum(1)
    assert np.all(np.abs(gv + (a * b).sum(1)) <= bound)


@pytest.mark.parametrize("dt", [np.float64, np.float32], ids=["f64", "f32"])
@pytest.mark.parametrize("k", [1, 2, 3, 4, 5, 6, 7, 8, 9, 12, 16])
def test_grad_rows(k, dt):
    import paper_2609_40159_gb300 as P
    for A_h in (S.diagonal(1, seed=1).astype(dt), S.band_random(33, 32, 0, 8, seed=2).astype(dt),
                S.band_random(1999, 500, 0, 40, seed=3).astype(dt)):
        plan = P.Plan(P.Matrix.from_host(A_h), transpose=True)
        gb, x = S.rhs(A_h.n, k, seed=4, dtype=dt), S.rhs(A_h.n, k, seed=5, dtype=dt)
        for pad, shift in ((0, 0), (1, 0), (3, 1), (4, 2), (4, 0)):
            def put(v):
                room = torch.zeros(A_h.n * (k + pad) + shift, dtype=torch.as_tensor(v).dtype, device="cuda")
                t = room[shift:].view(A_h.n, k + pad)[:, :k]
                t.copy_(torch.as_tensor(v))
                return t
            _check(plan.grad_vals(put(gb), put(x)).cpu().numpy(), A_h, gb, x, dt)


@pytest.mark.parametrize("dt", [np.float64, np.float32], ids=["f64", "f32"])
def test_grad_rows_batch(dt):
    import paper_2609_40159_gb300 as P
    hosts = [S.band_random(30 + 37 * m, 64, 0, 12, seed=m).astype(dt) for m in range(9)]
    ks = [4, 3, 8, 2, 16, 1, 6, 12, 5]
    plan = P.BatchPlan([P.Matrix.from_host(A) for A in hosts], nrhs=ks, transpose=True)
    gb = [S.rhs(A.n, k, seed=4, dtype=dt) for A, k in zip(hosts, ks)]
    x = [S.rhs(A.n, k, seed=5, dtype=dt) for A, k in zip(hosts, ks)]
    pack = lambda vs: torch.as_tensor(np.concatenate([v.reshape(-1) for v in vs])).cuda()
    gv = plan.grad_vals(pack(gb), pack(x)).cpu().numpy()
    for m, A in enumerate(hosts):
        _check(gv[plan.vals_offset[m]:plan.vals_offset[m + 1]], A, gb[m], x[m], dt)


@pytest.mark.parametrize("dt", [np.float64, np.float32], ids=["f64", "f32"])
@pytest.mark.parametrize("n", [3, 5, 38_912, 38_913, 77_824, 77_829])
def test_grad_rows_of_a_warp(n, dt):
    """On both sides of the sizes where a warp takes more rows."""
    import paper_2609_40159_gb300 as P
    A_h = S.band_random(n, 300, 0, 9, seed=n).astype(dt)
    plan = P.Plan(P.Matrix.from_host(A_h), mode="syncfree")
    for k in (1, 3, 4):
        gb, x = S.rhs(n, k, seed=4, dtype=dt), S.rhs(n, k, seed=5, dtype=dt)
        gv = plan.grad_vals(torch.as_tensor(gb).cuda(), torch.as_tensor(x).cuda())
        _check(gv.cpu().numpy(), A_h, gb, x, dt)
