"""Solves over strips with x in b's place, a right-hand side of which is not
finite: the second pass over the system must read the right-hand side, not the
solution that has taken its place.  The same bits as with buffers apart; a
solution in other columns of b's rows; the same call under capture."""
import numpy as np
import pytest
import torch

import synthetic as S

pytestmark = pytest.mark.gpu


def _same(x, y):
    # (a NaN's bits are not fixed)
    return torch.equal(torch.nan_to_num(x, nan=1.25e30), torch.nan_to_num(y, nan=1.25e30))


def _bad_rhs(n, k, value, dt):
    b = S.rhs(n, k, seed=1, dtype=dt)
    b[n // 3, k - 1] = value
    b[n - 2, 0] = value
    return torch.as_tensor(b).cuda()


@pytest.mark.parametrize("value", [1.0, np.inf, np.nan])
@pytest.mark.parametrize("dt", [np.float64, np.float32], ids=["f64", "f32"])
def test_block_in_place(dt, value):
    import paper_2609_40159_gb300 as P
    A_h = S.band_random(3001, 200, 0, 3, seed=7).astype(dt)
    plan = P.Plan(P.Matrix.from_host(A_h), mode="block", rows_per_warp=32, transpose=True)
    for k in (1, 3, 310):
        b = _bad_rhs(A_h.n, k, value, dt)
        for run in (plan.solve, plan.solve_transpose):
            want = run(b)
            y = b.clone()
            run(y, out=y)
            assert _same(y, want), k
            pad = torch.zeros(A_h.n, 2 * k + 1, dtype=b.dtype, device="cuda")
            pad[:, :k] = b
            run(pad[:, :k], out=pad[:, k:2 * k])  # beside b
            assert _same(pad[:, k:2 * k], want) and _same(pad[:, :k], b), k
            run(pad[:, :k], out=pad[:, :k])
            assert _same(pad[:, :k], want), k
    assert P.handle().status() == 0


@pytest.mark.parametrize("value", [np.inf, np.nan])
@pytest.mark.parametrize("dt", [np.float64, np.float32], ids=["f64", "f32"])
def test_batch_in_place(dt, value):
    import paper_2609_40159_gb300 as P
    hosts = [S.band_random(n, 60, 0, 3, seed=n).astype(dt) for n in (33, 700, 2100)]
    ks = [2, 5, 4]
    plan = P.BatchPlan([P.Matrix.from_host(A) for A in hosts], nrhs=ks, transpose=True)
    b = torch.cat([_bad_rhs(A.n, k, value, dt).reshape(-1) for A, k in zip(hosts, ks)])
    for run in (plan.solve, plan.solve_transpose):
        want = run(b)
        y = b.clone()
        run(y, out=y)
        assert _same(y, want)
    assert P.handle().status() == 0


def test_in_place_under_capture():
    import paper_2609_40159_gb300 as P
    A_h = S.band_random(2001, 60, 0, 3, seed=5)
    b = _bad_rhs(A_h.n, 2, np.inf, np.float64)
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        plan = P.Plan(P.Matrix.from_host(A_h), mode="block", rows_per_warp=32)
        want = plan.solve(b)
        y = torch.empty_like(b)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            plan.solve(y, out=y)
        for _ in range(2):
            y.copy_(b)
            g.replay()
            s.synchronize()
            assert _same(y, want)
        assert P.handle().status() == 0
    torch.cuda.synchronize()
