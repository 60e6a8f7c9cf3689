"""The level-ordered solve with one lane per row and column (level mode with 32
rows per warp) against the CPU oracle where its shape changes: rows of no to
many entries on both sides of the mean that picks how many are held, levels
ending inside a block's rows, one to more columns than a block takes, padded
leading dimensions, right-hand sides that hold infinities, NaN and the pattern
that marks an unsolved element, in-place solves, rewritten systems, and a row
that never comes.  Tolerances: the normwise ones of the other solve tests."""
import numpy as np
import pytest
import torch

import oracle
import synthetic as S
from helpers import TOL, relerr, two_wide_levels, wide_level, widened

pytestmark = pytest.mark.gpu

CASES = {
    "one_row": lambda: S.diagonal(1, seed=1),
    "diagonal": lambda: S.diagonal(1000, seed=2),
    "chain": lambda: S.chain(300, seed=3),
    "wide_level": lambda: wide_level(5001),
    "two_wide_levels": lambda: two_wide_levels(4001, seed=4),
    "lap3d": lambda: S.lap3d(21),
    "windows": lambda: S.band_random(6001, 2000, 0, 20, seed=5),  # up to five windows of four entries
    "few": lambda: S.band_random(5003, 1500, 0, 8, seed=6),
}


@pytest.mark.parametrize("dt", [np.float64, np.float32], ids=["f64", "f32"])
@pytest.mark.parametrize("name", list(CASES))
def test_level_cols_vs_oracle(name, dt):
    import paper_2609_40159_gb300 as P
    A_h = CASES[name]().astype(dt)
    W_h = widened(A_h)
    plan = P.Plan(P.Matrix.from_host(A_h), mode="level", rows_per_warp=32, transpose=True)
    for k in (1, 2, 3, 8, 20):
        b_h = S.rhs(A_h.n, k, seed=k, dtype=dt)
        pad = torch.zeros(A_h.n, k + 3, dtype=torch.as_tensor(b_h).dtype, device="cuda")
        pad[:, :k] = torch.as_tensor(b_h).cuda()
        for b in (pad[:, :k], pad[:, :k].contiguous()):
            for run, ref in ((plan.solve, oracle.solve), (plan.solve_transpose, oracle.solve_transpose)):
                x = torch.empty_strided(b.shape, b.stride(), dtype=b.dtype, device="cuda")
                run(b, out=x)
                assert relerr(x.cpu().numpy(), ref(W_h, b_h)) <= TOL[dt], k
    assert torch.equal(pad[:, k:], torch.zeros_like(pad[:, k:]))
    assert P.handle().status() == 0


@pytest.mark.parametrize("dt", [np.float64, np.float32], ids=["f64", "f32"])
def test_level_cols_not_finite(dt):
    import paper_2609_40159_gb300 as P
    A_h = S.band_random(3001, 1500, 0, 3, seed=7).astype(dt)
    plan = P.Plan(P.Matrix.from_host(A_h), mode="level", rows_per_warp=32, transpose=True)
    mark = {np.float64: np.uint64(0x7FF85A5AA5A53C3C), np.float32: np.uint32(0x7FC5A3C7)}[dt].view(dt)
    for v in (np.inf, np.nan, mark):
        b_h = S.rhs(A_h.n, 2, seed=1, dtype=dt)
        b_h[40, 1] = v
        for run, ref in ((plan.solve, oracle.solve), (plan.solve_transpose, oracle.solve_transpose)):
            with np.errstate(all="ignore"):
                want = ref(widened(A_h), b_h)
            x = run(torch.as_tensor(b_h).cuda()).cpu().numpy()
            fin = np.isfinite(want)
            assert np.array_equal(np.isfinite(x), fin)
            assert relerr(x[fin], want[fin]) <= TOL[dt]
    assert P.handle().status() == 0


def test_level_cols_in_place_rewritten_and_new_values():
    import paper_2609_40159_gb300 as P
    A_h = S.lap3d(24)
    an = oracle.analyze(A_h)
    rows, tg = S.narrowest_levels_list(an["nlevels"], an["level_ptr"], an["perm"], 0.05, 8)
    A = P.Matrix.from_host(A_h)
    Lp, T = P.rewrite(A, P.analyze(A).lev, rows, tg)
    b_h = S.rhs(A_h.n, 3, seed=1)
    b = torch.as_tensor(b_h).cuda()
    x = P.Plan(Lp, T, mode="level", rows_per_warp=32).solve(b)
    assert relerr(x.cpu().numpy(), oracle.solve(A_h, b_h)) <= 1e-12
    plan = P.Plan(A, mode="level", rows_per_warp=32, transpose=True)
    for run, ref in ((plan.solve, oracle.solve), (plan.solve_transpose, oracle.solve_transpose)):
        y = b.clone()
        run(y, out=y)
        assert relerr(y.cpu().numpy(), ref(A_h, b_h)) <= 1e-12
    A.vals.mul_(2.0)  # values may change between solves
    assert relerr(2.0 * plan.solve(b).cpu().numpy(), oracle.solve(A_h, b_h)) <= 1e-12
    assert relerr(2.0 * plan.solve_transpose(b).cpu().numpy(), oracle.solve_transpose(A_h, b_h)) <= 1e-12
    assert P.handle().status() == 0


@pytest.mark.parametrize("trans", [False, True], ids=["fwd", "transpose"])
def test_level_cols_bounded_wait(trans):
    import paper_2609_40159_gb300 as P
    A_h = S.lap3d(30)
    b_h = S.rhs(A_h.n, 2, seed=2)
    b = torch.as_tensor(b_h).cuda()
    plan = P.Plan(P.Matrix.from_host(A_h), mode="level", rows_per_warp=32, transpose=True, wait_limit_us=20_000)
    h = P.handle()
    run = plan.solve_transpose if trans else plan.solve
    plan.withhold(A_h.n // 2)
    run(b)
    assert h.status() == P._lib.SPTRSV_ETIMEOUT
    plan.withhold(-1)
    ref = (oracle.solve_transpose if trans else oracle.solve)(A_h, b_h)
    assert relerr(run(b).cpu().numpy(), ref) <= 1e-12
    assert h.status() == 0
