"""The cluster flow solve (the automatic hybrid schedule) against the CPU
oracle where its tables change shape: levels narrower and wider than a warp
and than the cluster, every length class of a row (up to 4, 16, 64 entries and
beyond the 128 staged ones), systems shorter than, at and beyond the
shared-memory ring (27,648 FP32 or 13,824 FP64 positions) so that old
dependencies come from global memory, one to many right-hand sides (one
cluster each), padded leading dimensions, rewritten systems, and a row that
never comes.  Tolerances: the normwise ones of the other solve tests."""
import numpy as np
import pytest
import torch

import oracle
import synthetic as S
from helpers import TOL, relerr, two_wide_levels, widened

pytestmark = pytest.mark.gpu


def _class_edges(n=3000):
    """Rows with 0, 1, 4, 5, 16, 17, 64, 65, 128, 129, 300 off-diagonals in turn."""
    rng = np.random.default_rng(3)
    lens = [0, 1, 4, 5, 16, 17, 64, 65, 128, 129, 300]
    rp, ci, v = [0], [], []
    for i in range(n):
        k = min(lens[i % len(lens)], i)
        c = np.sort(rng.choice(i, size=k, replace=False)) if k else np.zeros(0, int)
        off = rng.uniform(-1, 1, k)
        ci += [*c.tolist(), i]
        v += [*off.tolist(), 1.0 + np.abs(off).sum()]
        rp.append(len(ci))
    return S.CSR(n, np.array(rp, np.int32), np.array(ci, np.int32), np.array(v))


CASES = {
    "one_row": lambda: S.diagonal(1, seed=1),
    "classes": _class_edges,
    "chain": lambda: S.chain(700, seed=2),
    "wide": lambda: two_wide_levels(40_000, seed=4),       # levels wider than an epoch
    "ring_f64": lambda: S.lap2d(118),                      # 13,924 rows: just beyond one ring (FP64)
    "ring_f32": lambda: S.lap2d(167),                      # 27,889 rows: just beyond one ring (FP32)
    "far": lambda: S.powerlaw(60_000, seed=5),             # dependencies several rings back
    "lap3d": lambda: S.lap3d(31),
    "band": lambda: S.band_random(30_001, 4096, 4, 16, seed=6),
}


@pytest.mark.parametrize("dt", [np.float64, np.float32], ids=["f64", "f32"])
@pytest.mark.parametrize("name", list(CASES))
def test_flow_vs_oracle(name, dt):
    import paper_2609_40159_gb300 as P
    A_h = CASES[name]().astype(dt)
    A = P.Matrix.from_host(A_h)
    plan = P.Plan(A, mode="hybrid", transpose=True)
    for k in (1, 3, 20):
        b_h = S.rhs(A_h.n, k, seed=k, dtype=dt)
        pad = torch.zeros(A_h.n, k + 2, dtype=torch.as_tensor(b_h).dtype, device="cuda")
        pad[:, :k] = torch.as_tensor(b_h).cuda()
        for b in (pad[:, :k], pad[:, :k].contiguous()):
            x = torch.empty_strided(b.shape, b.stride(), dtype=b.dtype, device="cuda")
            for _ in range(2):  # a second solve on the same plan
                plan.solve(b, out=x)
                assert relerr(x.cpu().numpy(), oracle.solve(widened(A_h), b_h)) <= TOL[dt], k
                plan.solve_transpose(b, out=x)
                assert relerr(x.cpu().numpy(), oracle.solve_transpose(widened(A_h), b_h)) <= TOL[dt], ("T", k)
    assert P.handle().status() == 0


def test_flow_rewritten_and_new_values():
    import paper_2609_40159_gb300 as P
    A_h = S.lap2d(150)
    an = oracle.analyze(A_h)
    rows, tg = S.narrowest_levels_list(an["nlevels"], an["level_ptr"], an["perm"], 0.05, 8)
    A = P.Matrix.from_host(A_h)
    Lp, T = P.rewrite(A, P.analyze(A).lev, rows, tg)
    b_h = S.rhs(A_h.n, 2, seed=1)
    b = torch.as_tensor(b_h).cuda()
    assert relerr(P.Plan(Lp, T, mode="hybrid").solve(b).cpu().numpy(), oracle.solve(A_h, b_h)) <= 1e-12
    plan = P.Plan(A, mode="hybrid", transpose=True)
    plan.solve(b)
    A.vals.mul_(2.0)  # values may change between solves
    assert relerr(2.0 * plan.solve(b).cpu().numpy(), oracle.solve(A_h, b_h)) <= 1e-12
    assert relerr(2.0 * plan.solve_transpose(b).cpu().numpy(), oracle.solve_transpose(A_h, b_h)) <= 1e-12
    assert P.handle().status() == 0


@pytest.mark.parametrize("trans", [False, True], ids=["fwd", "transpose"])
def test_flow_bounded_wait(trans):
    """A row whose solution is never passed on (test hook): every block of
    the cluster gives up after the plan's wait limit, and the next solve is
    right."""
    import paper_2609_40159_gb300 as P
    A_h = S.lap2d(150)
    A = P.Matrix.from_host(A_h)
    b_h = S.rhs(A_h.n, 2, seed=2)
    b = torch.as_tensor(b_h).cuda()
    plan = P.Plan(A, mode="hybrid", transpose=True, wait_limit_us=20_000)
    h = P.handle()
    run = plan.solve_transpose if trans else plan.solve
    plan.withhold(150 * 75 + 75)
    run(b)
    assert h.status() == P._lib.SPTRSV_ETIMEOUT
    plan.withhold(-1)
    ref = (oracle.solve_transpose if trans else oracle.solve)(A_h, b_h)
    assert relerr(run(b).cpu().numpy(), ref) <= 1e-12
    assert h.status() == 0


@pytest.mark.parametrize("trans", [False, True], ids=["fwd", "transpose"])
def test_flow_gives_up_once_for_all_columns(trans):
    """One cluster per right-hand side, more of them than the GPU holds at a
    time (one block on an SM): a row that never comes ends the solve after
    about one wait limit, not after one for every wave of clusters."""
    import time

    import paper_2609_40159_gb300 as P
    A_h = S.lap2d(200)
    k = 4 * torch.cuda.get_device_properties(0).multi_processor_count  # four waves at least
    limit_s = 0.4
    b_h = S.rhs(A_h.n, k, seed=2, dtype=np.float32)
    b = torch.as_tensor(b_h).cuda()
    plan = P.Plan(P.Matrix.from_host(A_h.astype(np.float32)), mode="hybrid", transpose=True,
                  wait_limit_us=int(1e6 * limit_s))
    h = P.handle()
    run = plan.solve_transpose if trans else plan.solve
    run(b)
    torch.cuda.synchronize()
    plan.withhold(200 * 100 + 100)
    t0 = time.perf_counter()
    run(b)
    assert h.status() == P._lib.SPTRSV_ETIMEOUT
    # (the limit is counted at 2.2 GHz, above the clock: up to half as long again)
    assert time.perf_counter() - t0 < 2.5 * limit_s
    plan.withhold(-1)
    ref = (oracle.solve_transpose if trans else oracle.solve)(A_h, b_h[:, -3:].astype(np.float64))
    assert relerr(run(b).cpu().numpy()[:, -3:], ref) <= TOL[np.float32]
    assert h.status() == 0
