"""The one-lane-per-row block solve over prepared strips (block mode and
batched plans with 32 rows per warp) against the CPU oracle where its tables
change shape: ends of 32-row groups, rows with none up to more dependencies
than a group stages, dependencies older than the shared-memory ring, groups
whose dependencies are taken in steps, by the inverse of their triangle and,
where the inverse grows, by the triangle itself; one to four columns a block;
padded leading dimensions; new values; rewritten systems; infinite and NaN
right-hand sides; and a row that never comes.  Tolerances: the normwise ones of
the other solve tests."""
import numpy as np
import pytest
import torch

import oracle
import synthetic as S
from helpers import TOL, relerr, widened

pytestmark = pytest.mark.gpu


def _rows(n, pick, off=lambda rng, k: rng.uniform(-1, 1, k), diag=lambda o: 1.0 + np.abs(o).sum(), seed=3):
    rng = np.random.default_rng(seed)
    rp, ci, v = [0], [], []
    for i in range(n):
        c = np.unique(pick(rng, i)).astype(np.int64)
        o = off(rng, len(c))
        ci += [*c.tolist(), i]
        v += [*o.tolist(), diag(o)]
        rp.append(len(ci))
    return S.CSR(n, np.array(rp, np.int32), np.array(ci, np.int32), np.array(v))


def _some(rng, lo, hi, k):
    lo = max(lo, 0)
    return rng.choice(np.arange(lo, hi), size=min(k, hi - lo), replace=False) if hi > lo else np.zeros(0, int)


def _classes(n=2100):
    """0 to 40 dependencies on the last 64 rows and 0 to 60 older ones, rows alternating."""
    return _rows(n, lambda rng, i: np.concatenate([_some(rng, i - 64, i, (0, 3, 16, 17, 40)[i % 5]),
                                                   _some(rng, 0, i - 64, (0, 4, 28, 29, 60, 1, 8)[i % 7])]))


CASES = {
    "one_row": lambda: S.diagonal(1, seed=1),
    "rows31": lambda: S.band_random(31, 8, 0, 8, seed=2),
    "rows32": lambda: S.band_random(32, 8, 0, 8, seed=3),
    "rows33": lambda: S.band_random(33, 8, 0, 8, seed=4),
    "chain": lambda: S.chain(700, seed=2),
    "band64": lambda: S.band_random(4001, 64, 4, 16, seed=5),
    "dense_groups": lambda: _rows(330, lambda rng, i: np.arange(max(0, i - 40), i)),
    "growing": lambda: _rows(97, lambda rng, i: np.arange(i // 32 * 32, i), lambda rng, k: np.full(k, -0.2),
                             lambda o: 1.0),
    "classes": _classes,
    "far": lambda: S.band_random(9001, 4000, 4, 16, seed=6),   # beyond every ring
    "lap2d": lambda: S.lap2d(60),
}


@pytest.mark.parametrize("dt", [np.float64, np.float32], ids=["f64", "f32"])
@pytest.mark.parametrize("name", list(CASES))
def test_strip_vs_oracle(name, dt):
    import paper_2609_40159_gb300 as P
    A_h = CASES[name]().astype(dt)
    A = P.Matrix.from_host(A_h)
    W_h = widened(A_h)
    plan = P.Plan(A, mode="block", rows_per_warp=32, transpose=True)
    for k in (1, 3, 200, 310) if A_h.n < 2000 else (1, 3):  # 1, 1, 2 and 4 columns a block
        b_h = np.abs(S.rhs(A_h.n, k, seed=k, dtype=dt))
        pad = torch.zeros(A_h.n, k + 2, dtype=torch.as_tensor(b_h).dtype, device="cuda")
        pad[:, :k] = torch.as_tensor(b_h).cuda()
        ref, ref_t = oracle.solve(W_h, b_h), oracle.solve_transpose(W_h, b_h)
        for b in (pad[:, :k], pad[:, :k].contiguous()):
            x = torch.empty_strided(b.shape, b.stride(), dtype=b.dtype, device="cuda")
            plan.solve(b, out=x)
            assert relerr(x.cpu().numpy(), ref) <= TOL[dt], k
            plan.solve_transpose(b, out=x)
            assert relerr(x.cpu().numpy(), ref_t) <= TOL[dt], ("T", k)
    assert P.handle().status() == 0


@pytest.mark.parametrize("dt", [np.float64, np.float32], ids=["f64", "f32"])
@pytest.mark.parametrize("tile", [1, 2, 4, 8])
def test_strip_batch_vs_oracle(tile, dt):
    import paper_2609_40159_gb300 as P
    hosts = [f().astype(dt) for f in CASES.values()]
    ks = [1 + (3 * m) % 9 for m in range(len(hosts))]
    plan = P.BatchPlan([P.Matrix.from_host(A) for A in hosts], nrhs=ks, rows_per_warp=32, rhs_tile=tile,
                       transpose=True)
    bs = [np.abs(S.rhs(A.n, k, seed=k, dtype=dt)) for A, k in zip(hosts, ks)]
    b = torch.as_tensor(np.concatenate([v.reshape(-1) for v in bs])).cuda()
    for run, ref in ((plan.solve, oracle.solve), (plan.solve_transpose, oracle.solve_transpose)):
        x = run(b).cpu().numpy()
        for m, (A, bh) in enumerate(zip(hosts, bs)):
            xm = x[plan.rhs_offset[m]:plan.rhs_offset[m + 1]]
            assert relerr(xm, ref(widened(A), bh)) <= TOL[dt], (m, list(CASES)[m])
    assert P.handle().status() == 0


@pytest.mark.parametrize("dt", [np.float64, np.float32], ids=["f64", "f32"])
def test_strip_not_finite(dt):
    """An infinite and a NaN right-hand side reach the rows that depend on
    them and no others."""
    import paper_2609_40159_gb300 as P
    A_h = S.band_random(3001, 200, 0, 3, seed=7).astype(dt)
    dense = CASES["dense_groups"]().astype(dt)
    for M, bad in ((A_h, 40), (A_h, 2000), (dense, 300)):
        plan = P.Plan(P.Matrix.from_host(M), mode="block", rows_per_warp=32, transpose=True)
        for v in (np.inf, np.nan):
            b_h = S.rhs(M.n, 2, seed=1, dtype=dt)
            b_h[bad, 1] = v
            for run, ref in ((plan.solve, oracle.solve), (plan.solve_transpose, oracle.solve_transpose)):
                with np.errstate(all="ignore"):
                    want = ref(widened(M), b_h)
                x = run(torch.as_tensor(b_h).cuda()).cpu().numpy()
                fin = np.isfinite(want)
                assert np.array_equal(np.isfinite(x), fin)
                assert relerr(x[fin], want[fin]) <= TOL[dt]


def test_strip_rewritten_and_new_values():
    import paper_2609_40159_gb300 as P
    A_h = S.lap2d(150)
    an = oracle.analyze(A_h)
    rows, tg = S.narrowest_levels_list(an["nlevels"], an["level_ptr"], an["perm"], 0.05, 8)
    A = P.Matrix.from_host(A_h)
    Lp, T = P.rewrite(A, P.analyze(A).lev, rows, tg)
    b_h = S.rhs(A_h.n, 2, seed=1)
    b = torch.as_tensor(b_h).cuda()
    x = P.Plan(Lp, T, mode="block", rows_per_warp=32).solve(b)
    assert relerr(x.cpu().numpy(), oracle.solve(A_h, b_h)) <= 1e-12
    plan = P.Plan(A, mode="block", rows_per_warp=32, transpose=True)
    plan.solve(b)
    A.vals.mul_(2.0)  # values may change between solves
    assert relerr(2.0 * plan.solve(b).cpu().numpy(), oracle.solve(A_h, b_h)) <= 1e-12
    assert relerr(2.0 * plan.solve_transpose(b).cpu().numpy(), oracle.solve_transpose(A_h, b_h)) <= 1e-12
    assert P.handle().status() == 0


@pytest.mark.parametrize("trans", [False, True], ids=["fwd", "transpose"])
def test_strip_bounded_wait(trans):
    """A row whose group is never counted (test hook): the block gives up
    after the plan's wait limit, and the next solve is right."""
    import paper_2609_40159_gb300 as P
    A_h = S.band_random(4001, 64, 4, 16, seed=5)
    b_h = S.rhs(A_h.n, 2, seed=2)
    b = torch.as_tensor(b_h).cuda()
    plan = P.Plan(P.Matrix.from_host(A_h), mode="block", rows_per_warp=32, transpose=True, wait_limit_us=20_000)
    h = P.handle()
    run = plan.solve_transpose if trans else plan.solve
    plan.withhold(2000)
    run(b)
    assert h.status() == P._lib.SPTRSV_ETIMEOUT
    plan.withhold(-1)
    ref = (oracle.solve_transpose if trans else oracle.solve)(A_h, b_h)
    assert relerr(run(b).cpu().numpy(), ref) <= 1e-12
    assert h.status() == 0


def test_strip_refresh_takes_several_groups_a_warp():
    """More groups than the refresh has warps (2.49M rows): a warp goes from
    group to group, in a single system and across the systems of a batch, of
    which some have no strips."""
    import paper_2609_40159_gb300 as P
    dt = np.float32
    A_h = S.band_random(2_600_003, 40, 0, 4, seed=3).astype(dt)
    A, W_h = P.Matrix.from_host(A_h), widened(A_h)
    b_h = S.rhs(A_h.n, 1, seed=1, dtype=dt)
    refs = oracle.solve(W_h, b_h), oracle.solve_transpose(W_h, b_h)
    b = torch.as_tensor(b_h).cuda()
    plan = P.Plan(A, mode="block", rows_per_warp=32, transpose=True)
    assert relerr(plan.solve(b).cpu().numpy(), refs[0]) <= TOL[dt]
    assert relerr(plan.solve_transpose(b).cpu().numpy(), refs[1]) <= TOL[dt]
    small = S.band_random(1000, 30, 0, 8, seed=4).astype(dt)
    s_h = S.rhs(small.n, 1, seed=2, dtype=dt)
    mats, rpw = [], []
    for m in range(5):
        mats += [P.Matrix.from_host(small)]
        rpw += [32 if m % 2 else 16]
    plan = P.BatchPlan([*mats, A, *mats], nrhs=[1] * 11, rows_per_warp=[*rpw, 32, *rpw], transpose=True)
    packed = torch.as_tensor(np.concatenate([*[s_h.reshape(-1)] * 5, b_h.reshape(-1), *[s_h.reshape(-1)] * 5])).cuda()
    for run, ref, big in ((plan.solve, oracle.solve, refs[0]), (plan.solve_transpose, oracle.solve_transpose, refs[1])):
        x, want = run(packed), ref(widened(small), s_h)
        for m in range(11):
            assert relerr(plan.unpack(x, m).cpu().numpy(), big if m == 5 else want) <= TOL[dt], m
    assert P.handle().status() == 0
