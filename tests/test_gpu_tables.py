"""Plans whose schedule tables cannot be had (test hook), and settings that
call for other tables: whatever a solve needs is there before it, so that the
first one launches kernels only and can be captured; results against the CPU
oracle."""
import numpy as np
import pytest
import torch

import oracle
import synthetic as S
from helpers import relerr

pytestmark = pytest.mark.gpu


def _first_solves_captured(plan, A_h):
    """The plan's first forward and transpose solves, under capture."""
    import paper_2609_40159_gb300 as P
    b_h = S.rhs(A_h.n, 2, seed=2)
    s = torch.cuda.current_stream()
    b = torch.as_tensor(b_h).cuda()
    x, y = torch.zeros_like(b), torch.zeros_like(b)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        plan.solve(b, out=x)
        plan.solve_transpose(b, out=y)
    g.replay()
    s.synchronize()
    assert relerr(x.cpu().numpy(), oracle.solve(A_h, b_h)) <= 1e-12
    assert relerr(y.cpu().numpy(), oracle.solve_transpose(A_h, b_h)) <= 1e-12
    assert P.handle().status() == 0


def _loaded(A, mode):
    """The kernels of the mode are on the device before a capture."""
    import paper_2609_40159_gb300 as P
    b = torch.ones(A.n, 2, dtype=torch.float64, device="cuda")
    plan = P.Plan(A, mode=mode, transpose=True)
    plan.solve(b)
    plan.solve_transpose(b)


@pytest.mark.parametrize("mode", ["hybrid", "block"])
def test_without_tables(mode):
    import paper_2609_40159_gb300 as P
    A_h = S.lap2d(90)
    A = P.Matrix.from_host(A_h)
    with torch.cuda.stream(torch.cuda.Stream()):
        h = P.handle()
        try:
            h.limit_tables(0)
            _loaded(A, mode)
            plan = P.Plan(A, mode=mode, transpose=True)
            assert plan.info()["mode"] == P.Plan(A, mode=mode).info()["mode"]
            _first_solves_captured(plan, A_h)
        finally:
            h.limit_tables(-1)
        _loaded(A, mode)
        _first_solves_captured(P.Plan(A, mode=mode, transpose=True), A_h)
    torch.cuda.synchronize()


def test_batch_without_tables():
    import paper_2609_40159_gb300 as P
    hosts = [S.band_random(n, 60, 0, 6, seed=n) for n in (33, 700, 2100)]
    h = P.handle()
    h.limit_tables(0)
    try:
        plan = P.BatchPlan([P.Matrix.from_host(A) for A in hosts], nrhs=[1, 5, 2], transpose=True)
    finally:
        h.limit_tables(-1)
    bs = [S.rhs(A.n, k, seed=k) for A, k in zip(hosts, (1, 5, 2))]
    b = torch.as_tensor(np.concatenate([v.reshape(-1) for v in bs])).cuda()
    for run, ref in ((plan.solve, oracle.solve), (plan.solve_transpose, oracle.solve_transpose)):
        x = run(b)
        for m, (A, bh) in enumerate(zip(hosts, bs)):
            assert relerr(plan.unpack(x, m).cpu().numpy(), ref(A, bh)) <= 1e-12
    assert h.status() == 0


def test_settings_bring_their_tables():
    import paper_2609_40159_gb300 as P
    A_h = S.lap2d(90)
    A = P.Matrix.from_host(A_h)

    def thin_rows(p):   # to the automatic threshold while the mode is hybrid already
        p.set_thin_rows(100)
        p.set(mode="hybrid")
        p.set_thin_rows(0)

    def grid(p):        # to a capped grid
        p.set(mode="hybrid")
        p.set_blocks_per_sm(2)

    def full_grid(p):   # and back, tables first needed then
        p.set_blocks_per_sm(2)
        p.set(mode="hybrid")
        p.set_blocks_per_sm(0)

    with torch.cuda.stream(torch.cuda.Stream()):
        for change in (thin_rows, grid, full_grid):
            for first in (True, False):  # the kernels are loaded by then
                plan = P.Plan(A, mode="level", transpose=True)
                change(plan)
                if first:
                    b = torch.ones(A.n, 2, dtype=torch.float64, device="cuda")
                    plan.solve(b)
                    plan.solve_transpose(b)
                else:
                    _first_solves_captured(plan, A_h)
    torch.cuda.synchronize()


def _launches(run):
    """Number of nodes of run() under capture."""
    import ctypes
    with open("/proc/self/maps") as f:
        path = next(ln.split()[-1] for ln in f if "libcudart.so" in ln)
    rt = ctypes.CDLL(path)
    g = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(g, stream=torch.cuda.current_stream()):
        run()
    count = ctypes.c_size_t(0)
    assert rt.cudaGraphGetNodes(ctypes.c_void_p(g.raw_cuda_graph()), None, ctypes.byref(count)) == 0
    return count.value


def test_batch_lays_out_what_it_reads():
    """The launch that lays the values out in strips is there only while some
    system of the direction is solved over them, and a system comes back to
    them."""
    import paper_2609_40159_gb300 as P
    hosts = [S.band_random(n, 60, 0, 6, seed=n) for n in (33, 700, 2100)]
    ks, nmat = [1, 5, 2], 3
    bs = [S.rhs(A.n, k, seed=k) for A, k in zip(hosts, ks)]
    with torch.cuda.stream(torch.cuda.Stream()):
        plan = P.BatchPlan([P.Matrix.from_host(A) for A in hosts], nrhs=ks, transpose=True)
        b = torch.as_tensor(np.concatenate([v.reshape(-1) for v in bs])).cuda()
        out = torch.empty_like(b)

        def check():
            for run, ref in ((plan.solve, oracle.solve), (plan.solve_transpose, oracle.solve_transpose)):
                x = run(b)
                for m, (A, bh) in enumerate(zip(hosts, bs)):
                    assert relerr(plan.unpack(x, m).cpu().numpy(), ref(A, bh)) <= 1e-12
            return _launches(lambda: plan.solve(b, out=out)), _launches(lambda: plan.solve_transpose(b, out=out))

        strips = check()
        plan.set_schedule(["level"] * nmat)
        # (the transpose: L's values in CSC order instead)
        assert check() == (strips[0] - 1, strips[1])
        plan.set_schedule(["inorder"] * nmat)
        assert check() == strips
        plan.set_geometry([16] * nmat, direction="forward")
        assert check() == (strips[0] - 1, strips[1])
        plan.set_geometry([16, 32, 16], direction="forward")
        assert check() == strips
        assert P.handle().status() == 0
    torch.cuda.synchronize()
