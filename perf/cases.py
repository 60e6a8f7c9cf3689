"""Workloads that the library is timed on.

Every case is one thing that a program does with the library through its
public entry points, on seeded inputs made on the GPU.  ``op`` says what:

  solve       x = L^{-1} b with a plan that is kept
  apply       one preconditioner application: L^{-1} b, then L^{-T} of it
  columns     the column-major multi-right-hand-side solve
  train       a differentiable solve and its gradients (b and L's values)
  plan        a matrix that is new: plan, solve and transpose solve
  analyze     the level analysis
  move        one environment move: rewrite of the list of moved rows,
              incremental re-analysis, level summary
  batch       a batched forward solve
  batch_train a batched differentiable solve and its gradients, the second
              half of the systems rewritten

``pattern`` is the matrix: ``band`` (random banded rows), ``lap2d`` and
``lap3d`` (5- and 7-point grids in natural order with varying coefficients)
or ``powerlaw`` (skewed row lengths, far-reaching columns): the families and
ranges of the repository's tests and benchmark.
"""
import math
import random

import numpy as np
import torch

import paper_2609_40159_gb300 as P

DTYPES = {"f32": torch.float32, "f64": torch.float64}
CAP, NEAR, P_NEAR, ALPHA = 512, 256, 0.7, 2.1  # the power-law family


def listed():
    return [
        # the smallest call: one small banded system, where latency is all
        {"name": "band2k_solve_f64", "op": "solve", "pattern": "band", "n": 2000, "band": 64, "kmin": 0, "kmax": 8,
         "k": 1, "dtype": "f64"},
        # a deep, narrow system with several right-hand sides, both triangles
        {"name": "band60k_apply_f32", "op": "apply", "pattern": "band", "n": 60001, "band": 64, "kmin": 4, "kmax": 16,
         "k": 7, "dtype": "f32"},
        # preconditioner application of a 2D problem, the standard single-system case
        {"name": "lap2d_apply_f64", "op": "apply", "pattern": "lap2d", "n": 1024, "k": 1, "dtype": "f64"},
        # right-hand sides that the application keeps column by column
        {"name": "lap2d_columns_f32", "op": "columns", "pattern": "lap2d", "n": 401, "k": 4, "dtype": "f32"},
        # a solve inside a training loop on an odd-sized grid
        {"name": "lap2d_train_f32", "op": "train", "pattern": "lap2d", "n": 777, "k": 1, "mat_seed": 1,
         "dtype": "f32"},
        # a differentiated 3D problem with many right-hand sides: wide levels
        {"name": "lap3d_train_f64", "op": "train", "pattern": "lap3d", "n": 128, "k": 8, "mat_seed": 4,
         "dtype": "f64"},
        # an irregular DAG with tens of thousands of levels: the largest single system
        {"name": "powerlaw_solve_f64", "op": "solve", "pattern": "powerlaw", "n": 4000000, "k": 1, "dtype": "f64"},
        # a system that is solved once: everything from the matrix on
        {"name": "lap2d_plan_f64", "op": "plan", "pattern": "lap2d", "n": 300, "k": 2, "dtype": "f64"},
        # the level structure of a large banded system
        {"name": "band300k_analyze", "op": "analyze", "pattern": "band", "n": 300000, "band": 1024, "kmin": 4,
         "kmax": 16, "dtype": "f32"},
        # one move of the rewriting environment, late in an episode
        {"name": "lap2d_move_f64", "op": "move", "pattern": "lap2d", "n": 512, "moves": 48, "mat_seed": 11,
         "dtype": "f64"},
        # many small systems at once, where launches and waiting count
        {"name": "batch32_f64", "op": "batch", "nmat": 32, "n_lo": 300, "n_hi": 6000, "w_lo": 16, "w_hi": 1024,
         "k_hi": 8, "mat_seed": 13, "dtype": "f64"},
        # the training batch: uneven systems that fill the GPU, half of them rewritten
        {"name": "batch256_train_f32", "op": "batch_train", "nmat": 256, "n_lo": 1000, "n_hi": 40000, "w_lo": 16,
         "w_hi": 1024, "k_hi": 32, "mat_seed": 3, "dtype": "f32"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["solve", "apply", "columns", "train", "plan", "analyze", "move", "batch", "batch_train"])
    case = {"op": op, "dtype": rng.choice(["f32", "f64"]), "mat_seed": rng.randrange(1 << 20)}
    if op in ("batch", "batch_train"):
        n_hi = _log_int(rng, 2000, 40000)
        case.update(nmat=_log_int(rng, 4, 256 if n_hi <= 20000 else 128), n_lo=min(300, n_hi), n_hi=n_hi, w_lo=16,
                    w_hi=1024, k_hi=_log_int(rng, 1, 32 if case["dtype"] == "f32" else 8))
        return case
    case["pattern"] = rng.choice(["band", "lap2d", "lap3d", "powerlaw"])
    if op == "move" and case["pattern"] == "powerlaw":
        case["pattern"] = "band"
    if op == "analyze" and case["pattern"] in ("lap2d", "lap3d"):  # one structure for every seed
        case["pattern"] = "powerlaw"
    if case["pattern"] == "band":
        # (the move's list of rows is substituted one by one in exact())
        case["n"] = _log_int(rng, 500, 60000 if op == "move" else 300000)
        case["band"] = _log_int(rng, 16, 1024)
        case["kmin"], case["kmax"] = rng.choice([(0, 8), (4, 16)])
        rows = case["n"]
    elif case["pattern"] == "lap2d":
        case["n"] = _log_int(rng, 24, 512 if op in ("move", "plan") else 1024)
        rows = case["n"] ** 2
    elif case["pattern"] == "lap3d":
        case["n"] = _log_int(rng, 8, 64 if op in ("move", "plan") else 128)
        rows = case["n"] ** 3
    else:
        case["n"] = _log_int(rng, 1000, 4000000 if op == "solve" else 500000)
        rows = case["n"]
    if op == "move":
        case["moves"] = rng.randint(1, 64)
    elif op != "analyze":
        most = {"band": 32, "lap2d": 32, "lap3d": 8, "powerlaw": 4}[case["pattern"]]
        k = 1 if rows > 500000 and case["pattern"] == "powerlaw" else _log_int(rng, 1, most)
        case["k"] = max(1, min(k, (1 << 24) // rows))
    return case


# ------------------------------------------------------------------ matrices
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) % (1 << 62))


def _rand(shape, g, dtype=torch.float64):
    return torch.rand(shape, generator=g, device="cuda", dtype=dtype)


def _seeds(case, seed):
    """Generators of the structure and of the values.  Where the sizes of
    the results follow from the structure (gradients, rewritten systems) it
    belongs to the case, and the seed draws the values."""
    fixed = case["op"] in ("train", "move", "batch_train")
    return _gen(case["mat_seed"] if fixed else seed), _gen(seed * 7 + 3)


def _assemble(counts, cols, g, dtype):
    """CSR tensors from off-diagonals per row and their columns, row by row
    and ascending: values U(-1, 1), the diagonal 1 + sum |.| stored last."""
    n = counts.numel()
    rp = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(counts + 1, 0, out=rp[1:])
    rows = torch.repeat_interleave(torch.arange(n, device="cuda"), counts)
    pos = torch.arange(cols.numel(), device="cuda") + rows  # one diagonal before it per earlier row
    off = _rand(cols.numel(), g) * 2 - 1
    dsum = torch.ones(n, dtype=torch.float64, device="cuda")
    # ordered sums, so that the same seed gives the same bits
    c = torch.cat([torch.zeros(1, dtype=torch.float64, device="cuda"), torch.cumsum((off.abs() * 2 ** 40).long(), 0).double() / 2 ** 40])
    e = torch.cumsum(counts, 0)
    dsum += c[e] - c[e - counts]
    ci = torch.empty(cols.numel() + n, dtype=torch.int32, device="cuda")
    v = torch.empty(cols.numel() + n, dtype=dtype, device="cuda")
    ci[pos] = cols.to(torch.int32)
    v[pos] = off.to(dtype)
    ci[rp[1:] - 1] = torch.arange(n, dtype=torch.int32, device="cuda")
    v[rp[1:] - 1] = dsum.to(dtype)
    return rp.to(torch.int32), ci, v


def _band_columns(i, band, counts, kmax, g):
    """counts[q] distinct columns of [i[q] - m, i[q]), m = min(i, band), for
    every row q, flattened row by row and ascending."""
    m = torch.minimum(i, band)
    big = 1 << 60
    take = torch.arange(kmax, device="cuda")[None, :] < counts[:, None]
    out = torch.full(take.shape, big, dtype=torch.int64, device="cuda")
    small = m <= 64  # narrow windows: the first of a random order
    if bool(small.any()):
        ms = m[small]
        key = _rand((ms.numel(), 64), g, torch.float32)
        key[torch.arange(64, device="cuda")[None, :] >= ms[:, None]] = 2.0
        out[small] = torch.argsort(key, dim=1)[:, :kmax]
    wide = ~small
    if bool(wide.any()):
        mw, tw = m[wide], take[wide]
        d = (_rand(tw.shape, g) * mw[:, None]).long()
        while True:  # redraw what a row holds twice
            d = torch.where(tw, d, big).sort(dim=1).values
            twice = torch.zeros_like(tw)
            twice[:, 1:] = (d[:, 1:] == d[:, :-1]) & tw[:, 1:]
            if not bool(twice.any()):
                break
            d = torch.where(twice, (_rand(tw.shape, g) * mw[:, None]).long(), d)
        out[wide] = d
    out = torch.where(take, out, big).sort(dim=1).values
    return (out + (i - m)[:, None])[take]


def _band(n, band, kmin, kmax, g, gv, dtype):
    i = torch.arange(n, device="cuda")
    counts = torch.randint(kmin, kmax + 1, (n,), generator=g, device="cuda")
    counts = torch.minimum(counts, i.clamp(max=band))
    cols = _band_columns(i, torch.full_like(i, band), counts, kmax, g)
    return _assemble(counts, cols, gv, dtype)


def _grid(N, dims, g, dtype):
    n = N ** dims
    i = torch.arange(n, device="cuda")
    strides = [N ** d for d in reversed(range(dims))]
    has = torch.stack([(i // s) % N > 0 for s in strides], 1)
    counts = has.sum(1)
    rp = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(counts + 1, 0, out=rp[1:])
    ci = torch.empty(int(rp[-1]), dtype=torch.int32, device="cuda")
    v = torch.empty(int(rp[-1]), dtype=dtype, device="cuda")
    p = rp[:-1].clone()
    for d, s in enumerate(strides):
        h = has[:, d]
        ci[p[h]] = (i[h] - s).to(torch.int32)
        v[p[h]] = -(0.5 + _rand(int(h.sum()), g)).to(dtype)
        p += h
    ci[p] = i.to(torch.int32)
    v[p] = 2.0 * dims
    return rp.to(torch.int32), ci, v


def _zipf():
    p = np.arange(1, CAP + 1, dtype=np.float64) ** -ALPHA
    return p / p.sum()


def _powerlaw(n, g, gv, dtype):
    cdf = torch.as_tensor(np.cumsum(_zipf())).cuda()
    cdf[-1] = 1.0
    i = torch.arange(n, device="cuda")
    counts = torch.minimum(torch.searchsorted(cdf, _rand(n, g), right=True) + 1, i)
    rows = torch.repeat_interleave(i, counts)
    rank = torch.arange(rows.numel(), device="cuda") - (torch.cumsum(counts, 0) - counts)[rows]
    full = (2 * counts > i)[rows]  # the first rows take their nearest columns

    def fresh():
        lo = (rows - NEAR).clamp(min=0)
        u, near = _rand(rows.numel(), g), _rand(rows.numel(), g) < P_NEAR
        c = torch.where(near, lo + (u * (rows - lo)).long(), (u * rows).long())
        return torch.where(full, rows - 1 - rank, c)

    c = fresh()
    while True:
        c = (rows * n + c).sort().values - rows * n
        twice = torch.zeros_like(full)
        twice[1:] = (rows[1:] == rows[:-1]) & (c[1:] == c[:-1])
        if not bool(twice.any()):
            break
        c = torch.where(twice, fresh(), c)
    return _assemble(counts, c, gv, dtype)


def _system(case, seed):
    (g, gv), dt = _seeds(case, seed), DTYPES[case["dtype"]]
    if case["pattern"] == "band":
        return _band(case["n"], case["band"], case["kmin"], case["kmax"], g, gv, dt)
    if case["pattern"] == "powerlaw":
        return _powerlaw(case["n"], g, gv, dt)
    return _grid(case["n"], 2 if case["pattern"] == "lap2d" else 3, gv, dt)


def _rows(case):
    return case["n"] ** {"lap2d": 2, "lap3d": 3}.get(case["pattern"], 1)


def _batch_spec(case):
    """(rows, band, right-hand sides) of every system of a batch."""
    rng = random.Random(case["mat_seed"])
    return [(_log_int(rng, case["n_lo"], case["n_hi"]), _log_int(rng, case["w_lo"], case["w_hi"]),
             _log_int(rng, 1, case["k_hi"])) for _ in range(case["nmat"])]


def _batch_systems(case, seed):
    """The batch's systems, drawn together and cut apart."""
    spec, (g, gv) = _batch_spec(case), _seeds(case, seed)
    ns = torch.tensor([s[0] for s in spec], device="cuda")
    first = torch.cumsum(ns, 0) - ns
    sys_of = torch.repeat_interleave(torch.arange(len(spec), device="cuda"), ns)
    i = torch.arange(int(ns.sum()), device="cuda") - first[sys_of]
    band = torch.tensor([s[1] for s in spec], device="cuda")[sys_of]
    counts = torch.randint(4, 17, (i.numel(),), generator=g, device="cuda")
    counts = torch.minimum(counts, torch.minimum(i, band))
    cols = _band_columns(i, band, counts, 16, g)
    rp, ci, v = _assemble(counts, cols, gv, DTYPES[case["dtype"]])
    # (the diagonals hold the row of the whole batch: back to the system's own)
    ci[rp[1:].long() - 1] = i.to(torch.int32)
    cut = torch.cat([first, ns.sum()[None]]).tolist()
    ends = rp[cut].tolist()
    return [((rp[a:b + 1] - p).contiguous(), ci[p:q].contiguous(), v[p:q].contiguous())
            for a, b, p, q in zip(cut, cut[1:], ends, ends[1:])]


def _narrowest(lev, frac=0.01, depth=8):
    """Rows and target levels of the narrowest levels that hold `frac` of the
    rows, every run of at most `depth` consecutive levels moved above itself."""
    lev = lev.cpu().numpy()
    width = np.bincount(lev)
    order = np.lexsort((np.arange(1, len(width)), width[1:])) + 1
    count = int(np.searchsorted(np.cumsum(width[order]), math.ceil(frac * len(lev)))) + 1
    target = np.full(len(width), -1, np.int64)
    run = 0
    picked = np.zeros(len(width), bool)
    picked[order[:count]] = True
    for l in range(1, len(width)):
        if picked[l]:
            run = run + 1 if picked[l - 1] and run < depth else 1
            target[l] = l - run
        else:
            run = 0
    rows = np.flatnonzero(target[lev] >= 0)
    return rows.astype(np.int32), target[lev[rows]].astype(np.int32)


def _moves(lev, row_ptr, count, seed):
    """A list of moves: in randomly picked levels the row with the fewest
    dependencies, to a level up to 8 above it."""
    order = np.lexsort((np.arange(len(lev)), np.diff(row_ptr), lev))
    first = np.searchsorted(lev[order], np.arange(lev.max() + 1))
    rng = np.random.default_rng(seed)
    levels = rng.permutation(np.arange(1, lev.max() + 1))[:count]
    targets = np.maximum(0, levels - rng.integers(1, 9, size=len(levels)))
    return order[first[levels]].astype(np.int32), targets.astype(np.int32)


# ------------------------------------------------------------------- passes
def _rhs(n, k, seed, dtype, salt):
    return _rand((n, k) if k else (n,), _gen(seed * 7 + salt), dtype) * 2 - 1


def prepare(case, seed):
    op, dt = case["op"], DTYPES[case["dtype"]]
    if op in ("batch", "batch_train"):
        nrhs = [s[2] for s in _batch_spec(case)]
        mats = [P.Matrix(*t) for t in _batch_systems(case, seed)]
        Ts = [None] * len(mats)
        if op == "batch_train":
            for m in range(len(mats) // 2, len(mats)):
                lev = P.analyze(mats[m]).lev
                rows, targets = _narrowest(lev)
                mats[m], Ts[m] = P.rewrite(mats[m], lev, rows, targets)
        plan = P.BatchPlan(mats, Ts, nrhs, transpose=op == "batch_train")
        total = sum(A.n * k for A, k in zip(mats, nrhs))
        state = {"plan": plan, "b": _rhs(total, 0, seed, dt, 1), "w": _rhs(total, 0, seed, dt, 2),
                 "cut": sum(A.nnz for A in mats[:len(mats) // 2])}
        if op == "batch_train":
            plan.vals.requires_grad_(True)
            state["b"].requires_grad_(True)
    else:
        A = P.Matrix(*_system(case, seed))
        state = {"A": A}
        if op == "move":
            lev = P.analyze(A).lev
            rows, targets = _moves(lev.cpu().numpy(), A.row_ptr.cpu().numpy(), case["moves"], case["mat_seed"])
            before = lev
            if len(rows) > 1:
                before = P.analyze(P.rewrite(A, lev, rows[:-1], targets[:-1])[0]).lev
            state.update(lev=lev, rows=rows, targets=targets, before=before)
        elif op == "analyze":
            # the program's own tables, which fit any level structure
            state["tables"] = [torch.zeros(A.n + 1, dtype=dt, device="cuda") for dt in (torch.int32, torch.int64)]
        else:
            k = case["k"]
            state["b"] = _rhs(A.n, k, seed, dt, 1)
            if op == "columns":
                state["b"] = torch.empty(k, A.n, dtype=dt, device="cuda").copy_(state["b"].t())
            if op != "plan":
                state["plan"] = P.Plan(A, transpose=op in ("apply", "train"))
            if op == "train":
                A.vals.requires_grad_(True)
                state["b"].requires_grad_(True)
                state["w"] = _rhs(A.n, k, seed, dt, 2)
    state["op"] = op
    return state


def run(state):
    op = state["op"]
    if op == "solve":
        return state["plan"].solve(state["b"])
    if op == "apply":
        y = state["plan"].solve(state["b"])
        return [y, state["plan"].solve_transpose(y)]
    if op == "columns":
        return state["plan"].solve_columns(state["b"])
    if op == "train":
        x = P.solve(state["plan"], state["b"])
        gb, gv = torch.autograd.grad(x, (state["b"], state["A"].vals), state["w"])
        return [x, gb, gv]
    if op == "plan":
        plan = P.Plan(state["A"], transpose=True)
        return [plan.solve(state["b"]), plan.solve_transpose(state["b"])]
    if op == "batch":
        return state["plan"].solve(state["b"])
    if op == "batch_train":
        plan = state["plan"]
        x = P.batch_solve(plan, state["b"])
        gb, gv = torch.autograd.grad(x, (state["b"], plan.vals), state["w"])
        return [x, gb, gv[:state["cut"]], gv[state["cut"]:]]
    A = state["A"]
    if op == "analyze":
        an = P.analyze(A)
        for table, part in zip(state["tables"], (an.level_ptr, an.cost)):
            table[:part.numel()] = part
        return [an.lev, an.perm, *state["tables"], an.nlevels, an.stats]
    Lp, T = P.rewrite(A, state["lev"], state["rows"], state["targets"])
    an = P.analyze(Lp, prev_lev=state["before"], first_row=int(state["rows"][-1]))
    thin, pick, summary = P.level_summary(Lp, an)
    return [Lp.vals, T.vals, an.stats, Lp.row_ptr, Lp.col_idx, T.row_ptr, T.col_idx, an.lev, an.perm, an.level_ptr,
            an.cost, thin, pick, summary]


def _nnz(case):
    """Stored entries, as far as the case alone says (random rows: expected)."""
    n = case["n"]
    if case["pattern"] == "band":
        return n * (1 + 0.5 * (case["kmin"] + case["kmax"]))
    if case["pattern"] == "powerlaw":
        return n * (1 + float(np.dot(np.arange(1, CAP + 1), _zipf())))
    dims = 2 if case["pattern"] == "lap2d" else 3
    return n ** dims + dims * (n - 1) * n ** (dims - 1)


def work(case):
    w = 4 if case["dtype"] == "f32" else 8

    def solve(n, nnz, k):
        return nnz * (w + 4) + (n + 1) * 4 + 2 * n * k * w

    def grads(n, nnz, k):  # the transpose solve, and the value gradient from what is then at hand
        return solve(n, nnz, k) + nnz * (w + 4) + n * k * w

    op = case["op"]
    if op in ("batch", "batch_train"):
        total = flops = 0
        for n, _, k in _batch_spec(case):
            nnz = 11 * n
            total += solve(n, nnz, k) + (grads(n, nnz, k) if op == "batch_train" else 0)
            flops += 2 * nnz * k * (3 if op == "batch_train" else 1)
        return {"bytes": total, "flops": flops}
    n, nnz, k = _rows(case), _nnz(case), case.get("k", 0)
    if op in ("solve", "columns"):
        return {"bytes": solve(n, nnz, k), "flops": 2 * nnz * k}
    if op in ("apply", "plan"):
        return {"bytes": 2 * solve(n, nnz, k), "flops": 4 * nnz * k}
    if op == "train":
        return {"bytes": solve(n, nnz, k) + grads(n, nnz, k), "flops": 6 * nnz * k}
    table = nnz * 4 + n * 4 + 2 * n * 4  # the pattern read; levels and order written
    if op == "analyze":
        return {"bytes": table, "flops": nnz}
    return {"bytes": 2 * nnz * (w + 4) + 2 * n * 4 + table, "flops": nnz}


# -------------------------------------------------------------- in 64 bits
def _solve64(rp, ci, v, b, trans=False):
    """L^{-1} b or L^{-T} b by the iteration x <- D^{-1} (b - N x), which ends
    at the solution after at most as many steps as L has levels and, L being
    diagonally dominant, long before in 64 bits (to within the order in
    which a row's terms are added)."""
    n = rp.numel() - 1
    rows = torch.repeat_interleave(torch.arange(n, device="cuda"), (rp[1:] - rp[:-1]).long())
    cols, v, b = ci.long(), v.detach().double(), b.detach().double()
    b = b.reshape(n, -1)
    d = v[(rp[1:] - 1).long()][:, None]
    off = rows != cols
    to, fr, val = rows[off], cols[off], v[off][:, None]
    if trans:
        to, fr = fr, to
    y = b / d
    while True:
        for _ in range(16):
            x, y = y, (b - torch.zeros_like(b).index_add_(0, to, val * y[fr])) / d
        if float((y - x).abs().max()) <= 4e-15 * float(y.abs().max()):
            return y


def _grad64(rp, ci, gb, x):
    n = rp.numel() - 1
    rows = torch.repeat_interleave(torch.arange(n, device="cuda"), (rp[1:] - rp[:-1]).long())
    return -(gb.reshape(n, -1)[rows] * x.reshape(n, -1)[ci.long()]).sum(1)


def _levels(rp, ci):
    """Longest path to every row, by rounds over all rows until none moves."""
    n = rp.numel() - 1
    rows = torch.repeat_interleave(torch.arange(n, device="cuda"), (rp[1:] - rp[:-1]).long())
    cols = ci.long()
    off = rows != cols
    rows, cols = rows[off], cols[off]
    lev = torch.zeros(n, dtype=torch.int64, device="cuda")
    while True:
        old = lev
        for _ in range(32):
            lev = torch.zeros_like(lev).scatter_reduce_(0, rows, lev[cols] + 1, "amax")
        if torch.equal(lev, old):
            return lev.cpu().numpy()


def _stats(rp, lev):
    """ALC, ARL, AIR, CV of level costs and of rows per level, threshold."""
    offs = np.diff(rp) - 1
    cost, rows = np.bincount(lev, 2.0 * offs + 1), np.bincount(lev).astype(np.float64)
    cv = cost.std() / cost.mean()
    return np.array([cost.mean(), rows.mean(), offs.sum() / len(lev), cv, rows.std() / rows.mean(),
                     cost.mean() * (1 + max(0.0, 1 - cv))])


def _rewrite64(rp, ci, v, lev, rows, targets):
    """(values of L', values of T, L' as lists of columns): each listed row's
    predecessors at or above its target level substituted, largest first."""
    listed_ = dict(zip(rows.tolist(), targets.tolist()))
    vals, ends, pattern, t_vals, at = [], [], [], [], 0
    for i in sorted(listed_):
        acc = dict(zip(ci[rp[i]:rp[i + 1] - 1].tolist(), v[rp[i]:rp[i + 1] - 1].tolist()))
        sub = {}
        while True:
            todo = [j for j in acc if lev[j] >= listed_[i] and j not in sub]
            if not todo:
                break
            j = max(todo)
            m = acc[j] / v[rp[j + 1] - 1]
            sub[j] = -m
            for p in range(rp[j], rp[j + 1] - 1):
                acc[int(ci[p])] = acc.get(int(ci[p]), 0.0) - m * v[p]
        left = sorted(j for j in acc if j not in sub)
        vals += [v[rp[at]:rp[i]], np.array([acc[j] for j in left] + [v[rp[i + 1] - 1]])]
        pattern += [ci[rp[at]:rp[i]], np.array(left + [i])]
        ends.append((i, len(left) + 1))
        t_vals += [sub[j] for j in sorted(sub)]
        at = i + 1
    vals.append(v[rp[at]:])
    pattern.append(ci[rp[at]:])
    counts = np.diff(rp)
    for i, c in ends:
        counts[i] = c
    return np.concatenate(vals), np.array(t_vals), np.concatenate([[0], np.cumsum(counts)]), np.concatenate(pattern)


def exact(case, seed):
    op, dt = case["op"], DTYPES[case["dtype"]]
    if op in ("batch", "batch_train"):
        spec, systems = _batch_spec(case), _batch_systems(case, seed)
        total = sum(s[0] * s[2] for s in spec)
        b, w = _rhs(total, 0, seed, dt, 1), _rhs(total, 0, seed, dt, 2)
        x, gb, gv, a = [], [], [], 0
        for m, ((n, _, k), (rp, ci, v)) in enumerate(zip(spec, systems)):
            x.append(_solve64(rp, ci, v, b[a:a + n * k].view(n, k)))
            if op == "batch_train":
                # (a rewritten system has the original's solution and gradient)
                gb.append(_solve64(rp, ci, v, w[a:a + n * k].view(n, k), True))
                if m < len(spec) // 2:
                    gv.append(_grad64(rp, ci, gb[-1], x[-1]))
            a += n * k
        flat = torch.cat([t.reshape(-1) for t in x])
        if op == "batch":
            return flat
        return [flat, torch.cat([t.reshape(-1) for t in gb]), torch.cat(gv), None]
    rp, ci, v = _system(case, seed)
    if op in ("analyze", "move"):
        lev = _levels(rp, ci)
        rp, ci, v = (t.cpu().numpy() for t in (rp, ci, v.double()))
        if op == "analyze":
            return [None, None, None, None, None, _stats(rp, lev)]
        rows, targets = _moves(lev, rp, case["moves"], case["mat_seed"])
        vals, t_vals, rp2, ci2 = _rewrite64(rp, ci, v, lev, rows, targets)
        lev2 = _levels(torch.as_tensor(rp2).cuda(), torch.as_tensor(ci2).cuda())
        return [vals, t_vals, _stats(rp2, lev2)] + [None] * 11
    b = _rhs(rp.numel() - 1, case["k"], seed, dt, 1)
    x = _solve64(rp, ci, v, b)
    if op == "solve":
        return x
    if op == "columns":
        return x.t().contiguous()
    if op == "apply":
        return [x, _solve64(rp, ci, v, x, True)]
    if op == "plan":
        return [x, _solve64(rp, ci, v, b, True)]
    gb = _solve64(rp, ci, v, _rhs(rp.numel() - 1, case["k"], seed, dt, 2), True)
    return [x, gb, _grad64(rp, ci, gb, x)]
