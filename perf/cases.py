"""The calls whose speed is measured: what a program that uses the library has it do.

Each case is one call, or the short sequence of calls that belongs together, through the
package's entry points: builds (uniform, learned, adaptive counts, walk reuse, batched),
solves (PCG in FP64 and mixed, BiCGSTAB, batched), the bare preconditioner and SpMV, and
the training of the budget network.  Matrices are drawn on the GPU with the structure and
the distributions of the repository's workloads; drawn cases vary edges, walks, right-hand
sides and matrix counts up to the listed sizes.
"""
import math

import numpy as np
import torch

import paper_math_0609672_gb300 as P

# Entries of Y per row at the listed settings (rounded), for work().
FILL = {"grid2d": 9, "grid7": 35, "grid27": 70, "longrange": 60, "laplace": 13, "asym": 20, "rgg": 20}
# Stored entries of A per row (upper bound, interior rows).
ROW = {"grid2d": 5, "grid7": 7, "grid27": 27, "longrange": 9, "laplace": 7, "asym": 7, "rgg": 9}
TOL = 1e-6


def listed():
    return [
        # the smallest calls: a 32 x 32 grid, where latency and launches are the time
        {"name": "apply-grid2d-32", "do": "apply", "graph": "grid2d", "nx": 32, "ny": 32, "nz": 1, "walks": 200,
         "nrhs": 1},
        {"name": "build-grid2d-32", "do": "build", "graph": "grid2d", "nx": 32, "ny": 32, "nz": 1, "walks": 200},
        # an outer solver's matrix product, ragged edges and right-hand sides
        {"name": "spmv-grid27-ragged", "do": "spmv", "graph": "grid27", "nx": 101, "ny": 97, "nz": 89, "nrhs": 3},
        # the factor of a 64^3 7-point grid, and its solve for four right-hand sides
        {"name": "build-grid7-64", "do": "build", "graph": "grid7", "nx": 64, "ny": 64, "nz": 64, "walks": 500},
        {"name": "pcg-grid7-64-4rhs", "do": "pcg", "graph": "grid7", "nx": 64, "ny": 64, "nz": 64, "walks": 500,
         "nrhs": 4, "mixed": False},
        # mixed precision on the 1000^2 grid with long-range edges
        {"name": "pcg-longrange-1000-mixed", "do": "pcg", "graph": "longrange", "nx": 1000, "ny": 1000, "nz": 1,
         "walks": 200, "nrhs": 1, "mixed": True},
        # the library's headline: budgets from the network, then the factor built with them
        {"name": "learned-grid27-128", "do": "learned", "graph": "grid27", "nx": 128, "ny": 128, "nz": 128,
         "walks": 300},
        # the paper's own setting: random order, walk reuse, no dropping, Dirichlet Laplacian
        {"name": "reuse-laplace-70", "do": "reuse", "graph": "laplace", "nx": 70, "ny": 70, "nz": 70, "walks": 5},
        # many matrices at once: one walk launch, one block-diagonal solve
        {"name": "batch-rgg-24", "do": "batch", "graph": "rgg", "nmat": 24, "nmax": 100000, "walks": 200,
         "nrhs": 16},
        # the stopping rule of Sec. 5.1 instead of a network
        {"name": "adaptive-grid27-48", "do": "adaptive", "graph": "grid27", "nx": 48, "ny": 48, "nz": 48},
        # a nonsymmetric matrix, ragged
        {"name": "bicgstab-asym-ragged", "do": "bicgstab", "graph": "asym", "nx": 61, "ny": 64, "nz": 67,
         "walks": 300},
        # one training instance of the budget network: features, pilot walks, Adam
        {"name": "train-grid27-48", "do": "train", "graph": "grid27", "nx": 48, "ny": 48, "nz": 48, "epochs": 4},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _edges(rng, lo, hi, flat=False):
    """Grid edges, each its own, odd and even."""
    e = [_log(rng, lo, hi) for _ in range(2 if flat else 3)]
    return {"nx": e[0], "ny": e[1], "nz": 1 if flat else e[2]}


def draw(rng):
    do = rng.choice(["apply", "build", "spmv", "pcg", "pcg", "learned", "reuse", "batch", "adaptive", "bicgstab",
                     "train"])
    if do in ("apply", "build", "pcg"):
        graph = rng.choice(["grid2d", "grid7", "grid27", "longrange"])
        flat = graph in ("grid2d", "longrange")
        hi = {"grid2d": 500, "longrange": 1000, "grid7": 64, "grid27": 56}[graph]
        c = {"do": do, "graph": graph, **_edges(rng, 12 if flat else 8, hi, flat),
             "walks": _log(rng, 20, 200 if graph == "longrange" else 500)}
        if do != "build":
            c["nrhs"] = rng.choice([1, 1, 2, 3, 4, 4, 8, 16])
        if do == "pcg":
            c["mixed"] = rng.random() < 0.5
        return c
    if do == "spmv":
        graph = rng.choice(["grid2d", "grid7", "grid27", "longrange"])
        flat = graph in ("grid2d", "longrange")
        return {"do": do, "graph": graph, **_edges(rng, 16, 1000 if flat else 95, flat),
                "nrhs": rng.choice([1, 2, 3, 4, 7, 8, 16])}
    if do == "learned":
        return {"do": do, "graph": "grid27", **_edges(rng, 12, 96), "walks": _log(rng, 40, 300)}
    if do == "reuse":
        return {"do": do, "graph": "laplace", **_edges(rng, 20, 70), "walks": _log(rng, 3, 20)}
    if do == "batch":
        return {"do": do, "graph": "rgg", "nmat": rng.randint(2, 24), "nmax": _log(rng, 3000, 100000),
                "walks": _log(rng, 50, 200), "nrhs": rng.choice([1, 2, 4, 7, 16])}
    if do == "adaptive":
        return {"do": do, "graph": "grid27", **_edges(rng, 10, 48)}
    if do == "bicgstab":
        return {"do": do, "graph": "asym", **_edges(rng, 12, 64), "walks": _log(rng, 50, 300)}
    return {"do": "train", "graph": "grid27", **_edges(rng, 12, 48), "epochs": rng.randint(1, 4)}


# ---------------------------------------------------------------------------
# Matrices: symmetric pairs (row, col, weight) on the GPU, then CSR.  Every sum
# runs in a fixed order, so that one seed is one matrix.
# ---------------------------------------------------------------------------
OFF = {"grid2d": [(1, 0, 0), (0, 1, 0)], "longrange": [(1, 0, 0), (0, 1, 0)]}
OFF["grid7"] = OFF["laplace"] = OFF["asym"] = [(1, 0, 0), (0, 1, 0), (0, 0, 1)]
OFF["grid27"] = [o for o in ((a, b, c) for a in (-1, 0, 1) for b in (-1, 0, 1) for c in (-1, 0, 1)) if o > (0, 0, 0)]


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _logu(m, lo, hi, gen):
    u = torch.rand(m, generator=gen, device="cuda", dtype=torch.float64)
    return torch.exp(math.log(lo) + u * (math.log(hi) - math.log(lo)))


def _row_sums(n, row, val):
    """Sums of the values of each row (row ascending), left to right."""
    cnt = torch.bincount(row, minlength=n)
    start = torch.cumsum(cnt, 0) - cnt
    pos = torch.arange(row.numel(), device="cuda") - start[row]
    dense = torch.zeros((n, int(cnt.max()) if row.numel() else 1), dtype=torch.float64, device="cuda")
    dense[row, pos] = val
    return dense.sum(1)


def _sorted(n, row, col, val):
    """Entries by (row, column); repeated ones summed in their order."""
    key, at = torch.sort(row * n + col, stable=True)
    val = val[at]
    first = torch.ones_like(key, dtype=torch.bool)
    first[1:] = key[1:] != key[:-1]
    if not bool(first.all()):
        start = torch.nonzero(first).flatten()
        many = torch.diff(start, append=torch.tensor([key.numel()], device="cuda"))
        out = val[start]
        for k in range(1, int(many.max())):
            more = many > k
            out[more] += val[start[more] + k]
        key, val = key[start], out
    return torch.div(key, n, rounding_mode="floor"), key % n, val


def _csr(n, row, col, w, excess, wt=None):
    """A with A_ij = -w and the diagonal row sum + excess(row sums); (rowptr, col, val).  wt: the weights of
    the opposite direction (nonsymmetric matrices: the diagonal covers the larger sum)."""
    row1, col1, w1 = _sorted(n, row, col, w)
    total = _row_sums(n, row1, w1)
    if wt is not None:
        total = torch.maximum(total, _row_sums(n, row1, _sorted(n, row, col, wt)[2]))
    i = torch.arange(n, device="cuda")
    row2, col2, val = _sorted(n, torch.cat([row1, i]), torch.cat([col1, i]), torch.cat([-w1, total + excess(total)]))
    rowptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    rowptr[1:] = torch.cumsum(torch.bincount(row2, minlength=n), 0)
    return rowptr.to(torch.int32), col2.to(torch.int32).contiguous(), val.contiguous()


def _grid_pairs(case):
    """(tail, head, rows of the boundary) of a grid's edges, natural order."""
    s = (case["nx"], case["ny"], case["nz"])
    idx = torch.arange(s[0] * s[1] * s[2], device="cuda").reshape(s)
    tail, head = [], []
    for off in OFF[case["graph"]]:
        a = tuple(slice(max(0, -o), e - max(0, o)) for o, e in zip(off, s))
        b = tuple(slice(max(0, o), e - max(0, -o)) for o, e in zip(off, s))
        tail.append(idx[a].flatten())
        head.append(idx[b].flatten())
    edge = torch.zeros(s, dtype=torch.bool, device="cuda")
    for d in range(3 if s[2] > 1 else 2):
        edge.select(d, 0).fill_(True)
        edge.select(d, s[d] - 1).fill_(True)
    return torch.cat(tail), torch.cat(head), edge.flatten()


def _matrix(case, seed):
    """(rowptr int32, col int32, val float64) of the case's matrix."""
    gen, graph = _gen(seed), case["graph"]
    n = case["nx"] * case["ny"] * case["nz"]
    t, h, edge = _grid_pairs(case)
    f64 = {"dtype": torch.float64, "device": "cuda"}
    skew = None
    if graph in ("grid2d", "laplace"):
        g = torch.ones(t.numel(), **f64)
    elif graph == "longrange":
        src = torch.arange(n, device="cuda").repeat_interleave(2)
        dst = torch.randint(0, n - 1, (2 * n,), generator=gen, device="cuda")
        dst = dst + (dst >= src)
        g = torch.cat([torch.ones(t.numel(), **f64), _logu(2 * n, 0.01, 1.0, gen)])
        t, h = torch.cat([t, src]), torch.cat([h, dst])
    else:
        g = _logu(t.numel(), 0.1, 10.0, gen)
        if graph == "asym":
            skew = torch.rand(t.numel(), generator=gen, **f64) * 1.2 - 0.6
    frac = torch.rand(n, generator=gen, **f64)
    if graph not in ("grid2d", "laplace"):  # the seeded random symmetric ordering
        p = torch.randperm(n, generator=gen, device="cuda")
        t, h = p[t], p[h]
        edge = torch.empty_like(edge).scatter_(0, p, edge)
    excess = {"grid2d": lambda s: edge.double(), "longrange": lambda s: edge.double(),
              "laplace": lambda s: 6.0 - s, "grid7": lambda s: 1e-3 * frac * s, "grid27": lambda s: 1e-4 * s,
              "asym": lambda s: 1e-3 * frac * s}[graph]
    both, back = torch.cat([t, h]), torch.cat([h, t])
    if skew is not None:
        return _csr(n, both, back, torch.cat([g * (1 + skew), g * (1 - skew)]), excess,
                    torch.cat([g * (1 - skew), g * (1 + skew)]))
    return _csr(n, both, back, torch.cat([g, g]), excess)


def _sizes(case):
    """Nodes of each matrix of a batch, over the logarithm from 1000 to nmax."""
    k, hi = case["nmat"], math.log(case["nmax"])
    return [int(round(math.exp(math.log(1000) + (hi - math.log(1000)) * (i + 0.5) / k))) + i for i in range(k)]


def _rgg(case, seed):
    """Random geometric graphs (mean degree 8, conductance 1 / distance, excess 1 % of the row sum on 1 % of
    the rows and on one node of every component without one), as one block-diagonal CSR and its row offsets."""
    gen, f64 = _gen(seed), {"dtype": torch.float64, "device": "cuda"}
    rows, cols, ws, ground, row0 = [], [], [], [], [0]
    for n in _sizes(case):
        r = math.sqrt(8.0 / (math.pi * n))
        m = max(1, int(1.0 / r))
        pts = torch.rand((n, 2), generator=gen, **f64)
        cell2 = torch.clamp((pts * m).long(), max=m - 1)
        cell = cell2[:, 0] * m + cell2[:, 1]
        order = torch.sort(cell, stable=True)[1]
        cnt = torch.bincount(cell, minlength=m * m)
        start = torch.cumsum(cnt, 0) - cnt
        table = torch.full((m * m, int(cnt.max())), -1, dtype=torch.int64, device="cuda")
        slot = torch.arange(n, device="cuda") - start[cell[order]]
        table[cell[order], slot] = order
        i = torch.arange(n, device="cuda")[:, None]
        for a in (-1, 0, 1):
            for b in (-1, 0, 1):
                x, y = cell2[:, 0] + a, cell2[:, 1] + b
                inside = (x >= 0) & (x < m) & (y >= 0) & (y < m)
                j = torch.where(inside[:, None], table[torch.where(inside, x * m + y, 0)], -1)
                d = (pts[:, None, :] - pts[j.clamp(min=0)]).square().sum(2).sqrt()
                ok = (j >= 0) & (j != i) & (d <= r) & (d > 0)
                rows.append((i.expand_as(j)[ok]) + row0[-1])
                cols.append(j[ok] + row0[-1])
                ws.append(1.0 / d[ok])
        pick = torch.randperm(n, generator=gen, device="cuda")[: max(1, round(0.01 * n))]
        ground.append(pick + row0[-1])
        row0.append(row0[-1] + n)
    row, col, w, N = torch.cat(rows), torch.cat(cols), torch.cat(ws), row0[-1]
    lab = torch.arange(N, device="cuda")  # least node of each component
    while True:
        new = lab.scatter_reduce(0, row, lab[col], "amin")
        new = new[new]
        if bool((new == lab).all()):
            break
        lab = new
    has = torch.zeros(N, dtype=torch.bool, device="cuda")
    has[torch.cat(ground)] = True
    comp = torch.zeros(N, dtype=torch.bool, device="cuda")
    comp[lab[has]] = True
    has |= (lab == torch.arange(N, device="cuda")) & ~comp[lab]
    rp, cl, vl = _csr(N, row, col, w, lambda s: torch.where(has, 1e-2 * torch.where(s > 0, s, 1.0), 0.0))
    return rp, cl, vl, row0


def _rhs(n, nrhs, seed):
    return torch.randn((n, nrhs), generator=_gen(seed + 77), device="cuda", dtype=torch.float64)


def _walk_seed(seed):
    return (int(seed) * 2654435761 + 12345) & 0x7FFFFFFF


def _network(ctx, M, seed):
    """A budget network for the case: random hidden layers and an output layer fitted by ridge regression to
    pilot walks of a small grid of the same distribution (rounded, so that it is the same on every run)."""
    A = P.CSR(*_matrix({"graph": "grid27", "nx": 20, "ny": 20, "nz": 20}, 5))
    feat = torch.zeros((A.n, P.RW_FEATURE_STRIDE), device="cuda")
    P.rw_row_features(ctx, A, feat)
    mean, sd, label, has = (torch.zeros(A.n, device="cuda") for _ in range(4))
    P.rw_pilot_stats(ctx, A, 64, 1000, mean, sd, label, has, quantity=2)
    f, y = feat[has > 0].double().cpu(), label[has > 0].double().cpu()
    mu, s = f.mean(0), f.std(0)
    inv = torch.where(s > 1e-9, 1.0 / s, 0.0).float().numpy()
    g = torch.Generator().manual_seed(seed % 1000)
    w1 = torch.randn((64, 16), generator=g, dtype=torch.float64) * math.sqrt(2 / 12)
    w2 = torch.randn((64, 64), generator=g, dtype=torch.float64) * math.sqrt(2 / 64)
    w1[:, 12:] = 0
    x = (f - mu) * torch.from_numpy(inv).double()
    h = torch.relu(torch.relu(x @ w1.T) @ w2.T)
    h = torch.cat([h, torch.ones((h.shape[0], 1), dtype=torch.float64)], 1)
    w3 = torch.linalg.solve(h.T @ h + 1.0 * torch.eye(65, dtype=torch.float64), h.T @ y)
    w3 = torch.round(w3 * 4096) / 4096
    z = torch.zeros(64, dtype=torch.float64)
    params = torch.cat([w1.flatten(), z, w2.flatten(), z, w3]).float().numpy()
    M.set_params(params, np.concatenate([mu.float().numpy(), inv]).astype(np.float32))


# ---------------------------------------------------------------------------
# What the program has in hand
# ---------------------------------------------------------------------------
def prepare(case, seed):
    do = case["do"]
    ctx = P.Context(options=P.rw_options_default(reuse=1 if do == "reuse" else 0))
    st = {"case": case, "ctx": ctx, "seed": _walk_seed(seed), "F": None}
    if do == "batch":
        rp, cl, vl, row0 = _rgg(case, seed)
        st["A"], st["b"] = [], []
        at = rp.cpu().tolist()
        for m in range(case["nmat"]):
            a, e = row0[m], row0[m + 1]
            st["A"].append(P.CSR((rp[a:e + 1] - at[a]).contiguous(), (cl[at[a]:at[e]] - a).contiguous(),
                                 vl[at[a]:at[e]].contiguous()))
            st["b"].append(_rhs(e - a, case["nrhs"], seed + m))
        st["x"] = [torch.zeros_like(b) for b in st["b"]]
        return st
    A = st["A"] = P.CSR(*_matrix(case, seed))
    if do in ("apply", "spmv", "pcg", "bicgstab"):
        st["b"] = _rhs(A.n, case.get("nrhs", 1), seed)
        if do == "bicgstab":
            st["b"] = st["b"][:, 0].contiguous()
        st["x"] = torch.zeros_like(st["b"])
    if do in ("apply", "pcg", "bicgstab"):
        st["F"] = P.rw_build_factor(ctx, A, case["walks"], st["seed"], 1e-3)
    if do == "bicgstab":
        st["AT"] = P.rw_csr_transpose(ctx, A)
        st["FT"] = P.rw_build_factor(ctx, st["AT"], case["walks"], st["seed"] + 1, 1e-3)
    if do == "learned":
        st["M"] = P.rw_mlp_create(ctx, 0)
        _network(ctx, st["M"], seed)
    if do in ("build", "learned", "reuse"):
        st["room"] = _room(case, A.n)
    if do in ("learned", "adaptive"):
        st["budget"] = torch.zeros(A.n, dtype=torch.int32, device="cuda")
    if do == "reuse":
        st["perm"] = torch.empty(A.n, dtype=torch.int32, device="cuda")
    if do == "train":
        st["M"] = P.rw_mlp_create(ctx, seed % 100003)
        st["start"] = st["M"].params()
        st["feat"] = torch.zeros((A.n, P.RW_FEATURE_STRIDE), device="cuda")
        st["stats"] = [torch.zeros(A.n, device="cuda") for _ in range(4)]
    return st


def _room(case, n):
    """The program's own arrays for a factor's entries: the library's belong to the factor, and their number
    is the walks', so they are copied to arrays with room to spare."""
    m = (2 if case["graph"] == "grid27" else 4) * FILL[case["graph"]] * n + 4096
    i32, f64 = {"dtype": torch.int32, "device": "cuda"}, {"dtype": torch.float64, "device": "cuda"}
    return {"y_col": torch.zeros(m, **i32), "y_val": torch.zeros(m, **f64), "yt_col": torch.zeros(m, **i32),
            "yt_val": torch.zeros(m, **f64)}


class Arrays(dict):
    """Views of factors' arrays by name, which keep the factors."""

    def __init__(self, factors, arrays):
        super().__init__(arrays)
        self.factors = factors


def _factor(st, F, **more):
    """Keeps the new factor in place of the one before it; its rows, diagonal, counters and depths."""
    st["F"] = F
    t, d = F.tensors(), F.desc
    for k, room in st["room"].items():
        room[: d.nnz].copy_(t[k])
    same = {k: t[k] for k in ("y_row_ptr", "yt_row_ptr", "d", "walks", "visits", "ground")}
    return Arrays(F, {**more, **same, **st["room"], "levels": [d.fwd_levels, d.bwd_levels], "hops": d.total_hops})


def _drop(st):
    """A program that rebuilds gives the old factor back first."""
    if st["F"] is not None:
        for F in st["F"] if isinstance(st["F"], list) else [st["F"]]:
            F.destroy()
        st["F"] = None


def run(st):
    case, ctx, A = st["case"], st["ctx"], st["A"]
    do = case["do"]
    if do == "apply":
        P.rw_precond_apply(ctx, st["F"], st["b"], st["x"])
        return st["x"]
    if do == "spmv":
        P.rw_spmv(ctx, A, st["b"], st["x"])
        return st["x"]
    if do == "build":
        _drop(st)
        return _factor(st, P.rw_build_factor(ctx, A, case["walks"], st["seed"], 1e-3))
    if do == "pcg":
        prec = P.RW_FP32_MIXED if case["mixed"] else P.RW_FP64
        rc, stats, its, rel = P.pcg_solve(ctx, A, st["F"], st["b"], st["x"], TOL, 500, prec)
        # a mixed solve works in single precision: the program goes on with x in it
        return {"x": st["x"].float() if case["mixed"] else st["x"], "iterations": its}
    if do == "bicgstab":
        rc, stats = P.bicgstab_solve(ctx, A, st["F"], st["FT"], st["b"], st["x"], TOL, 200)
        return {"x": st["x"], "iterations": stats.iterations}
    if do == "learned":
        _drop(st)
        P.rw_budget_predict(ctx, A, st["M"], float(case["walks"]), 20, st["budget"])
        F = P.rw_build_factor_budget(ctx, A, st["budget"], st["seed"], 1e-3)
        return _factor(st, F, budget=st["budget"])
    if do == "reuse":
        _drop(st)
        P.rw_random_permutation(ctx, A.n, st["seed"], st["perm"])
        st["B"] = P.rw_permute_csr(ctx, A, st["perm"])
        return _factor(st, P.rw_build_factor(ctx, st["B"], case["walks"], st["seed"], 0.0))
    if do == "batch":
        _drop(st)
        Fs = P.rw_build_factor_batched(ctx, A, case["walks"], [st["seed"]] * case["nmat"], 1e-3)
        rc, stats, its, rel = P.pcg_solve_batched(ctx, A, Fs, st["b"], st["x"], TOL, 500)
        st["F"] = Fs
        return Arrays(Fs, {"x": st["x"], "iterations": its, "d": [F.tensors()["d"] for F in Fs]})
    if do == "adaptive":
        rounds = P.rw_adaptive_budget(ctx, A, st["seed"], 0.25, 2.5758293035489004, 20, 65535, 12, st["budget"])
        return {"budget": st["budget"], "rounds": rounds}
    if do == "train":
        P.rw_row_features(ctx, A, st["feat"])
        P.rw_pilot_stats(ctx, A, 64, st["seed"], *st["stats"], quantity=2)
        st["M"].set_params(*st["start"])
        losses = P.rw_mlp_train(ctx, st["M"], st["feat"], st["stats"][2], st["stats"][3], case["epochs"], 4096, 2e-3,
                                seed=1)
        params, norm = st["M"].params()
        return {"features": st["feat"], "mean": st["stats"][0], "sd": st["stats"][1], "label": st["stats"][2],
                "has": st["stats"][3], "losses": losses, "params": params, "norm": norm}
    raise ValueError(do)


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    """Inputs read once and outputs written once; a solve reads the matrix and the factor's two halves once an
    iteration (about seven, more for the mixed 27-point and fewer for BiCGSTAB's two halves)."""
    do, g = case["do"], case["graph"]
    n = sum(_sizes(case)) if do == "batch" else case["nx"] * case["ny"] * case["nz"]
    nr = case.get("nrhs", 1)
    a, y = ROW[g] * n, FILL[g] * n
    mat, vec = 12.0 * a + 4.0 * n, 8.0 * n * nr
    fac = 12.0 * y + 16.0 * n  # one half of the factor
    both = 2 * (16.0 * y + 8.0 * n) + 40.0 * n  # Y and Y^T with FP32 copies, D, counters
    it = 7
    if do == "spmv":
        return {"bytes": mat + 2 * vec, "flops": 2.0 * a * nr}
    if do == "apply":
        return {"bytes": 2 * fac + 2 * vec, "flops": 4.0 * y * nr}
    if do in ("pcg", "bicgstab"):
        small = 2.0 / 3.0 if case.get("mixed") else 1.0
        return {"bytes": it * (small * (mat + 2 * fac) + 6 * vec), "flops": it * nr * (2.0 * a + 4.0 * y)}
    if do == "batch":
        return {"bytes": mat + both + it * (mat + 2 * fac + 6 * vec), "flops": it * nr * (2.0 * a + 4.0 * y)}
    if do == "train":
        return {"bytes": mat + 80.0 * n + case["epochs"] * 64.0 * n, "flops": case["epochs"] * 6.0 * 5313 * n}
    if do == "adaptive":
        return {"bytes": mat + 4.0 * n, "flops": 0.0}
    more = {"bytes": 2 * mat, "flops": 0.0} if do == "reuse" else {"bytes": 0.0, "flops": 0.0}
    if do == "learned":
        more["flops"] = 2.0 * 5313 * n
    return {"bytes": mat + both + more["bytes"], "flops": more["flops"]}


# ---------------------------------------------------------------------------
# 64-bit answers
# ---------------------------------------------------------------------------
def _sparse(rp, cl, vl):
    n = rp.numel() - 1
    return torch.sparse_csr_tensor(rp.long(), cl.long(), vl, size=(n, n))


def _diag(rp, cl, vl):
    n = rp.numel() - 1
    row = torch.repeat_interleave(torch.arange(n, device="cuda"), torch.diff(rp.long()))
    return vl[row == cl.long()]


def _cg(rp, cl, vl, b, seg=None, most=6000):
    """A^-1 b by conjugate gradients with the diagonal, to 1e-13; None if it does not get there.  seg: the
    system of each row (block-diagonal A)."""
    A, d = _sparse(rp, cl, vl), _diag(rp, cl, vl)[:, None]
    seg = torch.zeros(b.shape[0], dtype=torch.int64, device="cuda") if seg is None else seg
    k = int(seg.max()) + 1

    def dot(u, v):
        if k == 1:
            return (u * v).sum(0, keepdim=True)
        return torch.zeros((k, b.shape[1]), dtype=b.dtype, device="cuda").index_add_(0, seg, u * v)

    x, r = torch.zeros_like(b), b.clone()
    z = r / d
    p, rho, bb = z.clone(), dot(r, z), dot(b, b)
    for it in range(most):
        q = A @ p
        pq = dot(p, q)
        alpha = torch.where(pq > 0, rho / pq, 0.0)
        x += alpha[seg] * p
        r -= alpha[seg] * q
        if it % 25 == 0 and bool((dot(r, r) <= 1e-26 * bb).all()):
            break
        z = r / d
        new = dot(r, z)
        p = z + torch.where(rho > 0, new / rho, 0.0)[seg] * p
        rho = new
    t = b - A @ x
    return x if bool((dot(t, t) <= 1e-22 * bb).all()) else None


def _bicg(rp, cl, vl, b, most=2000):
    """A^-1 b for a nonsymmetric A (BiCGSTAB with the diagonal, to 1e-13)."""
    A, d = _sparse(rp, cl, vl), _diag(rp, cl, vl)
    x, r = torch.zeros_like(b), b.clone()
    rh, p = r.clone(), r.clone()
    rho, nb = torch.dot(rh, r), float(torch.linalg.norm(b))
    for it in range(most):
        ph = p / d
        v = A @ ph
        alpha = rho / torch.dot(rh, v)
        s = r - alpha * v
        sh = s / d
        t = A @ sh
        om = torch.dot(t, s) / torch.dot(t, t)
        x += alpha * ph + om * sh
        r = s - om * t
        if float(torch.linalg.norm(r)) < 1e-13 * nb:
            break
        new = torch.dot(rh, r)
        p = r + (new / rho) * (alpha / om) * (p - om * v)
        rho = new
    return x if float(torch.linalg.norm(b - A @ x)) < 1e-11 * nb else None


def _features(rp, cl, vl):
    """The twelve features of the header's rw_row_features, in 64 bits."""
    n = rp.numel() - 1
    rp, cl = rp.long(), cl.long()
    row = torch.repeat_interleave(torch.arange(n, device="cuda"), torch.diff(rp))
    off = row != cl
    r, c, w = row[off], cl[off], -vl[off]
    dg = vl[~off]
    deg = torch.bincount(r, minlength=n).double()
    up = torch.bincount(r[c > r], minlength=n).double()
    W = _row_sums(n, r, w)
    exc = _row_sums(n, row, vl) / dg
    ent = -_row_sums(n, r, (w / W[r]) * torch.log(w / W[r]))
    big = torch.zeros(n, dtype=torch.float64, device="cuda").scatter_reduce(0, r, w, "amax")
    Sk = _row_sums(n, r, torch.where(c > r, -w, 0.0))
    mean = lambda v: _row_sums(n, r, v[c]) / deg  # noqa: E731
    key = row * n + cl
    past = torch.searchsorted(key, c * n + r, right=True)  # entries of row c up to column r
    two = _row_sums(n, r, torch.where(c > r, (rp[c + 1] - past - 1).double(), 0.0))
    k = torch.arange(n, device="cuda").double()
    f = torch.zeros((n, P.RW_FEATURE_STRIDE), dtype=torch.float64, device="cuda")
    cols = [torch.log1p(deg), up / deg, (deg - up) / deg, exc, -Sk / dg, ent, big / W, k / (n - 1), mean(exc),
            torch.log1p(mean(deg)), torch.log1p(two), torch.log(dg)]
    for i, v in enumerate(cols):
        f[:, i] = v
    return f


def exact(case, seed):
    """What has a value apart from the random draws: products, solutions and features.  A factor's entries are
    estimates of a random game and have none of their own (apply uses such a factor, and has none either)."""
    do = case["do"]
    if do == "spmv":
        rp, cl, vl = _matrix(case, seed)
        return _sparse(rp, cl, vl) @ _rhs(rp.numel() - 1, case["nrhs"], seed)
    if do == "pcg":
        rp, cl, vl = _matrix(case, seed)
        return {"x": _cg(rp, cl, vl, _rhs(rp.numel() - 1, case["nrhs"], seed)), "iterations": None}
    if do == "bicgstab":
        rp, cl, vl = _matrix(case, seed)
        return {"x": _bicg(rp, cl, vl, _rhs(rp.numel() - 1, 1, seed)[:, 0].contiguous()), "iterations": None}
    if do == "batch":
        rp, cl, vl, row0 = _rgg(case, seed)
        size = torch.diff(torch.tensor(row0, device="cuda"))
        seg = torch.repeat_interleave(torch.arange(case["nmat"], device="cuda"), size)
        b = torch.cat([_rhs(row0[m + 1] - row0[m], case["nrhs"], seed + m) for m in range(case["nmat"])])
        x = _cg(rp, cl, vl, b, seg)
        return {"x": None if x is None else list(torch.split(x, size.tolist())), "iterations": None, "d": None}
    if do == "train":
        return {"features": _features(*_matrix(case, seed))}
    return None
