"""The row solves of the widest levels (four rows of a level per warp) against
the one-row-per-warp solve and substitution: levels of widths that leave every
remainder, rows longer than one pass of a group, narrow levels behind them."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_math_0609672_gb300 as P
    from paper_math_0609672_gb300 import _build
    _build.build()
    return P


def _cliques(sizes, path, seed, hub=False):
    """Disjoint cliques (level k holds the k-th node of each) and a path; hub: its last node neighbours all the
    cliques' nodes (one row before the wide levels in one of the two directions)."""
    rng = np.random.default_rng(seed)
    ei, ej, base = [], [], 0
    for m in sizes:
        a, b = np.triu_indices(m, 1)
        ei.append(base + a)
        ej.append(base + b)
        base += m
    ei.append(base + np.arange(path - 1))
    ej.append(base + np.arange(1, path))
    if hub:
        ei.append(np.arange(base))
        ej.append(np.full(base, base + path - 1))
    ei, ej, n = np.concatenate(ei), np.concatenate(ej), base + path
    g = np.exp(rng.uniform(-1, 1, ei.size))
    return W.assemble(n, ei, ej, g, 1e-2 * W.conductance_sums(n, ei, ej, g))


# widths around the 2432 rows from which levels are packed: with the path one row more
CASES = {"short": [4] * 2431 + [3], "below": [5] * 2430, "one": [7] * 2432 + [5] * 2, "two": [6] * 2433,
         "hub": [7] * 2432 + [5] * 2, "long": [40] * 300 + [12] * 1800 + [5] * 500}


@pytest.mark.parametrize("name", CASES)
def test_packed_rows_match_substitution(P, name):
    import torch
    A = _cliques(CASES[name], 70, 5, name == "hub")
    packed, single = P.Context(), P.Context(options=P.rw_options_default(solve_mode=1))
    try:
        F = P.rw_build_factor(packed, P.CSR.from_host(A), 40, 3, 0.0)
        G = P.rw_build_factor(single, P.CSR.from_host(A), 40, 3, 0.0)
        t = {k: v.cpu().numpy() for k, v in F.tensors().items()}
        for nrhs in (1, 2, 3, 4, 7):
            r = np.random.default_rng(nrhs).standard_normal((A.n, nrhs))
            z, zs = (torch.empty((A.n, nrhs), dtype=torch.float64, device="cuda") for _ in range(2))
            P.rw_precond_apply(packed, F, torch.as_tensor(r).cuda(), z)
            P.rw_precond_apply(single, G, torch.as_tensor(r).cuda(), zs)
            z, zs = z.cpu().numpy(), zs.cpu().numpy()
            # M-matrix factors: both sides lose at most a few units of each row's length
            assert np.abs(z - zs).max() / np.abs(zs).max() < 1e-12
            if nrhs == 3:  # z solves Y^T D Y z = r
                y = _matvec(t["y_row_ptr"], t["y_col"], t["y_val"], z)
                back = _matvec(t["yt_row_ptr"], t["yt_col"], t["yt_val"], y * t["d"][:, None])
                assert np.abs(back - r).max() / np.abs(r).max() < 1e-11
        F.destroy()
        G.destroy()
    finally:
        packed.close()
        single.close()


def _matvec(rp, col, val, x):
    """(unit diagonal + the stored off-diagonal entries) x."""
    rows = np.repeat(np.arange(len(rp) - 1), np.diff(rp))
    out = x.copy()
    np.add.at(out, rows, val[:, None] * x[col])
    return out


@pytest.mark.parametrize("name", ["two", "long"])
def test_packed_rows_in_single_precision(P, name):
    # the FP32 solve takes the iterations of the FP64 one (within one) and reaches the tolerance
    import torch
    A = _cliques(CASES[name], 70, 6)
    c = P.Context()
    try:
        dA = P.CSR.from_host(A)
        F = P.rw_build_factor(c, dA, 40, 3, 0.0)
        for nrhs in (1, 3, 8):
            b = torch.as_tensor(np.random.default_rng(nrhs).standard_normal((A.n, nrhs))).cuda()
            its = {}
            for prec in (P.RW_FP64, P.RW_FP32_MIXED):
                x = torch.empty_like(b)
                rc, st, it, rel = P.pcg_solve(c, dA, F, b, x, 1e-6, 200, prec)
                assert rc == 0 and (rel < 1e-6).all()
                its[prec] = it
            assert (np.abs(its[P.RW_FP64] - its[P.RW_FP32_MIXED]) <= 1).all()
        F.destroy()
    finally:
        c.close()


@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("nrhs", [2, 4, 5, 8, 9, 12, 13, 16])
def test_unaligned_vectors(P, nrhs, offset):
    # vectors that start 8 bytes after a 16-byte boundary
    import torch
    A = W.grid3d(11, 10, 9, 7, np.random.default_rng(4), excess_frac=1e-3)
    for mode in (0, 1, 2):
        c = P.Context(options=P.rw_options_default(solve_mode=mode))
        try:
            F = P.rw_build_factor(c, P.CSR.from_host(A), 60, 3, 0.0)
            r = np.random.default_rng(nrhs).standard_normal((A.n, nrhs))
            store = torch.empty(A.n * nrhs + 1, dtype=torch.float64, device="cuda")
            z = store[offset:offset + A.n * nrhs].view(A.n, nrhs)
            P.rw_precond_apply(c, F, torch.as_tensor(r).cuda(), z)
            t = {k: v.cpu().numpy() for k, v in F.tensors().items()}
            y = _matvec(t["y_row_ptr"], t["y_col"], t["y_val"], z.cpu().numpy())
            back = _matvec(t["yt_row_ptr"], t["yt_col"], t["yt_val"], y * t["d"][:, None])
            assert np.abs(back - r).max() / np.abs(r).max() < 1e-11
            F.destroy()
        finally:
            c.close()
