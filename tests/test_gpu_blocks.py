"""The solves' blocks of narrow levels against substitution on the host: block
and stretch edges, rows longer than a thread block's share, every number of
right-hand sides, FP64 and (through PCG) FP32."""
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


def _hub(n, rng):
    """A path whose first node neighbours every other: rows of Y^T as long as the matrix."""
    ei = np.concatenate([np.arange(n - 1), np.zeros(n - 2, np.int64)])
    ej = np.concatenate([np.arange(1, n), np.arange(2, n)])
    g = np.exp(rng.uniform(-1, 1, ei.size))
    return W.assemble(n, ei, ej, g, 1e-2 * W.conductance_sums(n, ei, ej, g))


def _mixed(rng):
    """Narrow levels, wide ones, narrow ones again: a path, 600 leaves on it, a path on the leaves."""
    a, w, c = 300, 600, 290
    ei = np.concatenate([np.arange(a - 1), rng.integers(0, a, w), [a], np.arange(a + w, a + w + c - 1),
                         a + rng.integers(0, w, c)])
    ej = np.concatenate([np.arange(1, a), a + np.arange(w), [a + w], np.arange(a + w + 1, a + w + c),
                         a + w + np.arange(c)])
    ei, ej, g = W._dedup_edges(ei, ej, np.exp(rng.uniform(-1, 1, ei.size)))
    n = a + w + c
    return W.assemble(n, ei, ej, g, 1e-2 * W.conductance_sums(n, ei, ej, g))


def _matrix(name):
    rng = np.random.default_rng(8)
    if name.startswith("path"):
        return W.tridiag(int(name[4:]))
    return {"hub": lambda: _hub(1500, rng), "mixed": lambda: _mixed(rng), "grid": lambda: W.grid2d_5pt(37, 23),
            "grid27": lambda: W.grid3d(9, 8, 10, 27, rng, excess_frac=1e-3)}[name]()


def _solve(t, r):
    """(Y^T D Y)^-1 r by substitution."""
    w = r.copy()
    rp, cl, v = t["yt_row_ptr"], t["yt_col"], t["yt_val"]
    n = len(r)
    for i in range(n - 1, -1, -1):
        s, e = rp[i], rp[i + 1]
        w[i] -= v[s:e] @ w[cl[s:e]]
    w /= t["d"][:, None]
    rp, cl, v = t["y_row_ptr"], t["y_col"], t["y_val"]
    for i in range(n):
        s, e = rp[i], rp[i + 1]
        w[i] -= v[s:e] @ w[cl[s:e]]
    return w


@pytest.mark.parametrize("name", ["path15", "path17", "path255", "path256", "path257", "path513", "hub", "mixed",
                                  "grid", "grid27"])
def test_blocks_match_substitution(P, name):
    import torch
    A = _matrix(name)
    for mode, slices in ((2, -1), (2, 4), (1, -1), (0, -1)):
        c = P.Context(options=P.rw_options_default(solve_mode=mode, wide_slices=slices))
        try:
            F = P.rw_build_factor(c, P.CSR.from_host(A), 60, 3, 0.0)
            t = {k: v.cpu().numpy() for k, v in F.tensors().items()}
            lp, order = t["fwd_level_ptr"], t["fwd_order"]
            assert all((np.diff(order[a:b]) > 0).all() for a, b in zip(lp[:-1], lp[1:]))
            for nrhs in (1, 2, 3, 4, 8, 11, 16):
                r = np.random.default_rng(nrhs).standard_normal((A.n, nrhs))
                ref = _solve(t, r)
                z = torch.empty((A.n, nrhs), dtype=torch.float64, device="cuda")
                P.rw_precond_apply(c, F, torch.as_tensor(r).cuda(), z)
                # an M-matrix factor: both sides lose at most a few units of each row's length
                err = np.abs(z.cpu().numpy() - ref).max() / np.abs(ref).max()
                assert err < 1e-12, (mode, nrhs, err)
            F.destroy()
        finally:
            c.close()


@pytest.mark.parametrize("name", ["path257", "hub", "mixed", "grid27"])
def test_blocks_in_single_precision(P, name):
    # the FP32 solve takes the iterations of the FP64 one (within one) and reaches the tolerance
    import torch
    A = _matrix(name)
    c = P.Context()
    try:
        dA = P.CSR.from_host(A)
        F = P.rw_build_factor(c, dA, 60, 3, 0.0)
        for nrhs in (1, 3, 16):
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
