"""A non-finite value reaches the rows that depend on it and no others: the
solves against substitution on the host over the stored entries, and a batch in
which one matrix' single-precision residual overflows."""
import numpy as np
import pytest

import workloads as W

from test_gpu_blocks import _solve

pytestmark = pytest.mark.gpu

RW_ERR_BREAKDOWN = -6


@pytest.fixture(scope="module")
def P():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_math_0609672_gb300 as P
    from paper_math_0609672_gb300 import _build
    _build.build()
    return P


def _disjoint():
    """Three components whose rows share the blocks of narrow levels: two grids and a path, interleaved."""
    parts = [W.grid2d_5pt(13, 11), W.tridiag(150, diag=2.01), W.grid2d_5pt(7, 19)]
    ei, ej, g, ex, at = [], [], [], [], 0
    for A in parts:
        rows = np.repeat(np.arange(A.n), np.diff(A.rowptr))
        up = A.col > rows
        ei.append(rows[up] + at)
        ej.append(A.col[up] + at)
        g.append(-A.val[up])
        ex.append(np.bincount(rows, weights=A.val, minlength=A.n))
        at += A.n
    ei, ej, g = np.concatenate(ei), np.concatenate(ej), np.concatenate(g)
    rank = np.argsort(np.argsort(np.concatenate([(np.arange(A.n) + 0.5) / A.n for A in parts]), kind="stable"))
    a, b = rank[ei], rank[ej]
    excess = np.empty(at)
    excess[rank] = np.maximum(np.concatenate(ex), 0.0)
    a, b, g = W._dedup_edges(a, b, g)
    return W.assemble(at, a, b, g, excess), [rank[:parts[0].n], rank[parts[0].n:parts[0].n + parts[1].n],
                                             rank[parts[0].n + parts[1].n:]]


@pytest.mark.parametrize("mode", [0, 1, 2])
@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_nonfinite_values_stay_with_their_dependents(P, mode, bad):
    import torch
    A, parts = _disjoint()
    c = P.Context(options=P.rw_options_default(solve_mode=mode))
    try:
        F = P.rw_build_factor(c, P.CSR.from_host(A), 60, 3, 0.0)
        t = {k: v.cpu().numpy() for k, v in F.tensors().items()}
        for nrhs in (1, 2, 3, 4, 8, 16):
            r = np.random.default_rng(nrhs).standard_normal((A.n, nrhs))
            for i, p in enumerate(parts):
                if i != 1:
                    r[p[len(p) // 2], nrhs - 1] = bad
            with np.errstate(invalid="ignore"):
                ref = _solve(t, r)
            assert np.isfinite(ref[parts[1]]).all() and not np.isfinite(ref).all()
            z = torch.empty((A.n, nrhs), dtype=torch.float64, device="cuda")
            P.rw_precond_apply(c, F, torch.as_tensor(r).cuda(), z)
            z = z.cpu().numpy()
            fin = np.isfinite(ref)
            assert np.array_equal(np.isfinite(z), fin), nrhs
            assert np.array_equal(z[~fin], ref[~fin], equal_nan=True), nrhs
            assert np.abs(z[fin] - ref[fin]).max() / np.abs(ref[fin]).max() < 1e-12
        F.destroy()
    finally:
        c.close()


def test_overflow_of_one_matrix_leaves_the_others(P):
    # b of the first matrix is finite in FP64 and beyond the FP32 range
    import torch
    As = [W.grid2d_5pt(14, 12), W.tridiag(180, diag=2.01), W.grid2d_5pt(11, 16)]
    c = P.Context()
    try:
        dAs = [P.CSR.from_host(A) for A in As]
        Fs = P.rw_build_factor_batched(c, dAs, 60, [1, 2, 3], 0.0)
        B = P.Batch(c, dAs, Fs)
        for nrhs in (1, 4):
            bs = [np.random.default_rng(m).standard_normal((A.n, nrhs)) for m, A in enumerate(As)]
            ref = [torch.zeros((A.n, nrhs), dtype=torch.float64, device="cuda") for A in As]
            rc, _, _, _ = P.pcg_solve_batch(c, B, [torch.as_tensor(b).cuda() for b in bs], ref, 1e-6, 200,
                                              P.RW_FP32_MIXED)
            assert rc == 0
            bs[0] *= 1e60
            xs = [torch.zeros((A.n, nrhs), dtype=torch.float64, device="cuda") for A in As]
            with pytest.raises(P.RwError) as e:
                P.pcg_solve_batch(c, B, [torch.as_tensor(b).cuda() for b in bs], xs, 1e-6, 200, P.RW_FP32_MIXED)
            assert e.value.code == RW_ERR_BREAKDOWN
            for m in (1, 2):  # the same iterations, the same bits
                assert torch.equal(xs[m], ref[m])
        B.destroy()
        for F in Fs:
            F.destroy()
    finally:
        c.close()
