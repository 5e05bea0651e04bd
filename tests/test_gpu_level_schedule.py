"""The level schedule (solve_mode 0) takes narrow levels in blocks, as the default
does: a path of as many levels as rows is solved much faster than one hand-off
per level, in both directions, and mixed with wide levels it gives the same."""
import time

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


def _apply(P, c, F, r, reps):
    """The solution and the least seconds of a call."""
    import torch
    z = torch.empty_like(r)
    best = 1e9
    for _ in range(reps):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        P.rw_precond_apply(c, F, r, z)
        best = min(best, time.perf_counter() - t0)
    return z, best


@pytest.mark.parametrize("cluster_width", [0, 256])
def test_narrow_levels_of_the_level_schedule(P, cluster_width):
    import torch
    A = W.tridiag(3000, diag=2.001)
    r = torch.as_tensor(np.random.default_rng(0).standard_normal((A.n, 4))).cuda()
    level = P.Context(options=P.rw_options_default(solve_mode=0, cluster_width=cluster_width))
    rows = P.Context(options=P.rw_options_default(solve_mode=1))
    F = P.rw_build_factor(level, P.CSR.from_host(A), 50, 3, 0.0)
    assert F.desc.fwd_levels == F.desc.bwd_levels == 3000
    z, t_level = _apply(P, level, F, r, 5)
    zr, t_rows = _apply(P, rows, F, r, 5)
    assert (z - zr).abs().max() / zr.abs().max() < 1e-12
    assert t_level < 0.25 * t_rows, (t_level, t_rows)
    F.destroy()
    level.close()
    rows.close()


@pytest.mark.parametrize("wide_slices", [-1, 0, 4])
@pytest.mark.parametrize("cluster_width", [0, 400])
def test_blocks_between_levels(P, wide_slices, cluster_width):
    # narrow, wide, narrow again: the barrier words serve both kinds of launches in turn
    import torch
    from test_gpu_blocks import _matrix, _solve
    A = _matrix("mixed")
    c = P.Context(options=P.rw_options_default(solve_mode=0, wide_slices=wide_slices, cluster_width=cluster_width))
    F = P.rw_build_factor(c, P.CSR.from_host(A), 60, 3, 0.0)
    t = {k: v.cpu().numpy() for k, v in F.tensors().items()}
    for nrhs in (1, 3, 16):
        r = np.random.default_rng(nrhs).standard_normal((A.n, nrhs))
        ref = _solve(t, r)
        z = torch.empty((A.n, nrhs), dtype=torch.float64, device="cuda")
        for _ in range(3):
            P.rw_precond_apply(c, F, torch.as_tensor(r).cuda(), z)
            assert np.abs(z.cpu().numpy() - ref).max() / np.abs(ref).max() < 1e-12
    F.destroy()
    c.close()
