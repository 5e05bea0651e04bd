"""Explicit options of the row solves choose the kernel that they name, also for the
backward solve of one FP32 right-hand side, which takes lane groups by default."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def _solve(P, options, dA, b):
    """Names of the kernels of a mixed-precision solve."""
    import torch
    from torch.profiler import ProfilerActivity, profile
    c = P.Context(options=P.rw_options_default(**options))
    F = P.rw_build_factor(c, dA, 40, 3, 1e-3)
    x = torch.empty_like(b)
    for _ in range(4):  # (a session now and then records nothing)
        torch.cuda.synchronize()
        with profile(activities=[ProfilerActivity.CUDA]) as prof:
            rc, _, _, rel = P.pcg_solve(c, dA, F, b, x, 1e-6, 100, P.RW_FP32_MIXED)
            torch.cuda.synchronize()
        assert rc == 0 and (rel < 1e-6).all()
        names = {e.key for e in prof.key_averages() if "k_" in e.key}
        if names:
            break
    F.destroy()
    c.close()
    if not names:
        pytest.skip("the profiler records no kernels here")
    return names


@pytest.mark.parametrize("mode", [1, 2])
def test_options_choose_the_row_kernel(mode):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_math_0609672_gb300 as P
    from paper_math_0609672_gb300 import _build
    _build.build()
    A = W.grid3d(20, 21, 19, 27, np.random.default_rng(3), excess_frac=1e-2)
    dA = P.CSR.from_host(A)
    b = torch.as_tensor(np.random.default_rng(0).standard_normal((A.n, 1))).cuda()
    seen = {}
    for blocks in (0, 1, 2):
        names = _solve(P, {"solve_mode": mode, "solve_blocks_per_sm": blocks}, dA, b)
        seen[blocks] = {k for k in names if "k_rows" in k}
        assert any("k_rows_vec<float, 1" in k for k in seen[blocks]), names
    assert any("k_rows<float, 1>" in k for k in seen[0])
    assert not any("k_rows<" in k for k in seen[1] | seen[2]), seen
    assert any("k_rows_vec<float, 1, 2>" in k for k in seen[2]), seen
    names = _solve(P, {"solve_mode": mode, "wide_slices": 32}, dA, b)
    assert not any("k_rows_vec" in k for k in names)
