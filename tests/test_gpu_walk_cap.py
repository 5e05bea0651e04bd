"""A walk that reaches the step cap while the last walks of other warps run in
teams of lanes: the call ends with RW_ERR_WALK_CAP and the context stays usable."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

RW_ERR_WALK_CAP = -3


@pytest.fixture(scope="module")
def P():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_math_0609672_gb300 as P
    from paper_math_0609672_gb300 import _build
    _build.build()
    return P


def _paths(grounded, free, length):
    """Paths of `length` nodes: `grounded` ones end at ground (their first walks take about length^2 hops), `free`
    ones have no ground (their first walks run to the step cap)."""
    k = grounded + free
    i = (np.arange(k)[:, None] * length + np.arange(length - 1)).ravel()
    excess = np.zeros(k * length)
    excess[(np.arange(grounded) + 1) * length - 1] = 1.0
    return W.assemble(k * length, i, i + 1, np.ones(i.size), excess)


@pytest.mark.parametrize("kind", ["plain", "reuse", "batched", "adaptive"])
@pytest.mark.parametrize("max_steps", [4097, 8194, 30000])
def test_cap_stops_the_teams(P, kind, max_steps):
    import torch
    A, B = _paths(40, 3, 250), _paths(40, 0, 12)
    dA, dB = P.CSR.from_host(A), P.CSR.from_host(B)
    c = P.Context(options=P.rw_options_default(max_steps=max_steps, reuse=1 if kind == "reuse" else 0))
    try:
        with pytest.raises(P.RwError) as e:
            if kind == "batched":
                P.rw_build_factor_batched(c, [dB, dA, dA], 2, [1, 2, 3], 0.0)
            elif kind == "adaptive":
                P.rw_adaptive_budget(c, dA, 3, 0.5, 2.576, 20, 100, 4,
                                     torch.zeros(A.n, dtype=torch.int32, device="cuda"))
            else:
                P.rw_build_factor(c, dA, 2, 3, 0.0)
        assert e.value.code == RW_ERR_WALK_CAP
        F = P.rw_build_factor(c, dB, 5, 3, 0.0)  # its walks end at ground long before
        assert F.desc.total_walks == 5 * F.desc.n_walk_rows
        F.destroy()
    finally:
        c.close()
