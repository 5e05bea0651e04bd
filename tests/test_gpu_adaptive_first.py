"""The first rows of an adaptive count run further in the first launch round
than the others: the counts and the decision count stay the oracle's, with a
sixteenth of the rows at the edge of one row, at the cap of walks and where the
further run is shorter than the ordinary one."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu

# nodes, margin, z, least and most walks, decisions
CASES = [(15, 1, 0.2, 2.0, 4, 4000, 8), (16, 1, 0.2, 2.0, 4, 4000, 8), (40, 50, 0.25, 2.576, 20, 65535, 12),
         (40, 50, 0.05, 2.576, 8, 300, 6), (30, 31, 0.9, 1.0, 30, 4000, 5), (150, 130, 0.3, 2.0, 6, 4000, 1)]


@pytest.mark.parametrize("nx,ny,delta,z,least,most,decisions", CASES)
def test_first_rows_keep_the_counts(nx, ny, delta, z, least, most, decisions):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_math_0609672_gb300 as P
    from paper_math_0609672_gb300 import _build
    _build.build()
    A = W.grid2d_5pt(nx, ny)
    c = P.Context()
    try:
        b = torch.zeros(A.n, dtype=torch.int32, device="cuda")
        r = P.rw_adaptive_budget(c, P.CSR.from_host(A), 12, delta, z, least, most, decisions, b)
        ref, rr = oracle.adaptive_budget(A, 12, delta, z, min_walks=least, max_walks=most, max_rounds=decisions)
        assert r == rr and np.array_equal(b.cpu().numpy().view(np.uint32), ref)
    finally:
        c.close()
