"""The step cap in adaptive counts: a walk that only the run-ahead would use may
exceed it, one that a decision uses may not."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu

RW_ERR_WALK_CAP = -3
DELTA, Z, MOST, DECISIONS = 0.3, 2.0, 400, 8


def _dense(seed, n=480):
    """A random graph of 12 neighbours a node: walk lengths close to geometric."""
    rng = np.random.default_rng(seed)
    ei, ej, g = W._dedup_edges(rng.integers(0, n, 6 * n), rng.integers(0, n, 6 * n), np.ones(6 * n))
    s = W.conductance_sums(n, ei, ej, g)
    return W.assemble(n, ei, ej, g, np.where(s > 0, 2e-2 * s, 1.0))


def _longest(A, counts, seed):
    return int(oracle.build_factor(A, counts.astype(np.uint32), seed, 0.0, records=True)["rec_len"].max())


@pytest.mark.parametrize("seed,ahead", [(2, 100), (3, 25), (7, 400), (10, 100)])
def test_cap_counts_the_walks_that_decide(seed, ahead):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_math_0609672_gb300 as P
    from paper_math_0609672_gb300 import _build
    _build.build()
    A = _dense(seed)
    ref, rounds = oracle.adaptive_budget(A, seed, DELTA, Z, min_walks=20, max_walks=MOST, max_rounds=DECISIONS)
    cap = _longest(A, ref, seed)
    # the first rows' run of 2 (Z / DELTA)^2 walks in the first round holds a longer one
    first = np.where(np.arange(A.n) < A.n // 16, np.ceil(2 * (Z / DELTA) ** 2), 0)
    assert _longest(A, np.maximum(ref, first), seed) > cap
    dA = P.CSR.from_host(A)
    b = torch.zeros(A.n, dtype=torch.int32, device="cuda")
    for steps, ok in ((cap, True), (cap - 1, False)):
        c = P.Context(options=P.rw_options_default(max_steps=steps, adapt_ahead=ahead))
        try:
            if ok:
                r = P.rw_adaptive_budget(c, dA, seed, DELTA, Z, 20, MOST, DECISIONS, b)
                assert r == rounds and np.array_equal(b.cpu().numpy().view(np.uint32), ref)
            else:
                with pytest.raises(P.RwError) as e:
                    P.rw_adaptive_budget(c, dA, seed, DELTA, Z, 20, MOST, DECISIONS, b)
                assert e.value.code == RW_ERR_WALK_CAP
        finally:
            c.close()
