"""The walk kernels' rounds of four hops and their teams for a warp's last
walks, against the oracle (bit-exact): few walks, every node layout without
the largest class, and the step cap at each place in a round."""
import numpy as np
import pytest

import oracle
import workloads as W

from test_gpu_factor import assert_factor_equal, gpu_factor

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


def _classes(seed, n=600):
    """Nodes of one to eight groups of four slots (degree 0..31), none larger."""
    rng = np.random.default_rng(seed)
    deg = np.zeros(n, np.int64)
    ei, ej = [], []
    want = rng.integers(2, 32, n)
    for i in range(n):
        for j in rng.permutation(n)[: 3 * want[i]]:
            if deg[i] >= want[i]:
                break
            if j != i and deg[j] < 31:
                ei.append(min(i, j))
                ej.append(max(i, j))
                deg[i] += 1
                deg[j] += 1
    ei, ej, g = W._dedup_edges(ei, ej, np.exp(rng.uniform(np.log(0.1), np.log(10.0), len(ei))))
    rs = W.conductance_sums(n, ei, ej, g)
    A = W.assemble(n, ei, ej, g, np.where(rs > 0, 1e-2 * rs, 1.0))
    ng = (np.diff(A.rowptr) + 3) // 4
    assert ng.max() == 8 and len(np.unique(ng)) >= 7
    return A


def _matrix(name):
    rng = np.random.default_rng(5)
    return {"path": lambda: W.tridiag(6), "two": lambda: W.tridiag(2, diag=1.01),
            "grid": lambda: W.grid3d(9, 7, 5, 7, rng, excess_frac_hi=1e-2),
            "grid27": lambda: W.grid3d(6, 7, 5, 27, rng, excess_frac=1e-3),
            "classes": lambda: _classes(3)}[name]()


@pytest.mark.parametrize("reuse", [0, 1])
@pytest.mark.parametrize("name,walks", [("two", 1), ("path", 1), ("path", 7), ("grid", 1), ("grid27", 3),
                                        ("classes", 1), ("classes", 40)])
def test_last_walks_bit_exact(P, name, walks, reuse):
    A = _matrix(name)
    c = P.Context(options=P.rw_options_default(keep_records=1, reuse=reuse))
    try:
        t = gpu_factor(P, c, A, walks, 77, 1e-3)
        assert_factor_equal(t, oracle.build_factor(A, walks, 77, 1e-3, reuse=bool(reuse), records=True))
    finally:
        c.close()


@pytest.mark.parametrize("kind", ["plain", "reuse", "batched"])
@pytest.mark.parametrize("seed", range(4))
def test_step_cap_is_exact(P, kind, seed):
    # the longest walk may take exactly max_steps hops; with one less the build reports the cap
    A = _matrix("grid27" if seed % 2 else "grid")
    ref = oracle.build_factor(A, 2, seed, 1e-3, reuse=kind == "reuse", records=True)
    longest = int(ref["rec_len"].max())
    dA = P.CSR.from_host(A)
    for cap, ok in ((longest, True), (longest - 1, False)):
        c = P.Context(options=P.rw_options_default(max_steps=cap, reuse=1 if kind == "reuse" else 0))
        try:
            if kind == "batched":
                build = lambda: P.rw_build_factor_batched(c, [dA], 2, [seed], 1e-3)[0]  # noqa: E731
            else:
                build = lambda: P.rw_build_factor(c, dA, 2, seed, 1e-3)  # noqa: E731
            if ok:
                F = build()
                assert F.desc.total_hops == int(ref["hops"].sum())
                F.destroy()
            else:
                with pytest.raises(P.RwError) as e:
                    build()
                assert e.value.code == -3
        finally:
            c.close()


def test_batched_last_walks_bit_exact(P):
    # a warp's last walks belong to different matrices, some without a live walk
    As = [_matrix(n) for n in ("path", "grid", "grid27", "classes", "two")]
    c = P.Context()
    try:
        Fs = P.rw_build_factor_batched(c, [P.CSR.from_host(A) for A in As], 2, list(range(5)), 1e-3)
        for m, (A, F) in enumerate(zip(As, Fs)):
            t = {k: v.cpu().numpy() for k, v in F.tensors().items()}
            t["total_hops"] = int(F.desc.total_hops)
            assert_factor_equal(t, oracle.build_factor(A, 2, m, 1e-3, matrix_index=m), records=False)
            F.destroy()
    finally:
        c.close()
