"""Lines of the autotuner's cache: one written for earlier kernels or for a matrix
of other row lengths is not installed."""
import json

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


def _keys(path):
    return [json.loads(line)["key"] for line in open(path).read().strip().splitlines()]


def test_lines_of_earlier_kernels_are_not_installed(P, tmp_path):
    A = P.CSR.from_host(W.grid2d_5pt(24, 20))
    c = P.Context()
    F = P.rw_build_factor(c, A, 40, 2, 1e-3)
    now = str(tmp_path / "now.jsonl")
    P.rw_autotune(c, A, F, 2, P.RW_FP64, now)
    # the same problem as the first format of the cache named it
    key = "|".join(p for p in _keys(now)[0].split("|") if not p.startswith(("gen", "apr")))
    old = tmp_path / "old.jsonl"
    old.write_text('{"key":"%s","solve_mode":1,"solve_mode_bwd":-1,"thin_cluster":0,"thin_flags":0,"thin_lanes":8,'
                   '"wide_slices":16,"solve_blocks_per_sm":1,"cluster_width":0,"spmv_slices":16,"precond_ms":1.0,'
                   '"spmv_ms":1.0}\n' % key)
    _, ms = P.rw_autotune(c, A, F, 2, P.RW_FP64, str(old))
    assert ms[0] > 0 and ms[1] > 0  # timed, not read
    _, ms = P.rw_autotune(c, A, F, 2, P.RW_FP64, str(old))
    assert ms == (0.0, 0.0)  # the line just written
    F.destroy()
    c.close()


def test_row_lengths_of_the_matrix_are_told_apart(P, tmp_path):
    # one factor, two matrices of its size: Y's entries and levels are the same, A's rows are not
    n = 500
    rng = np.random.default_rng(1)
    a, b = np.triu_indices(n, 1)
    keep = rng.random(a.size) < 0.1
    dense = W.assemble(n, a[keep], b[keep], np.ones(keep.sum()), 1.0)
    path = W.tridiag(n)
    c = P.Context()
    F = P.rw_build_factor(c, P.CSR.from_host(path), 20, 2, 1e-3)
    cache = str(tmp_path / "tune.jsonl")
    for A in (path, dense):
        _, ms = P.rw_autotune(c, P.CSR.from_host(A), F, 1, P.RW_FP64, cache)
        assert ms[1] > 0
    assert len(set(_keys(cache))) == 2
    F.destroy()
    c.close()
