"""SpMV of long rows (a warp per row throughout): every average length around the
lines at which the form changes, its residual and dot products through PCG, and
the time per entry, which must not grow with the rows' length."""
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


def _random(P, n, length, rng):
    """(device CSR, rows, columns, values) of n rows of `length` random entries each."""
    import torch
    rp = (np.arange(n + 1) * length).astype(np.int32)
    col = rng.integers(0, n, rp[-1]).astype(np.int32)
    val = rng.standard_normal(rp[-1])
    return P.CSR(*(torch.as_tensor(v).cuda() for v in (rp, col, val))), np.repeat(np.arange(n), length), col, val


# 512 / max(4, right-hand sides rounded up to a power of two) entries: 128, 64, 32
@pytest.mark.parametrize("n,length", [(257, 31), (250, 32), (133, 63), (131, 64), (70, 127), (71, 128), (5, 1843),
                                      (9, 4000), (1, 700)])
@pytest.mark.parametrize("nrhs", [1, 2, 3, 4, 8, 13, 16])
def test_long_rows(P, n, length, nrhs):
    import torch
    rng = np.random.default_rng(length + nrhs)
    A, row, col, val = _random(P, n, length, rng)
    x = rng.standard_normal((n, nrhs))
    t = val[:, None] * x[col]
    ref, mag = np.zeros((n, nrhs)), np.zeros((n, nrhs))
    np.add.at(ref, row, t)
    np.add.at(mag, row, np.abs(t))
    c = P.Context()
    y = torch.full((n, nrhs), float("nan"), dtype=torch.float64, device="cuda")
    P.rw_spmv(c, A, torch.as_tensor(x).cuda(), y)
    # two sums of m rounded products in any two orders differ by at most 2 (m + 1) u of the terms' size
    assert (np.abs(y.cpu().numpy() - ref) <= 2.0 * (length + 1) * 2.0 ** -53 * mag).all()
    c.close()


@pytest.mark.parametrize("nrhs", [1, 3, 16])
def test_pcg_of_a_dense_graph(P, nrhs):
    # the FP64 and the FP32 operator, the true residual and the dot products of long rows
    import torch
    rng = np.random.default_rng(2)
    n = 400
    a, b = np.triu_indices(n, 1)
    keep = rng.random(a.size) < 0.6
    g = np.exp(rng.uniform(-1, 1, keep.sum()))
    A = W.assemble(n, a[keep], b[keep], g, 1e-2 * W.conductance_sums(n, a[keep], b[keep], g))
    c = P.Context()
    dA = P.CSR.from_host(A)
    F = P.rw_build_factor(c, dA, 40, 3, 0.0)
    r = rng.standard_normal((n, nrhs))
    ref = np.linalg.solve(A.to_dense(), r)
    for prec, tol in ((P.RW_FP64, 1e-11), (P.RW_FP32_MIXED, 1e-6)):
        x = torch.empty((n, nrhs), dtype=torch.float64, device="cuda")
        rc, _, _, rel = P.pcg_solve(c, dA, F, torch.as_tensor(r).cuda(), x, tol, 100, prec)
        true = np.linalg.norm(r - A.to_dense() @ x.cpu().numpy(), axis=0) / np.linalg.norm(r, axis=0)
        assert rc == 0 and (true < 1.01 * tol).all() and np.abs(true / rel - 1.0).max() < 1e-2
        # ||x - ref|| <= ||A^-1|| ||r - A x||: the condition number of this matrix is below 200
        assert np.linalg.norm(x.cpu().numpy() - ref) / np.linalg.norm(ref) < 200 * tol
    F.destroy()
    c.close()


@pytest.mark.parametrize("nrhs", [1, 16])
def test_time_per_entry(P, nrhs):
    import torch
    rng = np.random.default_rng(1)
    per = {}
    c = P.Context()
    for n, length in ((8000, 500), (2200, 1800)):  # 4 million entries each
        A = _random(P, n, length, rng)[0]
        x = torch.randn((n, nrhs), dtype=torch.float64, device="cuda")
        y = torch.empty_like(x)
        best = 1e9
        for _ in range(10):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            for _ in range(5):
                P.rw_spmv(c, A, x, y)
            best = min(best, time.perf_counter() - t0)
        per[length] = best / (n * length)
    c.close()
    assert per[1800] < 1.6 * per[500], per
