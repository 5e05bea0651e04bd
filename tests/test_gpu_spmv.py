"""SpMV against FP64 sums on the host: every right-hand-side count and entry
slicing, row lengths around the copied pass and the long-row limit."""
import numpy as np
import pytest

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


def _rows(kind, rng):
    """Row lengths (each at least 1)."""
    return {"one": np.ones(1), "short": rng.integers(1, 4, 1500), "stencil": np.full(777, 27),
            "ragged": rng.integers(1, 40, 1031), "full": np.full(64, 64),
            "long": np.where(np.arange(600) % 97 == 5, 300, 3), "huge": np.where(np.arange(90) == 40, 5000, 2),
            "limit": np.concatenate([np.full(32, 64), np.full(32, 65), np.full(33, 2049)])}[kind].astype(np.int64)


@pytest.mark.parametrize("nrhs", [1, 2, 3, 4, 7, 8, 16])
@pytest.mark.parametrize("kind", ["one", "short", "stencil", "ragged", "full", "long", "huge", "limit"])
def test_spmv(P, kind, nrhs):
    import torch
    rng = np.random.default_rng(11 + nrhs)
    length = _rows(kind, rng)
    n = len(length)
    rp = np.concatenate([[0], np.cumsum(length)]).astype(np.int32)
    col = rng.integers(0, n, rp[-1]).astype(np.int32)
    val = rng.standard_normal(rp[-1])
    x = rng.standard_normal((n, nrhs))
    row = np.repeat(np.arange(n), length)
    t = val[:, None] * x[col]
    ref, mag = np.zeros((n, nrhs)), np.zeros((n, nrhs))
    np.add.at(ref, row, t)
    np.add.at(mag, row, np.abs(t))
    # two sums of m rounded products in any two orders differ by at most 2 (m + 1) u of the terms' size
    bound = 2.0 * (length[:, None] + 1) * 2.0 ** -53 * mag
    A = P.CSR(*(torch.as_tensor(v).cuda() for v in (rp, col, val)))
    dx = torch.as_tensor(x).cuda()
    for slices in (0, 1, 4, 32):
        c = P.Context(options=P.rw_options_default(spmv_slices=slices))
        try:
            y = torch.full_like(dx, float("nan"))
            P.rw_spmv(c, A, dx, y)
            assert (np.abs(y.cpu().numpy() - ref) <= bound).all(), slices
        finally:
            c.close()
