"""Memory of the solves' blocks: a short stretch of narrow levels takes what its
rows need, and a factor whose blocks cannot be allocated keeps those that can,
the other rows one by one, with the same solution."""
import numpy as np
import pytest

import workloads as W

from test_gpu_failures import FailingAllocator
from test_gpu_rows import _matvec

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


class SmallAllocator(FailingAllocator):
    """No request of `limit` bytes or more is met."""

    def __init__(self, limit):
        super().__init__()
        self.limit = limit
        self.refused = 0

    def alloc(self, nbytes, stream):
        if nbytes >= self.limit:
            self.refused += 1
            return 0
        return super().alloc(nbytes, stream)


def _check(P, c, F, n, nrhs):
    import torch
    t = {k: v.cpu().numpy() for k, v in F.tensors().items()}
    r = np.random.default_rng(nrhs).standard_normal((n, nrhs))
    z = torch.empty((n, nrhs), dtype=torch.float64, device="cuda")
    P.rw_precond_apply(c, F, torch.as_tensor(r).cuda(), z)
    y = _matvec(t["y_row_ptr"], t["y_col"], t["y_val"], z.cpu().numpy())
    back = _matvec(t["yt_row_ptr"], t["yt_col"], t["yt_val"], y * t["d"][:, None])
    assert np.abs(back - r).max() / np.abs(r).max() < 1e-11


def test_short_stretches_take_little(P):
    fa = FailingAllocator()
    c = P.Context(allocator=(fa.alloc, fa.free))
    F = P.rw_build_factor(c, P.CSR.from_host(W.tridiag(20, diag=2.1)), 20, 3, 0.0)
    # per direction: a triangle of 20 rows (210 entries), 42 KB of slots, and arrays of one 256-byte piece each
    assert sum(fa.live.values()) < 2 * (44 << 10) + (24 << 10)
    _check(P, c, F, 20, 3)
    F.destroy()
    c.close()
    assert not fa.live


@pytest.mark.parametrize("fp32", [0, 1])
def test_blocks_that_cannot_be_allocated(P, fp32):
    n = 60000  # 62 MB of FP64 inverses per direction
    A = W.tridiag(n, diag=2.1)
    dA = P.CSR.from_host(A)
    fa = SmallAllocator(40 << 20)
    c = P.Context(allocator=(fa.alloc, fa.free), options=P.rw_options_default(store_fp32=fp32))
    F = P.rw_build_factor(c, dA, 20, 3, 0.0)
    assert fa.refused >= 1
    for nrhs in (1, 4):
        _check(P, c, F, n, nrhs)
    B = P.Batch(c, [dA, dA], [F, F])  # 124 MB: the same for a batch
    B.destroy()
    F.destroy()
    c.close()
    assert not fa.live
