"""Two-game calls that share F_AT and not F_A may overlap: F_AT is only read."""
import threading

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nrhs", [1, 5])
def test_overlapping_two_game_calls(nrhs):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_math_0609672_gb300 as P
    from paper_math_0609672_gb300 import _build
    _build.build()
    rng = np.random.default_rng(4)
    A = W.asym_grid((15, 14, 9), rng, skew=0.5)  # narrow levels, then wide ones
    dA = P.CSR.from_host(A)
    streams = [torch.cuda.Stream() for _ in range(3)]
    ctxs = [P.Context(stream=s) for s in streams]
    dAT = P.rw_csr_transpose(ctxs[0], dA)
    FAT = P.rw_build_factor(ctxs[0], dAT, 80, 4, 1e-3)
    FA = [P.rw_build_factor(c, dA, 80, 10 + i, 1e-3) for i, c in enumerate(ctxs[:2])]
    rs = [torch.as_tensor(rng.standard_normal((A.n, nrhs))).cuda() for _ in range(3)]
    b = [r[:, 0].contiguous() for r in rs]

    def work(i, out):
        """The two games with F_A number i; the third one applies F_AT by itself."""
        for _ in range(20):
            z = torch.empty_like(rs[i])
            if i == 2:
                P.rw_precond_apply(ctxs[2], FAT, rs[2], z)
                out.append(z)
                continue
            P.rw_precond_apply_ldu(ctxs[i], FA[i], FAT, rs[i], z)
            x = torch.empty_like(b[i])
            rc, _ = P.bicgstab_solve(ctxs[i], dA, FA[i], FAT, b[i], x, 1e-8, 200)
            assert rc == 0
            out += [z, x]

    ref = [[], [], []]
    for i in range(3):  # one after the other
        with torch.cuda.stream(streams[i]):
            work(i, ref[i])
    torch.cuda.synchronize()
    out = [[], [], []]
    fail = []

    def run(i):
        try:
            with torch.cuda.stream(streams[i]):
                work(i, out[i])
        except Exception as e:  # noqa: BLE001
            fail.append(e)

    ts = [threading.Thread(target=run, args=(i,)) for i in range(3)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    torch.cuda.synchronize()
    assert not fail, fail
    for i in range(3):
        assert len(out[i]) == len(ref[i])
        assert all(torch.equal(a, r) for a, r in zip(out[i], ref[i])), i
    for F in FA + [FAT]:
        F.destroy()
    for c in ctxs:
        c.close()
