"""After a wait of the triangular solve, LSQR or the line search gave up, the next
call gives the bits of an undisturbed problem: records that a launch without its
waits left behind, under the tags of the next one, are not taken for results."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import rfm_workloads as W  # noqa: E402


@pytest.mark.parametrize("M", [48, 200])  # 6 and 25 blocks of 64 rows: one helper target each
def test_next_call_after_a_timeout(M):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_04170_gb300 import build, rfm
    build.build()
    desc = W.small_3d(M=M, q=7)
    n = 8 * M
    c = torch.as_tensor(W.random_coeffs(n, seed=3, scale=0.1), device="cuda")
    d = -1.3 * c + 0.01 * torch.as_tensor(W.random_coeffs(n, seed=4), device="cuda")
    b = torch.as_tensor(np.random.default_rng(1).standard_normal(n), device="cuda")
    ref, gp = rfm.Problem(desc), rfm.Problem(desc)
    for p in (ref, gp):
        F, _ = p.rfm_assemble(c)
        p.rfm_sketch("count", 3 * n, 0, copy_out=False)
        p.rfm_qr(copy_out=False)
    f0 = ref.rfm_residual(c)[1]
    calls = [lambda p: p.rfm_trsv(b), lambda p: p.rfm_trsv(b, trans=1), lambda p: p.rfm_linesearch(c, d, f0),
             lambda p: p.rfm_lsqr(-F)]
    want = [call(ref) for call in calls]

    def same(x, y):
        return torch.equal(x, y) if torch.is_tensor(x) else \
            all(same(i, j) for i, j in zip(x, y)) if isinstance(x, tuple) else x == y

    for _ in range(10):
        for call, w in zip(calls, want):
            gp.rfm_set_wait_limit(-1)
            with pytest.raises(rfm.RfmError) as e:
                call(gp)
            assert e.value.status == rfm.RFM_ETIMEOUT
            gp.rfm_set_wait_limit(0)
            assert same(call(gp), w)
