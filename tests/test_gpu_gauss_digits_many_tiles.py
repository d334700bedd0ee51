"""The Gaussian sketch's digit kernel where every CTA forms hundreds of tiles: its
queue of pairs that FP32 cannot decide fills and is worked off many times, and
all threads of a CTA have to agree on when."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import rfm_workloads as W  # noqa: E402
from perf.cases import _gauss_columns  # noqa: E402


@pytest.mark.parametrize("s", [16384, 16130])
def test_every_digit_and_repeated_bits(s):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_04170_gb300 import build, rfm
    build.build()
    # 124,416 rows in 64 blocks: 128 x 2,240 tiles for 1,216 CTAs
    desc = W.problem(3, (4, 4, 4), 16, (12, 12, 12), (6, 6, 6), (6, 6, 6))
    gp = rfm.Problem(desc)
    gp.rfm_assemble(torch.as_tensor(W.random_coeffs(gp.n, seed=2, scale=0.1), device="cuda"))
    gp.rfm_set_precision(1)
    B = gp.rfm_sketch("gauss", s, 2)
    for _ in range(4):
        assert torch.equal(gp.rfm_sketch("gauss", s, 2), B)
    Jp, Js, blk = gp.rfm_get_jacobian()
    e0, e1 = blk[:, 0], blk[:, 1]
    iface = torch.arange(gp.m, device="cuda") >= gp.m_int
    iface &= torch.arange(gp.m, device="cuda") < gp.m_int + gp.m_iface
    for b in range(gp.G):
        r, r2 = torch.nonzero(e0 == b)[:, 0], torch.nonzero((e1 == b) & iface)[:, 0]
        rows, J = torch.cat([r, r2]), torch.cat([Jp[r], Js[r2 - gp.m_int]])
        S = _gauss_columns(s, rows, 2, desc["seed"])
        # a product rounded once against one of `rows` rounded terms; a wrong digit
        # (1/16 of a Jacobian entry of order 1 to 100) is far outside
        tol = 2.3e-16 * rows.numel() * (S.abs() @ J.abs())
        assert bool(((B[b * 16:(b + 1) * 16].T - S @ J).abs() <= tol).all())
