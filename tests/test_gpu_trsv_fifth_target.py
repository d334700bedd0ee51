"""Triangular solves where a helper CTA of the chain owns a fifth target block
(35,841 <= n <= 38,848): held to the componentwise backward error of a
backward-stable solve and to torch's own triangular solve, as at the smaller
sizes, and repeated bit for bit."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import rfm_workloads as W  # noqa: E402


@pytest.mark.parametrize("trans", [0, 1])
def test_fifth_target(trans):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_04170_gb300 import build, rfm
    build.build()
    gp = rfm.Problem(W.problem(3, (4, 4, 4), 563, (4, 4, 4), (3, 3, 3), (3, 3, 3)))
    n, u = gp.n, 2.0 ** -53
    assert n == 36032
    g = torch.Generator(device="cuda").manual_seed(7)
    Rt = torch.randn(n, n, dtype=torch.float64, device="cuda", generator=g).tril_().div_(n ** 0.5)
    Rt.diagonal().add_(2.0)
    gp.rfm_set_r(Rt)  # R^T in row-major order is R column-major
    b = torch.randn(n, dtype=torch.float64, device="cuda", generator=g)
    x = gp.rfm_trsv(b, trans)
    assert torch.equal(gp.rfm_trsv(b, trans), x)
    A = Rt.T if trans == 0 else Rt
    ref = torch.linalg.solve_triangular(A, b[:, None], upper=(trans == 0))[:, 0]
    assert (torch.linalg.vector_norm(x - ref) / torch.linalg.vector_norm(ref)).item() <= 10 * u * n
    res = (b - A @ x).abs()
    assert torch.all(res <= 10 * n * u * (A.abs() @ x.abs()))
