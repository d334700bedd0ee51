"""Triangular solves and Jacobian products at the edges of their blocks: one
block, a block and one row, ragged last blocks, one and several targets per
helper CTA; row counts that are no multiple of the rows per warp, and the rows of
a column block split over several CTAs.

Bounds: a solve by 64 x 64 diagonal inverses of a matrix with a dominant diagonal
is componentwise backward stable, |b - R x| <= 10 n u |R| |x|; a product summed in
any order is within n_terms u |J| |x| of the exact one, twice that between two."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import rfm_workloads as W  # noqa: E402

U = 2.0 ** -53


@pytest.fixture(scope="module")
def rfm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_04170_gb300 import build, rfm as _rfm
    build.build()
    return _rfm


@pytest.mark.parametrize("g,M", [((1, 1, 1), 1), ((1, 1, 1), 63), ((1, 1, 1), 64), ((1, 1, 1), 65), ((1, 1, 1), 128),
                                 ((2, 1, 1), 97), ((2, 2, 2), 31), ((2, 2, 2), 129), ((3, 3, 3), 340),
                                 ((3, 3, 4), 505)])
def test_triangular_solve_sizes(rfm, g, M):
    gp = rfm.Problem(W.problem(3, g, M, (3, 3, 3), (2, 2, 2), (2, 2, 2)))
    n = gp.n
    gen = torch.Generator(device="cuda").manual_seed(n)
    R = torch.randn(n, n, dtype=torch.float64, device="cuda", generator=gen).triu_() / n ** 0.5
    R.diagonal().add_(2.0)
    gp.rfm_set_r(R.T.contiguous())
    b = torch.randn(n, dtype=torch.float64, device="cuda", generator=gen)
    for trans in (0, 1):
        A = R if trans == 0 else R.T
        x = gp.rfm_trsv(b, trans)
        assert bool(((b - A @ x).abs() <= 10 * n * U * (A.abs() @ x.abs())).all())
        for _ in range(3):  # deterministic, whatever the previous solve left behind
            assert torch.equal(gp.rfm_trsv(b, trans), x)


@pytest.mark.parametrize("g,M,q,qf,fields", [(1, 3, 3, 2, 1), (1, 70, 5, 4, 1), (2, 37, 9, 5, 1), (2, 65, 13, 7, 1),
                                             (3, 20, 7, 4, 2)])
def test_jacobian_product_sizes(rfm, g, M, q, qf, fields):
    gp = rfm.Problem(W.problem(3, (g,) * 3, M, (q,) * 3, (qf,) * 3, (qf,) * 3, fields=fields,
                               pde_kind=1 if fields == 2 else 0))
    gen = torch.Generator(device="cuda").manual_seed(M)
    gp.rfm_assemble(0.1 * torch.randn(gp.n, dtype=torch.float64, device="cuda", generator=gen))
    Jp, Js, blk = gp.rfm_get_jacobian()
    J = torch.zeros(gp.m, gp.n, dtype=torch.float64, device="cuda")
    cols = torch.arange(gp.W, device="cuda")
    J.scatter_(1, blk[:, :1].long() * gp.W + cols, Jp)
    if gp.m_iface:
        fa = slice(gp.m_int, gp.m_int + gp.m_iface)
        J[fa] = J[fa].scatter(1, blk[fa, 1:].long() * gp.W + cols, Js)
    x = torch.randn(gp.n, dtype=torch.float64, device="cuda", generator=gen)
    y = torch.randn(gp.m, dtype=torch.float64, device="cuda", generator=gen)
    assert bool(((gp.rfm_jmv(x, 0) - J @ x).abs() <= 2 * 2 * gp.W * U * (J.abs() @ x.abs())).all())
    z = gp.rfm_jmv(y, 1)
    assert bool(((z - J.T @ y).abs() <= 2 * gp.m * U * (J.T.abs() @ y.abs())).all())
    assert torch.equal(gp.rfm_jmv(y, 1), z)
