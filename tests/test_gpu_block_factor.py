"""The cooperative block factorisation (k_block) at the edges of its panels,
blocks and row slabs, on the FP64 and the tensor-core QR.

R is fixed by R^T R = B^T B with a positive diagonal.  Householder QR is
columnwise backward stable, ||(B + dB) - Q R|| with ||dB_j|| <= c s n u ||B_j||
for a small constant c (Higham, Theorem 19.4), so entry (i, j) of R^T R is
within 2 c s n u ||B_i|| ||B_j||; c = 1 is used here (rounding errors add up
like a random walk and stay far below the worst case), with sqrt(s n) for s n."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

U = 2.0 ** -53


@pytest.fixture(scope="module")
def rfm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_04170_gb300 import build, rfm as _rfm
    build.build()
    return _rfm


def factor(rfm, B, tc):
    fn = rfm.rfm_householder_r_tc if tc else rfm.rfm_householder_r
    s, n = B.shape
    # a copy: the entry point overwrites its input (B.T of one column shares B's storage)
    R, low = fn(B.T.clone(memory_format=torch.contiguous_format), s, n)
    return R.T.contiguous(), low


def holds(B, R):
    s, n = B.shape
    G, H = B.T @ B, R.T @ R
    nb = torch.linalg.vector_norm(B, dim=0)
    tol = 8.0 * (s * n) ** 0.5 * U * nb[:, None] * nb[None, :]
    assert torch.equal(R, R.triu()) and bool((R.diagonal() > 0).all())
    assert bool(((G - H).abs() <= tol).all()), float(((G - H).abs() / tol).max())


# one column; one row per column; a panel, a block and one more; rows that leave
# some CTAs of the last cluster empty; a slab of many rows per warp; outer blocks
# of 256 and 512 columns, whole and ragged, and blocks built from 64 columns
SIZES = [(1, 1), (33, 1), (32, 32), (33, 33), (65, 31), (130, 129), (257, 96), (500, 127), (1201, 128), (2999, 161),
         (20000, 130), (40001, 140), (66000, 70),
         (1300, 700), (2600, 1100), (3100, 1537), (20000, 600)]


@pytest.mark.parametrize("s,n", SIZES)
@pytest.mark.parametrize("tc", [False, True])
def test_factor_sizes(rfm, s, n, tc):
    g = torch.Generator(device="cuda").manual_seed(s + n)
    B = torch.randn(s, n, dtype=torch.float64, device="cuda", generator=g)
    R, low = factor(rfm, B, tc)
    holds(B, R)
    assert torch.equal(factor(rfm, B, tc)[0], R)  # fixed order of all sums


@pytest.mark.parametrize("scale", [-455, -300, 300, 500])
def test_factor_exponent_range(rfm, scale):
    """Column norms whose squares lie near the ends of the FP64 range."""
    g = torch.Generator(device="cuda").manual_seed(1)
    B = torch.randn(300, 40, dtype=torch.float64, device="cuda", generator=g)
    R, _ = factor(rfm, B * 2.0 ** scale, False)
    holds(B, R * 2.0 ** -scale)


def test_factor_zero_tails_and_non_finite(rfm):
    """Columns without entries below the diagonal need no reflector; a zero
    column raises the rank flag; a NaN reaches R."""
    g = torch.Generator(device="cuda").manual_seed(2)
    T = torch.randn(48, 48, dtype=torch.float64, device="cuda", generator=g).triu()
    B = torch.zeros(200, 48, dtype=torch.float64, device="cuda")
    B[:48] = T
    R, low = factor(rfm, B, False)
    assert not low and torch.equal(R, T * torch.sign(T.diagonal())[:, None])
    B[:, 20] = 0.0
    assert factor(rfm, B, False)[1]
    B = torch.randn(200, 48, dtype=torch.float64, device="cuda", generator=g)
    B[100, 10] = float("nan")
    R, _ = factor(rfm, B, False)
    assert bool(torch.isnan(R[10, 10]))
