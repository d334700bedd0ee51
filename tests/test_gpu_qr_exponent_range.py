"""R of matrices whose column norms squared leave the normal FP64 range or come
within a few octaves of its end, on every QR entry point."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("entry", ["rfm_householder_r", "rfm_householder_r_tc", "rfm_householder_r_noalloc"])
@pytest.mark.parametrize("scale", [-518, 506])
def test_norms_near_the_ends_of_the_range(entry, scale):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import ctypes
    from paper_2510_04170_gb300 import build, rfm
    build.build()
    s, n = 300, 140
    g = torch.Generator(device="cuda").manual_seed(1)
    B = torch.randn(s, n, dtype=torch.float64, device="cuda", generator=g)
    A = (B * 2.0 ** scale).T.contiguous()
    if entry == "rfm_householder_r_noalloc":
        R = torch.empty(n, n, dtype=torch.float64, device="cuda")
        flag = ctypes.c_int()
        torch.cuda.synchronize()
        assert rfm.load().rfm_householder_r_noalloc(ctypes.c_void_p(A.data_ptr()), s, n, None,
                                                    ctypes.c_void_p(R.data_ptr()), ctypes.byref(flag)) == 0
    else:
        R, low = getattr(rfm, entry)(A, s, n)
        assert not low
    R = R.T.triu() * 2.0 ** -scale  # exact: R's entries are normal numbers
    assert bool(torch.isfinite(R).all()) and bool((R.diagonal() > 0).all())
    # Products of two entries are near 2^(2 scale): at 2^-1036 each is rounded to a
    # multiple of 2^-1074, so a sum of s of them is off by s 2^-1075 at most where it
    # is of the order s 2^-1036, 2^-39 relative, once per reflector and twice in R^T R.
    # Otherwise the bound of Householder QR, as in the block factorisation's test.
    nb = torch.linalg.vector_norm(B, dim=0)
    unit = 2.0 * n * 2.0 ** -39 if scale < 0 else 8.0 * (s * n) ** 0.5 * 2.0 ** -53
    assert bool(((B.T @ B - R.T @ R).abs() <= unit * nb[:, None] * nb[None, :]).all())
