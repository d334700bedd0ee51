"""Outputs that are pinned bit for bit, and the LSQR step counts that follow them.

The LSQR of a solve stops by a test on rounded numbers, and at cond(R) = 1e8 ..
1e9 the last bits of J, R and of a triangular solve decide on about every fourth
problem whether that is one step sooner or later.  The order and the roundings of
those sums are therefore part of the results: a kernel may spread the work
differently but returns the same bits.  The digests (SHA-256 of the bytes) and
the counts were recorded on a GB300 with 152 SMs; the row split of the QR's sums
depends on the number of SMs."""
import hashlib

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import rfm_workloads as W  # noqa: E402


@pytest.fixture(scope="module")
def rfm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("recorded with 152 SMs")
    from paper_2510_04170_gb300 import build, rfm as _rfm
    build.build()
    return _rfm


def vec(count, tag):
    """Fixed values in [-1, 1) (a multiplicative hash of the index)."""
    i = np.arange(1, count + 1, dtype=np.uint64) * np.uint64(0x9E3779B97F4A7C15)
    i += np.uint64(tag * 0xD1B54A32D192ED03 % 2 ** 64)
    i ^= i >> np.uint64(29)
    i *= np.uint64(0xBF58476D1CE4E5B9)
    return torch.as_tensor((i >> np.uint64(11)).astype(np.float64) * 2.0 ** -52 - 1.0, device="cuda")


def digest(*tensors):
    h = hashlib.sha256()
    for t in tensors:
        h.update(t.contiguous().cpu().numpy().tobytes())
    return h.hexdigest()[:16]


PROBLEMS = {
    "kind0_2d": lambda: W.problem(2, (3, 2), 37, (11, 9), (7, 7), (8, 8)),
    "kind0": lambda: W.problem(3, (2, 2, 2), 45, (6, 6, 6), (4, 4, 4), (4, 4, 4)),
    "kind1": lambda: W.problem(3, (2, 2, 2), 33, (6, 6, 6), (5, 5, 5), (5, 5, 5), fields=2, pde_kind=1),
    "kind2_2d": lambda: W.problem(2, (2, 2), 100, (20, 20), (20, 20), (20, 20), pde_kind=2),
    "kind2": lambda: W.problem(3, (3, 2, 2), 64, (7, 6, 6), (4, 5, 4), (4, 4, 4), pde_kind=2),
    "kind4": lambda: W.problem(3, (2, 2, 2), 45, (6, 6, 6), (4, 4, 4), (4, 4, 4), pde_kind=4),
    "kind5": lambda: W.problem(3, (3, 3, 3), 45, (6, 6, 6), (4, 4, 4), (4, 4, 4), pde_kind=5),
    "kind6": lambda: W.problem(3, (2, 2, 2), 70, (6, 6, 6), (4, 4, 4), (4, 4, 4), pde_kind=6),
    "kind7": lambda: W.ball(40, 6, 300),
}


def assembled(rfm, name):
    gp = rfm.Problem(PROBLEMS[name]())
    c = vec(gp.n, 1) * 0.1
    return gp, c, gp.rfm_assemble(c)


def run_assemble(rfm, name):
    gp, c, (F, lam) = assembled(rfm, name)
    Jp, Js, _ = gp.rfm_get_jacobian()
    alpha, f = gp.rfm_linesearch(c, -1.3 * c + 0.01 * vec(gp.n, 2), gp.rfm_residual(c)[1])
    return F, lam, Jp, Js, gp.rfm_residual(0.9 * c)[0], torch.tensor([alpha, f], dtype=torch.float64)


ASSEMBLE = {
    'kind0_2d': '54d0f2806fdab43b',
    'kind0': '71b1dc80055421ae',
    'kind1': '710a4b07b0e2f40d',
    'kind2_2d': 'b2d3531204a5271e',
    'kind2': 'b9cf1088f4b9fa08',
    'kind4': '2f0f81e7361b7a3c',
    'kind5': '0d798da6bfa5350a',
    'kind6': '59e2fcada769b1ba',
    'kind7': '0ade3f6f2625de8a',
}


@pytest.mark.parametrize("name", list(PROBLEMS))
def test_assembly(rfm, name):
    assert digest(*run_assemble(rfm, name)) == ASSEMBLE[name]


def run_products(rfm, name):
    gp, _, _ = assembled(rfm, name)
    return gp.rfm_jmv(vec(gp.n, 3), 0), gp.rfm_jmv(vec(gp.m, 4), 1)


PRODUCTS = {
    'kind0_2d': '56263d4b738cc017',
    'kind0': 'edc0e124226aacdb',
    'kind1': '55c71b4d50daed1a',
    'kind2_2d': 'dde1f21b9d699edd',
    'kind2': '842de401eac0491a',
    'kind4': 'c88cb634dcd007b0',
    'kind5': '6e4cebc1da280bba',
    'kind6': 'a0a74712fc3ad251',
    'kind7': '946183647454707e',
}


@pytest.mark.parametrize("name", list(PROBLEMS))
def test_products(rfm, name):
    assert digest(*run_products(rfm, name)) == PRODUCTS[name]


def triangular(n):
    """Upper triangle with a dominant diagonal, column-major."""
    return (vec(n * n, 5).view(n, n).tril() / n ** 0.5 + 2.0 * torch.eye(n, dtype=torch.float64, device="cuda")).contiguous()


def run_trsv(rfm, gm):
    g, M = gm
    gp = rfm.Problem(W.problem(3, (g,) * 3, M, (4, 4, 4), (3, 3, 3), (3, 3, 3)))
    gp.rfm_set_r(triangular(gp.n))
    return gp.rfm_trsv(vec(gp.n, 6), 0), gp.rfm_trsv(vec(gp.n, 7), 1)


# subdomains per axis and features: part of a block, one block, ragged last
# blocks, one to four targets per helper
TRSV_CASES = [(1, 24), (1, 64), (1, 65), (1, 257), (2, 45), (2, 250), (3, 300), (4, 300)]
TRSV = {
    (1, 24): '5a51774327bb7dda',
    (1, 64): 'befd79fcc94dfefb',
    (1, 65): '8997f9cfce975ae0',
    (1, 257): 'bcb68d129ecd3685',
    (2, 45): '89cc4096fec1c028',
    (2, 250): 'db3a7760a77a696c',
    (3, 300): '9c6a510765ef454b',
    (4, 300): '07655576d44365ca',
}


@pytest.mark.parametrize("gm", TRSV_CASES)
def test_triangular_solves(rfm, gm):
    assert digest(*run_trsv(rfm, gm)) == TRSV[gm]


def run_lsqr(rfm, name):
    gp, _, (F, _) = assembled(rfm, name)
    gp.rfm_set_r(triangular(gp.n))
    d, itn, istop = gp.rfm_lsqr(-F, 1e-13, 1e30, 37)
    return d, torch.tensor([itn, istop])


LSQR = {
    'kind0_2d': '78f42e8c55b48476',
    'kind0': '5021ed33954c6a9d',
    'kind1': '5abcb4e490c50fd2',
    'kind2_2d': 'e8bbcee8b3a8b776',
    'kind2': 'c08c548e08893da2',
    'kind4': 'd0a9c56839f707b7',
    'kind5': '7d979debcb430daf',
    'kind6': '86b4da82ff667a57',
    'kind7': 'eeb25b7e41f1f7e3',
}


@pytest.mark.parametrize("name", list(PROBLEMS))
def test_lsqr_directions(rfm, name):
    assert digest(*run_lsqr(rfm, name)) == LSQR[name]


def run_qr(rfm, key):
    tc, s, n = key
    B = vec(s * n, 8).view(n, s)
    return (rfm.rfm_householder_r_tc if tc else rfm.rfm_householder_r)(B, s, n)[0],


# one chunk, chunks shorter than 64 rows, a chunk per SM and fewer, chunks of one
# remainder modulo 32 in one to five parts, slabs too tall for a cluster, and
# several panels and blocks with ragged ends
QR_CASES = [(tc, s, n) for tc in (False, True) for s, n in
            [(1, 1), (33, 31), (65, 65), (97, 40), (500, 127), (1201, 400), (9800, 70), (12288, 300), (60001, 64),
             (108000, 33), (121000, 33), (2600, 1100), (3100, 1537)]]
QR = {
    (False, 1, 1): 'bc05bd1b03a6a949',
    (False, 33, 31): '5da962065938d2dd',
    (False, 65, 65): '238b021675072f69',
    (False, 97, 40): '84bfcf09206c0163',
    (False, 500, 127): 'a192cc852199bf9b',
    (False, 1201, 400): 'fc01d0a62250ab00',
    (False, 9800, 70): 'ec9db505b490e487',
    (False, 12288, 300): 'a9b63c2abc3a56f5',
    (False, 60001, 64): 'f347feef90be2b13',
    (False, 108000, 33): '5a58bbf3a495bd14',
    (False, 121000, 33): '9d88379da04bb48f',
    (False, 2600, 1100): '30fcd7c2c4e11e4b',
    (False, 3100, 1537): '97ca3b4134858f93',
    (True, 1, 1): 'bc05bd1b03a6a949',
    (True, 33, 31): '5da962065938d2dd',
    (True, 65, 65): '238b021675072f69',
    (True, 97, 40): '84bfcf09206c0163',
    (True, 500, 127): 'a192cc852199bf9b',
    (True, 1201, 400): '9214c5787df07174',
    (True, 9800, 70): 'ec9db505b490e487',
    (True, 12288, 300): '9f74559f327ec14b',
    (True, 60001, 64): 'f347feef90be2b13',
    (True, 108000, 33): '5a58bbf3a495bd14',
    (True, 121000, 33): '9d88379da04bb48f',
    (True, 2600, 1100): '4a0af2138da670df',
    (True, 3100, 1537): '8b6af6291aa10a2c',
}


@pytest.mark.parametrize("key", QR_CASES)
def test_r(rfm, key):
    assert digest(*run_qr(rfm, key)) == QR[key]


def run_solve(rfm, key):
    name, precision, first, count = key
    out = []
    for seed in range(first, first + count):
        d = dict(W.config_c1()) if name == "c1" else W.problem(3, (2, 2, 2), 512, (12, 12, 12), (6, 6, 6), (6, 6, 6),
                                                               pde_kind=2)
        d["seed"] = W.FEATURE_SEED + 1000 * seed
        gp = rfm.Problem(d)
        info = gp.rfm_ipn_solve(W.solve_opts(precision=precision))[1]
        out.append(info["lsqr_iters_total"])
    return out


# whole IPN solves of C1 and of a C5-sized problem over feature seeds: LSQR steps
SOLVE_CASES = [("c1", 0, 112, 16), ("c5", 2, 100, 8), ("c5", 0, 100, 8)]
SOLVE = {
    ('c1', 0, 112, 16): [90, 90, 93, 86, 88, 86, 88, 97, 93, 87, 87, 92, 85, 87, 88, 87],
    ('c5', 2, 100, 8): [137, 133, 139, 128, 127, 133, 132, 133],
    ('c5', 0, 100, 8): [137, 132, 139, 128, 127, 133, 132, 132],
}


@pytest.mark.parametrize("key", SOLVE_CASES)
def test_step_counts(rfm, key):
    assert run_solve(rfm, key) == SOLVE[key]
