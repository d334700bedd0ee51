"""Cases that stand for what a user of this library has it do, each through its
public entry points (`paper_2510_04170_gb300.rfm`): two whole Newton solves, and
the steps a solve consists of (assembly, sketch, sketch + QR, LSQR, triangular
solves, Jacobian products, line search) over the sizes of this repository's
configurations: C1 (2D, n = 400), C4 (n = 1,024 .. 16,384), C5 (n = 4,096), the
paper's 3D settings (n = 3,200) and C2 (n = 32,768).

In all of them the seed gives the features, the coefficients and the right-hand
sides.  `exact` restates each step in plain FP64 torch / numpy.
"""
import math
import random

import numpy as np
import torch

import rfm_workloads as W
from paper_2510_04170_gb300 import rfm

C_SCALE = 100.0


def listed():
    return [
        # Whole IPN solve of C1: the smallest 2D problem, FP64 throughout (the
        # default precision), about 100 LSQR steps: latency and launches.
        dict(name="ipn_2d", op="solve", solver="ipn", dim=2, g=2, M=100, q=20, qf=20, kind=0, precision=0),
        # Whole IPN solve of one C5 instance (n = 4,096) at precision 2, the
        # solve that the warm-start experiment repeats for each parameter.
        dict(name="ipn_3d", op="solve", solver="ipn", dim=3, g=2, M=512, q=12, qf=6, kind=2, precision=2),
        # One Jacobian assembly of C2 (124,416 rows of 512): closed-form rows.
        dict(name="assemble_box", op="assemble", dim=3, g=4, M=512, q=12, qf=6, kind=0),
        # One Jacobian assembly at the paper's 3D settings (83,200 rows of 400),
        # strongly nonlinear operator: rows through the 2-jet of u.
        dict(name="assemble_jet", op="assemble", dim=3, g=2, M=400, q=20, qf=20, kind=6),
        # Gaussian sketch on the tensor cores (C2's kind, 16,384 columns).
        dict(name="sketch_gauss", op="sketch", dim=3, g=4, M=256, q=12, qf=6, kind=0, sketch="gauss", gamma=2.0,
             precision=2),
        # Preconditioner (count sketch, then QR) in FP64 at C4's smallest size.
        dict(name="precond_small", op="precond", dim=3, g=2, M=128, q=12, qf=6, kind=2, sketch="count", gamma=3.0,
             precision=0),
        # The same at C5's size with the QR update on the tensor cores.
        dict(name="precond_mid", op="precond", dim=3, g=2, M=512, q=12, qf=6, kind=2, sketch="count", gamma=3.0,
             precision=2),
        # Gaussian sketch and QR as in C2, half its columns (n = 16,384): the
        # step that a large solve spends its time on.
        dict(name="precond_large", op="precond", dim=3, g=4, M=256, q=12, qf=6, kind=0, sketch="gauss", gamma=2.0,
             precision=2),
        # LSQR to eta = 1e-6 at C4's smallest size: a few dozen steps of small
        # products and triangular solves.
        dict(name="lsqr_small", op="lsqr", dim=3, g=2, M=128, q=12, qf=6, kind=2, sketch="count", gamma=3.0,
             precision=0),
        # R^{-1} b and R^{-T} b at C2's size, as each of its LSQR steps does.
        dict(name="trsv_large", op="trsv", dim=3, g=4, M=512, q=6, qf=3, kind=0),
        # J x and J^T y with C2's Jacobian, the other half of an LSQR step.
        dict(name="jacobian_products", op="products", dim=3, g=4, M=512, q=12, qf=6, kind=0),
        # Golden-section line search of a C5 instance.
        dict(name="linesearch", op="linesearch", dim=3, g=2, M=512, q=12, qf=6, kind=2),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    """A step or a solve of a random problem: subdomains per axis, features per
    subdomain (odd counts included), grids and operator spread over what the
    configurations span.  2D problems keep M small and LSQR M <= 160: beyond,
    the coefficients and R are not determined to nine digits in FP64 by any
    algorithm (cond(J) ~ 1e9), so there is nothing to compare."""
    op = rng.choice(["solve", "assemble", "assemble", "sketch", "precond", "precond", "precond", "lsqr", "trsv",
                     "products", "linesearch"])
    dim = 3 if rng.random() < 0.8 else 2
    case = dict(op=op, dim=dim)
    if op in ("assemble", "products", "linesearch"):
        kind = rng.choice([0, 1, 2, 3, 4, 5, 6]) if dim == 3 else rng.choice([0, 2, 3])
        M = _log_int(rng, 24, 512 if kind != 1 else 256)
        q = rng.randint(7, 16) if dim == 3 else rng.randint(10, 40)
        case.update(kind=kind, M=M, g=rng.randint(1, 4), q=q, qf=rng.randint(3, q))
        return case
    if op == "trsv":
        case.update(kind=0, M=_log_int(rng, 24, 512), g=rng.randint(1, 4), q=4, qf=3)
        return case
    M = _log_int(rng, 24, {"solve": 320, "precond": 400, "sketch": 512, "lsqr": 160}[op]) if dim == 3 \
        else rng.randint(20, 48)
    # enough interior points for every unknown
    q = max(int(math.ceil((1.6 * M) ** (1.0 / dim))), 5) + rng.randint(1, 3)
    case.update(kind=rng.choice([0, 2, 4, 5] if dim == 3 else [0, 2]), M=M, q=q, qf=rng.randint(4, max(4, q - 1)))
    if op == "solve":
        case.update(solver=rng.choice(["ipn", "ipn", "amipn"]), kind=rng.choice([0, 2]), g=rng.randint(1, 2),
                    precision=rng.choice([0, 2]))
        return case
    if op == "lsqr":
        case.update(g=rng.randint(1, 2 if dim == 3 else 4), sketch="count", gamma=3.0, precision=rng.choice([0, 2]))
        return case
    precision = rng.choice([0, 2])
    gmax = 3 if precision == 2 else 2
    case.update(g=rng.randint(1, gmax), sketch=rng.choice(["count", "gauss"]), precision=precision,
                gamma=round(rng.uniform(2.0, 3.0), 2))
    return case


# ------------------------------------------------------------------- inputs
def _desc(case, seed):
    fields = 2 if case["kind"] == 1 else 1
    d, g, q, qf = case["dim"], case["g"], case["q"], case["qf"]
    return W.problem(d, (g,) * d, case["M"], (q,) * d, (qf,) * d, (qf,) * d, fields=fields, pde_kind=case["kind"],
                     seed=W.FEATURE_SEED + 1000 * int(seed))


def _sketch_rows(case, n):
    s = int(math.ceil(case["gamma"] * n))
    return s + s % 2


def _sizes(case):
    d, g, q, qf = case["dim"], case["g"], case["q"], case["qf"]
    fields = 2 if case["kind"] == 1 else 1
    G = g ** d
    m_int = G * fields * q ** d
    m_iface = d * (g - 1) * g ** (d - 1) * fields * 2 * qf ** (d - 1)
    m_bdy = 2 * d * g ** (d - 1) * fields * qf ** (d - 1)
    return dict(G=G, W=fields * case["M"], n=G * fields * case["M"], m_int=m_int, m_iface=m_iface,
                m=m_int + m_iface + m_bdy)


def _vec(count, seed, tag, scale=1.0):
    g = torch.Generator(device="cpu").manual_seed(7919 * (int(seed) + 1) + tag)
    return (scale * torch.randn(count, dtype=torch.float64, generator=g)).cuda()


def _coeffs(case, seed):
    """Coefficients of a function of order one (an iterate of the solver)."""
    return _vec(_sizes(case)["n"], seed, 1, 1.0 / math.sqrt(case["M"]))


def _rhs(case, seed):
    z = _sizes(case)
    r = _vec(z["m"], seed, 2)
    r[z["m_int"]:z["m_int"] + z["m_iface"]] = 0.0
    return r


def _direction(case, seed):
    """A step that takes the iterate past the minimum of the residual."""
    c = _coeffs(case, seed)
    return -1.3 * c + _vec(c.numel(), seed, 3, 0.02 / math.sqrt(case["M"]))


def _triangular(n, seed):
    """Upper-triangular factor with a dominant diagonal, column-major."""
    g = torch.Generator(device="cuda").manual_seed(31 * int(seed) + 5)
    R = torch.randn(n, n, dtype=torch.float64, device="cuda", generator=g).tril_() / n ** 0.5
    R.diagonal().add_(2.0)
    return R  # lower triangle in row-major order: R^T, that is R in column-major order


def prepare(case, seed):
    op = case["op"]
    gp = rfm.Problem(_desc(case, seed))
    st = dict(case=case, gp=gp)
    if op == "solve":
        st["opts"] = W.solve_opts(precision=case["precision"])
        st["X"] = torch.as_tensor(W.eval_grid(gp.desc), device="cuda")
        return st
    if op == "trsv":
        gp.rfm_set_r(_triangular(gp.n, seed))
        st["b"], st["bt"] = _vec(gp.n, seed, 4), _vec(gp.n, seed, 5)
        return st
    gp.rfm_set_rhs(_rhs(case, seed))
    c = st["c"] = _coeffs(case, seed)
    if op == "assemble":
        return st
    F, _ = gp.rfm_assemble(c, C_SCALE)
    if op == "products":
        st["x"], st["y"] = _vec(gp.n, seed, 4), _vec(gp.m, seed, 5)
        return st
    if op == "linesearch":
        st["d"] = _direction(case, seed)
        st["f0"] = gp.rfm_residual(c)[1]
        return st
    gp.rfm_set_precision(case["precision"])
    st["s"], st["kJ"] = _sketch_rows(case, gp.n), int(seed) % 5
    if op == "lsqr":
        gp.rfm_sketch(case["sketch"], st["s"], st["kJ"], copy_out=False)
        gp.rfm_qr(copy_out=False)
        st["b"] = -F
    return st


def run(st):
    gp, op = st["gp"], st["case"]["op"]
    if op == "solve":
        # The solution is u; the coefficient vector that represents it is not
        # determined to the working precision (cond(J) ~ 1e9), so u is returned
        # on the evaluation grid, with the iteration counts and the residual.
        fn = gp.rfm_ipn_solve if st["case"]["solver"] == "ipn" else gp.rfm_amipn_solve
        c, info = fn(st["opts"])
        return dict(u=gp.rfm_eval(c, st["X"]), outer_iters=info["outer_iters"], n_jac=info["n_jac"],
                    lsqr_iters=info["lsqr_iters_total"], status=info["status"], resid=info["final_resid"])
    if op == "assemble":
        F, lam = gp.rfm_assemble(st["c"], C_SCALE)
        Jp, Js, blk = gp.rfm_get_jacobian()
        return dict(F=F, lam=lam, Jp=Jp, Js=Js, blk=blk)
    if op == "products":
        return dict(Jx=gp.rfm_jmv(st["x"], 0), Jty=gp.rfm_jmv(st["y"], 1))
    if op == "linesearch":
        alpha, f = gp.rfm_linesearch(st["c"], st["d"], st["f0"])
        return dict(alpha=alpha, f=f)
    if op == "trsv":
        return dict(x=gp.rfm_trsv(st["b"], 0), xt=gp.rfm_trsv(st["bt"], 1))
    if op == "lsqr":
        d, itn, istop = gp.rfm_lsqr(st["b"])
        return dict(d=d, itn=itn, istop=istop)
    kind = st["case"]["sketch"]
    if op == "sketch":
        return dict(B=gp.rfm_sketch(kind, st["s"], st["kJ"]))
    gp.rfm_sketch(kind, st["s"], st["kJ"], copy_out=False)
    R, low = gp.rfm_qr()
    return dict(R=R, rank_low=low)


def work(case):
    """Bytes of the inputs and outputs of a pass, and the FP64 operations of the
    step's own formulas (30 per feature for a tanh and its row entry)."""
    op, z = case["op"], _sizes(case)
    m, n, nnz = z["m"], z["n"], (z["m"] + z["m_iface"]) * z["W"]
    if op == "assemble":  # F, lambda and J written twice over: assembled, then read out
        return dict(bytes=8.0 * (3 * nnz + 2 * m + n), flops=30.0 * nnz)
    if op == "products":
        return dict(bytes=8.0 * (2 * nnz + 2 * m + 2 * n), flops=4.0 * nnz)
    if op == "linesearch":
        return dict(bytes=8.0 * (2 * n + 8 * m), flops=30.0 * nnz)
    if op == "trsv":
        return dict(bytes=8.0 * (n * (n + 1.0) + 4 * n), flops=2.0 * n * n)
    s = _sketch_rows(case, n) if op != "solve" else 3 * n
    sk = 2.0 * nnz * (s if case.get("sketch") == "gauss" else 1)
    if op == "sketch":
        return dict(bytes=8.0 * (nnz + 2.0 * s * n), flops=sk)
    qr = 2.0 * n * n * (s - n / 3.0)
    if op == "precond":
        return dict(bytes=8.0 * (nnz + s * n + 1.5 * n * n), flops=qr + sk)
    step = 4.0 * nnz + 2.0 * n * n  # an LSQR step: both products, both solves
    if op == "lsqr":
        return dict(bytes=8.0 * 35 * (2.0 * nnz + n * n), flops=35 * step)
    return dict(bytes=8.0 * 4 * (nnz + s * n + 25.0 * (2.0 * nnz + n * n)), flops=4 * (qr + 30.0 * nnz + 25 * step))


# -------------------------------------------- the same in plain FP64 torch / numpy
_M32 = 0xFFFFFFFF


def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 on int64 tensors (32-bit words)."""
    k0, k1 = seed & _M32, (seed >> 32) & _M32
    for r in range(10):
        if r:
            k0, k1 = (k0 + 0x9E3779B9) & _M32, (k1 + 0xBB67AE85) & _M32
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57  # modulo 2^64: the bits are the same
        c0, c1, c2, c3 = ((p1 >> 32) & _M32) ^ c1 ^ k0, p1 & _M32, ((p0 >> 32) & _M32) ^ c3 ^ k1, p0 & _M32
    return c0, c1, c2, c3


def _u53(a, b):
    return ((a >> 5) * 67108864 + (b >> 6)).double() * 2.0 ** -53


def _features(desc, G):
    count, d = G * desc["fields"] * desc["M"], desc["dim"]
    i = torch.arange(count, dtype=torch.int64, device="cuda")
    vals = []
    for r in range((d + 2) // 2):
        x = _philox(torch.zeros_like(i), i, torch.full_like(i, r), torch.zeros_like(i), desc["seed"])
        vals += [_u53(x[0], x[1]), _u53(x[2], x[3])]
    v = desc["feat_range"] * (2.0 * torch.stack(vals[:d + 1], 1) - 1.0)
    return v.view(G, desc["fields"], desc["M"], d + 1)


def _segments(case):
    """Runs of rows that share subdomains: (type, e0, e1, axis, order, field,
    points), in row order; type 0 interior, 1 interface, 2 boundary."""
    d, g, q, qf = case["dim"], case["g"], case["q"], case["qf"]
    fields = 2 if case["kind"] == 1 else 1
    line = lambda j, k: j / g + (np.arange(k) / (k - 1)) / g  # noqa: E731
    grid = lambda axes: np.stack([a.reshape(-1) for a in np.meshgrid(*axes, indexing="ij")], 1)  # noqa: E731
    cells = [tuple(int(v) for v in np.unravel_index(e, (g,) * d)) for e in range(g ** d)]
    out = []
    for e, idx in enumerate(cells):
        P = grid([line(j, q) for j in idx])
        out += [(0, e, -1, -1, 0, f, P) for f in range(fields)]

    def face(idx, a, x):
        axes = [line(j, qf) for j in idx]
        axes[a] = np.array([x])
        return grid(axes)

    for a in range(d):
        for e, idx in enumerate(cells):
            if idx[a] + 1 < g:
                e2 = int(np.ravel_multi_index([j + (b == a) for b, j in enumerate(idx)], (g,) * d))
                P = face(idx, a, (idx[a] + 1) / g)
                out += [(1, e, e2, a, s, f, P) for f in range(fields) for s in (0, 1)]
    for a in range(d):
        for side in (0, 1):
            for e, idx in enumerate(cells):
                if idx[a] == (0 if side == 0 else g - 1):
                    out += [(2, e, -1, a, 0, f, face(idx, a, float(side))) for f in range(fields)]
    return out


class _System:
    """F and J of a case in FP64, row block by row block."""

    def __init__(self, case, seed):
        self.case, self.desc, self.z = case, _desc(case, seed), _sizes(case)
        self.d, self.g, self.kind, self.p = case["dim"], case["g"], case["kind"], self.desc["pde_params"]
        self.feat = _features(self.desc, self.z["G"])
        self.cells = [np.unravel_index(e, (self.g,) * self.d) for e in range(self.z["G"])]
        self.segs = [(*s[:6], torch.as_tensor(s[6], device="cuda")) for s in _segments(case)]
        self.rhs = _rhs(case, seed) if case["op"] != "solve" else None

    def _phi(self, e, f, X):
        k, b = self.feat[e, f, :, :self.d], self.feat[e, f, :, self.d]
        h = 0.5 / self.g
        mu = torch.as_tensor([(j + 0.5) / self.g for j in self.cells[e]], dtype=torch.float64, device="cuda")
        t = torch.tanh(((X - mu) / h) @ k.T + b)
        return t, 1.0 - t * t, k / h

    def _interior(self, e, f, X, c, want_j):
        """(F without the source, J rows [r, W])"""
        M, p, kind = self.case["M"], self.p, self.kind
        t, s1, k = self._phi(e, f, X)
        lap = -2.0 * t * s1 * (k * k).sum(1)
        cf = c[e, f]
        if kind == 1:
            o = 1 - f
            to = self._phi(e, o, X)[0]
            own, oth = t @ cf, to @ c[e, o]
            u, v = (own, oth) if f == 0 else (oth, own)
            lin = -p[f] * lap
            Fc, kk = p[2], p[3]
            if f == 0:
                R, du, dv = lin @ cf + u * v * v - Fc * (1.0 - u), v * v + Fc, 2.0 * u * v
            else:
                R, du, dv = lin @ cf - u * v * v + (Fc + kk) * v, -v * v, Fc + kk - 2.0 * u * v
            if not want_j:
                return R, None
            J = torch.empty(X.shape[0], 2 * M, dtype=torch.float64, device="cuda")
            t0, t1 = (t, to) if f == 0 else (to, t)
            J[:, :M], J[:, M:] = du[:, None] * t0, dv[:, None] * t1
            J[:, f * M:(f + 1) * M] += lin
            return R, J
        u = t @ cf
        if kind in (0, 2, 3):
            if kind == 0:
                lin = -lap
            else:
                a = 1.0 + 0.5 * torch.sin(2 * math.pi * X[:, 0])
                ax = math.pi * torch.cos(2 * math.pi * X[:, 0])
                lin = -a[:, None] * lap - ax[:, None] * (s1 * k[:, 0])
            R = lin @ cf + p[0] * u ** 3
            return R, lin + (3.0 * p[0] * u * u)[:, None] * t if want_j else None
        if kind == 4:
            return lap @ cf + p[0] * u + p[1] * torch.cosh(u), \
                lap + (p[0] + p[1] * torch.sinh(u))[:, None] * t if want_j else None
        h = -2.0 * t * s1
        gu = (s1 * cf) @ k                                  # grad u
        Hu = torch.einsum("rm,ma,mb->rab", h * cf, k, k)    # Hess u
        lu, gg = lap @ cf, (gu * gu).sum(1)
        gphi = s1 * (gu @ k.T)                              # grad u . grad phi_j
        if kind == 5:
            R = -(1.0 + u * u) * lu - 2.0 * u * gg
            J = -(1.0 + u * u)[:, None] * lap - (2.0 * u * lu + 2.0 * gg)[:, None] * t - (4.0 * u)[:, None] * gphi
            return R, J if want_j else None
        Hg = torch.einsum("rab,rb->ra", Hu, gu)
        R = -(1.0 + gg) * lu - 2.0 * (gu * Hg).sum(1)
        J = -(1.0 + gg)[:, None] * lap - (2.0 * lu)[:, None] * gphi - 4.0 * s1 * (Hg @ k.T) - 2.0 * h * (gu @ k.T) ** 2
        return R, J if want_j else None

    def rows(self, c, want_j=True):
        """Unscaled F [m], and Jp [m, W], Js [m_iface, W] with their row maxima."""
        z, M = self.z, self.case["M"]
        c = c.view(z["G"], -1, M)
        F = torch.empty(z["m"], dtype=torch.float64, device="cuda")
        Jp = torch.zeros(z["m"], z["W"], dtype=torch.float64, device="cuda") if want_j else None
        Js = torch.zeros(z["m_iface"], z["W"], dtype=torch.float64, device="cuda") if want_j else None
        r0 = 0
        for typ, e0, e1, ax, order, f, X in self.segs:
            sl = slice(r0, r0 + X.shape[0])
            r0 = sl.stop
            if typ == 0:
                F[sl], J = self._interior(e0, f, X, c, want_j)
                if want_j:
                    Jp[sl] = J
                continue
            tot = 0.0
            for side, e in enumerate([e0, e1] if typ == 1 else [e0]):
                t, s1, k = self._phi(e, f, X)
                v = (t if order == 0 else s1 * k[:, ax]) * (1.0 - 2.0 * side)
                tot = tot + v @ c[e, f]
                if want_j and side == 0:
                    Jp[sl, f * M:(f + 1) * M] = v
                elif want_j:
                    Js[sl.start - z["m_int"]:sl.stop - z["m_int"], f * M:(f + 1) * M] = v
            F[sl] = tot
        return F - self.rhs, Jp, Js

    def scaled(self, c):
        F, Jp, Js = self.rows(c)
        z = self.z
        mx = Jp.abs().amax(1)
        fa = slice(z["m_int"], z["m_int"] + z["m_iface"])
        if z["m_iface"]:
            mx[fa] = torch.maximum(mx[fa], Js.abs().amax(1))
        lam = torch.where(mx > 0, C_SCALE / mx, torch.ones_like(mx))
        return lam * F, lam, Jp.mul_(lam[:, None]), Js.mul_(lam[fa][:, None])

    def blocks(self, Jp, Js):
        """Per subdomain: the rows touching it and their entries in its columns."""
        e0 = torch.cat([torch.full((s[6].shape[0],), s[1], device="cuda") for s in self.segs])
        e1 = torch.cat([torch.full((s[6].shape[0],), s[2], device="cuda") for s in self.segs])
        m0 = self.z["m_int"]
        for b in range(self.z["G"]):
            r, r2 = torch.nonzero(e0 == b)[:, 0], torch.nonzero(e1 == b)[:, 0]
            yield b, torch.cat([r, r2]), torch.cat([Jp[r], Js[r2 - m0]])


def _gauss_columns(s, rows, kJ, seed):
    """Columns `rows` of the Gaussian sketch, [s, len(rows)]."""
    q = torch.arange(s // 2, dtype=torch.int64, device="cuda")[:, None].expand(s // 2, rows.numel())
    i = rows[None, :].expand_as(q)
    x = _philox(torch.full_like(q, 2), i, q, torch.full_like(q, kJ), seed)
    rad = torch.sqrt(-2.0 * torch.log(1.0 - _u53(x[0], x[1])))
    th = 6.283185307179586 * _u53(x[2], x[3])
    out = torch.empty(s, rows.numel(), dtype=torch.float64, device="cuda")
    out[0::2], out[1::2] = rad * torch.cos(th), rad * torch.sin(th)
    return torch.round(16.0 * out) / 16.0


def _sketch(sysm, case, Jp, Js, s, kJ):
    """B [s, n]"""
    z = sysm.z
    B = torch.zeros(s, z["n"], dtype=torch.float64, device="cuda")
    i = torch.arange(z["m"], dtype=torch.int64, device="cuda")
    o = torch.ones_like(i)
    x = _philox(o, i, o * kJ, o * 0, sysm.desc["seed"])
    bucket, sign = (x[0] * s) >> 32, 1.0 - 2.0 * (x[1] & 1).double()
    for b, rows, J in sysm.blocks(Jp, Js):
        cols = slice(b * z["W"], (b + 1) * z["W"])
        if case["sketch"] == "count":
            B[:, cols] = torch.zeros(s, z["W"], dtype=torch.float64, device="cuda").index_add_(
                0, bucket[rows], sign[rows][:, None] * J)
        else:
            for r in range(0, rows.numel(), 512):
                B[:, cols] += _gauss_columns(s, rows[r:r + 512], kJ, sysm.desc["seed"]) @ J[r:r + 512]
    return B


def _qr_r(B):
    R = torch.linalg.qr(B, mode="r")[1]
    return R * torch.where(R.diagonal() < 0, -1.0, 1.0)[:, None]


def _lsqr(mv, rmv, b, n, eta=1e-6, conlim=1e8):
    """LSQR of Paige and Saunders, x_0 = 0, no damping."""
    nrm = lambda v: float(torch.linalg.vector_norm(v))  # noqa: E731
    x = torch.zeros(n, dtype=torch.float64, device="cuda")
    beta = nb = nrm(b)
    u = b / beta
    v = rmv(u)
    alpha = nrm(v)
    v = v / alpha
    w, phibar, rhobar, sumsq, dd = v, beta, alpha, 0.0, 0.0
    for _ in range(2 * n):
        u = mv(v) - alpha * u
        beta = nrm(u)
        u = u / beta
        sumsq += alpha * alpha + beta * beta
        v = rmv(u) - beta * v
        alpha = nrm(v)
        v = v / alpha
        rho = math.hypot(rhobar, beta)
        c, s = rhobar / rho, beta / rho
        rhobar, phi, phibar, theta = -c * alpha, c * phibar, s * phibar, s * alpha
        dk = w / rho
        x, w = x + phi * dk, v - (theta / rho) * w
        dd += nrm(dk) ** 2
        nA = math.sqrt(sumsq)
        if phibar <= eta * nb + eta * nA * nrm(x) or alpha * abs(c) <= eta * nA or nA * math.sqrt(dd) >= conlim:
            break
    return x


def _golden(phi, f0):
    k = (math.sqrt(5.0) - 1.0) / 2.0
    a, b = 0.0, 1.0
    x1, x2 = b - k * (b - a), a + k * (b - a)
    f1, f2 = phi(x1), phi(x2)
    got = [(x1, f1), (x2, f2)]
    while b - a > 1e-3:
        if f1 < f2:
            b, x2, f2 = x2, x1, f1
            x1 = b - k * (b - a)
            f1 = phi(x1)
            got.append((x1, f1))
        else:
            a, x1, f1 = x1, x2, f2
            x2 = a + k * (b - a)
            f2 = phi(x2)
            got.append((x2, f2))
    got.append((1.0, phi(1.0)))
    low = min(f for _, f in got)
    best = max(x for x, f in got if f <= low * (1.0 + 1e-12))
    f = min(f for x, f in got if x == best)
    return (best, f) if f < f0 else (0.0, f0)


def exact(case, seed):
    op = case["op"]
    if op == "solve":
        return None  # an iteration stopped by its tolerance: no value of its own
    z = _sizes(case)
    if op == "trsv":
        Rt = _triangular(z["n"], seed)  # R^T, lower triangular
        b, bt = _vec(z["n"], seed, 4)[:, None], _vec(z["n"], seed, 5)[:, None]
        return dict(x=torch.linalg.solve_triangular(Rt.T, b, upper=True)[:, 0],
                    xt=torch.linalg.solve_triangular(Rt, bt, upper=False)[:, 0])
    if op == "precond" and work(case)["flops"] > 4e12:
        return None  # 20 s and more with a library's QR in FP64
    sysm = _System(case, seed)
    c = _coeffs(case, seed)
    F, lam, Jp, Js = sysm.scaled(c)
    if op == "assemble":
        return dict(F=F, lam=lam, Jp=Jp, Js=Js, blk=None)
    if op == "products":
        x, y = _vec(z["n"], seed, 4), _vec(z["m"], seed, 5)
        Jx, Jty = torch.zeros_like(y), torch.zeros_like(x)
        for b, rows, J in sysm.blocks(Jp, Js):
            cols = slice(b * z["W"], (b + 1) * z["W"])
            Jx.index_add_(0, rows, J @ x[cols])
            Jty[cols] = J.T @ y[rows]
        return dict(Jx=Jx, Jty=Jty)
    if op == "linesearch":
        d = _direction(case, seed)
        phi = lambda a: float(torch.linalg.vector_norm(lam * sysm.rows(c + a * d, False)[0]))  # noqa: E731
        alpha, f = _golden(phi, phi(0.0))
        return dict(alpha=alpha, f=f)
    s, kJ = _sketch_rows(case, z["n"]), int(seed) % 5
    B = _sketch(sysm, case, Jp, Js, s, kJ)
    if op == "sketch":
        return dict(B=B.T.contiguous())
    R = _qr_r(B)
    if op == "precond":
        return dict(R=R.T.contiguous(), rank_low=None)
    J = torch.zeros(z["m"], z["n"], dtype=torch.float64, device="cuda")
    for b, rows, Jb in sysm.blocks(Jp, Js):
        J[rows, b * z["W"]:(b + 1) * z["W"]] = Jb
    sol = lambda v: torch.linalg.solve_triangular(R, v[:, None], upper=True)[:, 0]  # noqa: E731
    solt = lambda v: torch.linalg.solve_triangular(R.T, v[:, None], upper=False)[:, 0]  # noqa: E731
    y = _lsqr(lambda v: J @ sol(v), lambda u: solt(J.T @ u), -F, z["n"])
    return dict(d=sol(y), itn=None, istop=None)
