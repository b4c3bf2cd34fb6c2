"""What a user of this framework has it do, as timed cases.

A case is a dict of plain values; ``prepare`` makes its inputs and what a
program keeps (a factorization, for the calls that reuse one), ``run`` is one
pass through the public entry points, ``work`` the bytes and operations that
the pass cannot do without, and ``exact`` the same outputs from plain torch in
64 bits.  Four kinds of pass:

- ``factor``: a new factorization and a solve refined against the direct sum,
  what a program does for each new set of coefficients (Helmholtz and batches
  of independent problems among them);
- ``sweep``: one application of F, F^T, F^-1 or F^-T of a kept factorization,
  the fast apply and the preconditioner of a user's own iteration;
- ``matvec``: the direct sum A x or A^T x, the residual operator;
- ``adjoint``: forward and backward of the autograd solve on a kept
  factorization, one step of an optimization over f, a, b and c.

Sizes are those of the configurations, tests and benchmark of this repository
(n = 64, 256, 512 and 1024 in 2D; batches of n = 32, 48, ..., 256; 3D grids)
and ragged ones between them.  Factorizations in 32 bits are always followed by
refinement: they are not meant to be used without it.
"""
import math

import numpy as np
import torch

from paper_1307_2666_gb300 import Factorization, HIFSolve

# bytes of factors per unknown that a sweep has to read once: factor_bytes / N
# of the symmetric 64-bit factorization at N = 4,096 and eps = 1e-6 (2,210);
# larger and unsymmetric problems hold up to 7,800, explicit inverses included
FACTOR_BYTES = 2200


def listed():
    return [
        # the smallest whole call: one right-hand side on a 64 x 64 grid, unit coefficients
        dict(name="factor_n64", kind="factor", dim=2, n=64, eps=1e-6, precision="fp64", nrhs=1, coef="one",
             jitter=0.0, trans=False, method="ir", tol=1e-10),
        # the benchmark: a million unknowns, 32-bit factorization, 8 right-hand sides to 1e-10
        dict(name="factor_n1024_fp32", kind="factor", dim=2, n=1024, eps=1e-6, precision="fp32", nrhs=8,
             coef="smooth", jitter=0.0, trans=False, method="ir", tol=1e-10),
        # an ordinary unsymmetric system (b != c) of ragged size, adjoint solve by GMRES
        dict(name="factor_n200_general", kind="factor", dim=2, n=200, eps=1e-6, precision="fp64", nrhs=2,
             coef="general", jitter=0.0, trans=True, method="gmres", tol=1e-10),
        # a 3D volume equation: cells, faces and edges
        dict(name="factor_3d_n32", kind="factor", dim=3, n=32, eps=1e-3, precision="fp32", nrhs=16, coef="smooth",
             jitter=0.0, trans=False, method="ir", tol=1e-10),
        # many small and middling problems at once, uneven sizes
        dict(name="factor_batch24", kind="batch", dim=2, n=256, count=24, size_seed=1004, eps=1e-6, precision="fp32",
             nrhs=4, coef="smooth", tol=1e-10),
        # scattering: the complex kernel, two wavelengths across the square, GMRES to 1e-12
        dict(name="helmholtz_n64", kind="helmholtz", dim=2, n=64, kappa=2.0, eps=1e-6, precision="fp64", nrhs=1,
             tol=1e-12),
        # one gradient step through the solver at high accuracy
        dict(name="adjoint_n256", kind="adjoint", dim=2, n=256, eps=1e-9, precision="fp64", nrhs=1, coef="smooth",
             tol=1e-12),
        # the preconditioner inside a user's own iteration: smallest call, and a block of vectors on a large grid
        dict(name="solve_n64", kind="sweep", dim=2, n=64, eps=1e-6, precision="fp64", nrhs=1, coef="smooth",
             op="solve"),
        dict(name="solve_n512", kind="sweep", dim=2, n=512, eps=1e-6, precision="fp64", nrhs=8, coef="smooth",
             op="solve"),
        # the fast apply of an unsymmetric operator, transposed, odd number of vectors
        dict(name="apply_t_n200_general", kind="sweep", dim=2, n=200, eps=1e-6, precision="fp64", nrhs=3,
             coef="general", op="apply_transpose"),
        # the residual operator on a grid and on scattered points
        dict(name="matvec_n512", kind="matvec", dim=2, n=512, nrhs=8, coef="smooth", jitter=0.0, trans=False),
        dict(name="matvec_scattered_16k", kind="matvec", dim=2, n=128, nrhs=2, coef="general", jitter=0.2,
             trans=True),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["factor", "factor", "factor", "batch", "helmholtz", "adjoint", "sweep", "sweep", "matvec",
                       "matvec"])
    coef = rng.choice(["smooth", "smooth", "general"])
    if kind == "factor":
        dim = rng.choice([2, 2, 3])
        precision = rng.choice(["fp32", "fp64"])
        jitter = rng.choice([0.0, 0.0, 0.2])
        hi = 112 if jitter else 640 if precision == "fp32" else 256
        n = _log(rng, 24, hi) if dim == 2 else _log(rng, 10, 24)
        return dict(kind="factor", dim=dim, n=n, eps=rng.choice([1e-3, 1e-4] if dim == 3 else [1e-4, 1e-6, 1e-8]),
                    precision=precision, nrhs=rng.randint(1, 17), coef=coef, jitter=jitter if dim == 2 else 0.0,
                    trans=rng.random() < 0.3, method=rng.choice(["ir", "ir", "gmres"]), tol=1e-10)
    if kind == "batch":
        return dict(kind="batch", dim=2, n=_log(rng, 64, 256), count=rng.randint(2, 24),
                    size_seed=rng.randrange(1 << 20), eps=1e-6, precision=rng.choice(["fp32", "fp32", "fp64"]),
                    nrhs=rng.randint(1, 5), coef=coef, tol=1e-10)
    if kind == "helmholtz":
        n = _log(rng, 24, 80)
        return dict(kind="helmholtz", dim=2, n=n, kappa=round(n / 32.0, 3), eps=rng.choice([1e-4, 1e-6]),
                    precision="fp64", nrhs=rng.randint(1, 2), tol=1e-12)
    if kind == "adjoint":
        return dict(kind="adjoint", dim=2, n=_log(rng, 48, 256), eps=1e-9, precision="fp64", nrhs=1, coef=coef,
                    tol=1e-12)
    if kind == "sweep":
        dim = rng.choice([2, 2, 2, 3])
        n = _log(rng, 32, 512) if dim == 2 else _log(rng, 10, 24)
        return dict(kind="sweep", dim=dim, n=n, eps=1e-6 if dim == 2 else 1e-3, precision="fp64",
                    nrhs=rng.choice([1, 1, 2, 5, 8, 13, 16]), coef=coef,
                    op=rng.choice(["solve", "solve_transpose", "apply", "apply_transpose"]))
    jitter = rng.choice([0.0, 0.0, 0.2])
    dim = rng.choice([2, 2, 3])
    n = (_log(rng, 40, 512) if dim == 2 else _log(rng, 10, 56)) if not jitter else \
        (_log(rng, 24, 128) if dim == 2 else _log(rng, 8, 24))
    return dict(kind="matvec", dim=dim, n=n, nrhs=rng.choice([1, 2, 5, 8, 16]), coef=coef, jitter=jitter,
                trans=rng.random() < 0.4)


# ---- inputs ------------------------------------------------------------------

def _grid(n, dim):
    h = 1.0 / n
    g = (torch.arange(n, dtype=torch.float64, device="cuda") + 0.5) * h
    mesh = torch.meshgrid(*([g] * dim), indexing="ij")
    pts = torch.stack([m.reshape(-1) for m in mesh], dim=1).contiguous()
    return pts, torch.full((n ** dim,), h ** dim, dtype=torch.float64, device="cuda")


def _field(pts, rng, terms=16, kmax=4):
    """1 + 0.5 phi, phi the mean of 16 random-phase cosines."""
    dim = pts.shape[1]
    ks = []
    while len(ks) < terms:
        k = rng.integers(-kmax, kmax + 1, size=dim)
        if np.any(k != 0):
            ks.append(k)
    k = torch.as_tensor(np.asarray(ks, dtype=np.float64), device="cuda")
    theta = torch.as_tensor(rng.uniform(0.0, 2.0 * math.pi, size=terms), device="cuda")
    phi = torch.zeros(pts.shape[0], dtype=torch.float64, device="cuda")
    for j in range(terms):
        phi += torch.cos(2.0 * math.pi * (pts * k[j]).sum(dim=1) + theta[j])
    return 1.0 + (0.5 / terms) * phi


def _vectors(N, nrhs, seed, dtype=torch.float64):
    """Standard normal vectors, column-major as the library takes them."""
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    if dtype.is_complex:
        x = torch.randn(nrhs, N, 2, dtype=torch.float64, device="cuda", generator=gen)
        return torch.view_as_complex(x).t()
    return torch.randn(nrhs, N, dtype=torch.float64, device="cuda", generator=gen).t()


def _problem(n, dim, coef, jitter, rng):
    pts, w = _grid(n, dim)
    if jitter:
        shift = torch.as_tensor(rng.uniform(-jitter, jitter, size=(n ** dim, dim)) / n, device="cuda")
        pts = (pts + shift).contiguous()
    a = torch.ones(n ** dim, dtype=torch.float64, device="cuda")
    b = torch.ones_like(a) if coef == "one" else _field(pts, rng)
    c = _field(pts, rng) if coef == "general" else b.clone()
    return pts, w, a, b, c


def _proxy(dim):
    if dim == 2:
        return None
    g = np.random.default_rng(7).standard_normal((512, 3))
    return g / np.linalg.norm(g, axis=1, keepdims=True)


def _sizes(case):
    choices = list(range(32, case["n"] + 1, 16))
    idx = np.random.default_rng(case["size_seed"]).integers(0, len(choices), size=case["count"])
    return [choices[i] for i in idx]


def _inputs(case, seed):
    rng = np.random.default_rng([int(seed) & 0x7FFFFFFF, 1])
    kind, n, dim = case["kind"], case["n"], case["dim"]
    s = {"case": case}
    if kind == "batch":
        s["problems"] = [_problem(m, 2, case["coef"], 0.0, rng) for m in _sizes(case)]
        s["f"] = _vectors(sum(p[0].shape[0] for p in s["problems"]), case["nrhs"], seed)
        return s
    if kind == "helmholtz":
        pts, w = _grid(n, 2)
        centre = torch.as_tensor(0.5 + rng.uniform(-0.05, 0.05, size=2), device="cuda")
        k = 2.0 * math.pi * case["kappa"]
        b = k * torch.exp(-16.0 * ((pts - centre) ** 2).sum(dim=1))
        s["problem"] = (pts, w, torch.ones_like(w), b, b.clone())
        s["wavenumber"] = k
        s["f"] = _vectors(n * n, case["nrhs"], seed, torch.complex128)
        return s
    s["problem"] = _problem(n, dim, case["coef"], case.get("jitter", 0.0), rng)
    s["proxy"] = _proxy(dim)
    f = _vectors(n ** dim, case["nrhs"], seed)
    if kind == "adjoint":
        s["f"], s["target"] = f[:, 0].contiguous(), _vectors(n ** dim, 1, seed + 1)[:, 0].contiguous()
    else:
        s["f"] = f
    return s


def prepare(case, seed):
    s = _inputs(case, seed)
    kid = 0 if case["dim"] == 2 else 1
    if case["kind"] in ("sweep", "adjoint"):
        s["fac"] = Factorization(*s["problem"], kid, case["eps"], precision=case["precision"],
                                 proxy_dirs=s["proxy"])
    elif case["kind"] == "matvec":      # the sum does not depend on the factorization
        s["fac"] = Factorization(*s["problem"], kid, 1e-2, precision="fp32", proxy_dirs=s["proxy"])
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "sweep":
        return getattr(s["fac"], case["op"])(s["f"])
    if kind == "matvec":
        return s["fac"].matvec(s["f"], trans=case["trans"])
    if kind == "adjoint":
        leaves = [s["f"], *s["problem"][2:]]
        leaves = [x.detach().requires_grad_(True) for x in leaves]
        u = HIFSolve.apply(*leaves, s["fac"], case["tol"])
        grads = torch.autograd.grad(0.5 * ((u - s["target"]) ** 2).sum(), leaves)
        return [u.detach(), *grads]
    if kind == "batch":
        fac = Factorization.batched(s["problems"], 0, case["eps"], precision=case["precision"])
        u, _, _ = fac.solve_refined(s["f"], tol=case["tol"])
    elif kind == "helmholtz":
        fac = Factorization(*s["problem"], 2, case["eps"], precision=case["precision"], wavenumber=s["wavenumber"])
        u, _, _ = fac.solve_refined(s["f"], tol=case["tol"], method="gmres")
    else:
        fac = Factorization(*s["problem"], 0 if case["dim"] == 2 else 1, case["eps"], precision=case["precision"],
                            proxy_dirs=s["proxy"])
        u, _, _ = fac.solve_refined(s["f"], trans=case["trans"], tol=case["tol"], method=case["method"])
    fac.close()
    return u


def work(case):
    """Inputs read and outputs written once; the operations of one direct sum
    where the pass contains one (a refined solve measures its residual at
    least once, an adjoint step twice); a sweep reads the factors once."""
    kind, nrhs, dim = case["kind"], case["nrhs"], case["dim"]
    sizes = [m ** 2 for m in _sizes(case)] if kind == "batch" else [case["n"] ** dim]
    N = sum(sizes)
    vec = 16 if kind == "helmholtz" else 8
    data = 8 * N * (dim + 4)
    if kind == "sweep":
        return {"bytes": FACTOR_BYTES * N + 2 * vec * N * nrhs, "flops": 0.25 * FACTOR_BYTES * N * nrhs}
    pair = 8.0 if kind == "helmholtz" else 2.0
    flops = pair * sum(float(m) ** 2 for m in sizes) * nrhs * (2 if kind == "adjoint" else 1)
    out = 2 * vec * N * nrhs
    if kind == "adjoint":
        out += 8 * N * 8 + 2 * FACTOR_BYTES * N
    return {"bytes": data + out, "flops": flops}


# ---- the same outputs in 64 bits, from plain torch -------------------------

def _self_term(h, dim):
    if dim == 2:
        return -(h * h / (2.0 * math.pi)) * (math.log(h) - 0.5 * math.log(2.0) - 1.5 + 0.25 * math.pi)
    return (h * h / (4.0 * math.pi)) * (3.0 * math.log(2.0 + math.sqrt(3.0)) - 0.5 * math.pi)


def _green(r2, dim):
    return -torch.log(r2) / (4.0 * math.pi) if dim == 2 else 1.0 / (4.0 * math.pi * torch.sqrt(r2))


class _GridSum:
    """K v on the uniform grid by zero-padded FFT convolution."""

    def __init__(self, n, dim):
        h = 1.0 / n
        off = torch.arange(2 * n, dtype=torch.float64, device="cuda")
        off = torch.where(off < n, off, off - 2 * n)
        r2 = sum(o ** 2 for o in torch.meshgrid(*([off] * dim), indexing="ij")) * (h * h)
        r2.reshape(-1)[0] = 1.0
        t = _green(r2, dim) * h ** dim
        t.reshape(-1)[0] = _self_term(h, dim)
        self.n, self.dim, self.axes = n, dim, tuple(range(dim))
        self.ft = torch.fft.rfftn(t, dim=self.axes)

    def __call__(self, v):
        full = [2 * self.n] * self.dim
        y = torch.fft.irfftn(self.ft * torch.fft.rfftn(v.reshape([self.n] * self.dim), s=full, dim=self.axes), s=full,
                             dim=self.axes)
        for k in range(self.dim):
            y = y.narrow(k, 0, self.n)
        return y.reshape(-1)


class _PointSum:
    """K v on scattered points, block of rows by block of rows."""

    def __init__(self, pts, w):
        self.pts, self.w, self.dim = pts, w, pts.shape[1]
        self.kself = torch.tensor([_self_term(float(w[0]) ** (1.0 / self.dim), self.dim)], device=pts.device,
                                  dtype=torch.float64)

    def rows(self, i0, i1):
        d = self.pts[i0:i1, None, :] - self.pts[None, :, :]
        r2 = (d * d).sum(dim=2)
        i = torch.arange(i0, i1, device=r2.device)
        r2[i - i0, i] = 1.0
        K = _green(r2, self.dim) * self.w[None, :]
        K[i - i0, i] = self.kself
        return K

    def __call__(self, v):
        N = v.shape[0]
        return torch.cat([self.rows(i, min(N, i + 2048)) @ v for i in range(0, N, 2048)])


def _operator(problem, n, dim, jitter, trans):
    pts, w, a, b, c = problem
    K = _PointSum(pts, w) if jitter else _GridSum(n, dim)
    if trans:                               # all weights are equal, so K is symmetric
        b, c = c, b
    return lambda x: a * x + b * K(c * x)


def _gmres(op, f, tol=1e-14, maxit=120):
    """Plain GMRES with one restart, Gram-Schmidt twice."""
    x = torch.zeros_like(f)
    for _ in range(2):
        r = f - op(x)
        beta = r.norm()
        if float(beta) <= tol * float(f.norm()):
            break
        Q, H = [r / beta], []
        for j in range(maxit):
            v = op(Q[j])
            col = torch.zeros(j + 1, dtype=f.dtype, device=f.device)
            B = torch.stack(Q)
            for _ in range(2):
                g = B.conj() @ v
                v = v - g @ B
                col = col + g
            nv = v.norm()
            H.append((col, nv))
            m = j + 1
            M = torch.zeros(m + 1, m, dtype=f.dtype, device=f.device)
            for q, (h, z) in enumerate(H):
                M[: q + 1, q] = h
                M[q + 1, q] = z
            e = torch.zeros(m + 1, dtype=f.dtype, device=f.device)
            e[0] = beta
            y = torch.linalg.lstsq(M, e[:, None]).solution[:, 0]
            if float((e - M @ y).norm()) <= tol * float(f.norm()) or float(nv) == 0.0:
                break
            Q.append(v / nv)
        x = x + y @ torch.stack(Q[: len(H)])
    return x


def _solve(op, F):
    return torch.stack([_gmres(op, F[:, q].contiguous()) for q in range(F.shape[1])]).t()


def _hankel(x):
    """H_0^(1)(x) by Miller's backward recurrence for J_m and Neumann's series
    Y_0 = (2/pi) (ln(x/2) + gamma) J_0 - (4/pi) sum_m (-1)^m J_2m / m
    (torch's own Bessel functions are good to 1e-7 only)."""
    M = 2 * int(0.75 * float(np.max(x)) + 24)
    up, at = np.zeros_like(x), np.full_like(x, 1e-300)      # J_{m+1}, J_m up to a factor
    norm, series = np.zeros_like(x), np.zeros_like(x)
    for m in range(M, 0, -1):
        if m % 2 == 0:
            norm += 2.0 * at
            series += (1.0 if m % 4 == 0 else -1.0) * at * (2.0 / m)
        up, at = at, (2.0 * m / x) * at - up
        big = np.abs(at) > 1e200
        for v in (up, at, norm, series):
            v[big] *= 1e-200
    norm += at
    j0 = at / norm
    return j0 + 1j * ((2.0 / math.pi) * (np.log(0.5 * x) + np.euler_gamma) * j0 - (4.0 / math.pi) * series / norm)


def _helmholtz_dense(s, case):
    _, w, a, b, c = s["problem"]
    n, k = case["n"], s["wavenumber"]
    h = 1.0 / n
    i, j = np.meshgrid(np.arange(n), np.arange(n), indexing="ij")
    r = h * np.sqrt((i * i + j * j).astype(np.float64))
    r[0, 0] = 1.0
    table = 0.25j * _hankel(k * r) * (h * h)
    # the self term in polar coordinates: eight right triangles, r = R t^2 against the logarithm
    g, gw = np.polynomial.legendre.leggauss(96)
    t, tw = 0.5 * (g + 1.0), 0.5 * gw
    R = 0.5 * h / np.cos(t * (0.25 * math.pi))
    inner = (0.25j * _hankel(k * R[:, None] * t[None, :] ** 2) * (tw * 2.0 * t ** 3)[None, :]).sum(axis=1) * R * R
    table[0, 0] = 8.0 * 0.25 * math.pi * (inner * tw).sum()
    table = torch.as_tensor(table, device="cuda")
    o = torch.arange(n, device="cuda")
    o = (o[:, None] - o[None, :]).abs()
    K = table[o[:, None, :, None], o[None, :, None, :]].reshape(n * n, n * n)
    return torch.diag(a.to(K.dtype)) + b[:, None] * K * c[None, :]


def exact(case, seed):
    s = _inputs(case, seed)
    kind = case["kind"]
    if kind == "helmholtz":
        return torch.linalg.solve(_helmholtz_dense(s, case), s["f"].contiguous())
    if kind == "batch":
        out, at = [], 0
        for m, p in zip(_sizes(case), s["problems"]):
            out.append(_solve(_operator(p, m, 2, 0.0, False), s["f"][at:at + m * m]))
            at += m * m
        return torch.cat(out)
    args = (s["problem"], case["n"], case["dim"], case.get("jitter", 0.0))
    if kind == "adjoint":
        _, _, a, b, c = s["problem"]
        K = _GridSum(case["n"], 2)
        u = _gmres(_operator(*args, False), s["f"])
        lam = _gmres(_operator(*args, True), u - s["target"])
        return [u, lam, -lam * u, -lam * K(c * u), -u * K(b * lam)]
    if kind == "factor":
        return _solve(_operator(*args, case["trans"]), s["f"])
    if kind == "matvec":
        op = _operator(*args, case["trans"])
    else:
        op = _operator(*args, case["op"].endswith("transpose"))
        if case["op"].startswith("solve"):
            return _solve(op, s["f"])
    return torch.stack([op(s["f"][:, q].contiguous()) for q in range(case["nrhs"])]).t()
