"""The work users of this framework have it do, as measurable cases.

Four kinds of pass through the public entry points of paper_1804_02297_gb300, in
3-D (grids n^3: 4 ... 128 and 256, powers of two, 48 and 96) and in 2-D (grids
n x n, any n up to 1024):

  apply    y = A x, or y = Q A x: the operator of every Krylov iteration and residual
  precond  y = S^-1 (Q v): the preconditioner of every Krylov iteration
  solve    the whole preconditioned GMRES solve of A x = g
  setup    stencil fit, assembly and factor of S, then the first preconditioned vector

complex64 is what the iterations run in, complex128 the outer residual and the FP64
solves; one right-hand side is a single incident wave, more are a block of waves.
Media are tapered Gaussian bumps on the unit cube or square, seeded; the wavenumbers
are those of the repository's workloads (about 8 points per wavelength in 3-D, 6 in
2-D).  The stencil tables of Q A are seeded orthonormal ones (Q's cost does not depend
on their values); the preconditioner uses the library's own fit.
"""
import math

import numpy as np
import torch

import paper_1804_02297_gb300 as spm

SIZES_3D = (4, 8, 16, 32, 48, 64, 96, 128, 256)


def listed():
    return [
        # the smallest correctness-size problem, FP64: launches and latency
        dict(name="apply3_n16_c128", kind="apply", dim=3, n=16, prec="c128", nrhs=1, op="QA"),
        # the headline: one operator and Q of a GMRES iteration for one incident wave
        dict(name="apply3_n64_c64", kind="apply", dim=3, n=64, prec="c64", nrhs=1, op="QA"),
        # a block of incident waves through the same operator
        dict(name="apply3_n64_c64_rhs16", kind="apply", dim=3, n=64, prec="c64", nrhs=16, op="QA"),
        # the largest grid: the intermediates leave the L2
        dict(name="apply3_n256_c64", kind="apply", dim=3, n=256, prec="c64", nrhs=1, op="A"),
        # the FP64 residual of an outer step on a radix-3 grid
        dict(name="apply3_n96_c128", kind="apply", dim=3, n=96, prec="c128", nrhs=1, op="A"),
        # the preconditioner of a single-wave iteration: the factor is read once
        dict(name="precond3_n32_c64", kind="precond", dim=3, n=32, prec="c64", nrhs=1),
        # the preconditioner of a block of waves: the factor's bytes serve 16 fields
        dict(name="precond3_n32_c64_rhs16", kind="precond", dim=3, n=32, prec="c64", nrhs=16),
        # the 2-D preconditioner of an FP64 iteration (second size of the paper's 2-D tables)
        dict(name="precond2_n239_c128", kind="precond", dim=2, n=239, prec="c128", nrhs=1),
        # the largest 2-D size of the paper's tables, complex64
        dict(name="apply2_n959_c64", kind="apply", dim=2, n=959, prec="c64", nrhs=1, op="A"),
        # an FP64 iteration's operator and Q at the third size of the 2-D tables
        dict(name="apply2_n479_c128", kind="apply", dim=2, n=479, prec="c128", nrhs=1, op="QA"),
        # a whole 3-D solve as users run it: complex64 iterations, FP64 residuals
        dict(name="solve3_n32_mixed", kind="solve", dim=3, n=32, prec="c64", nrhs=1),
        # set-up of a new medium at the first size of the 2-D tables, FP64
        dict(name="setup2_n119_c128", kind="setup", dim=2, n=119, prec="c128", nrhs=1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["apply", "apply", "apply", "apply", "precond", "precond", "solve", "setup"])
    dim = 2 if kind == "setup" else rng.choice([2, 3])
    if kind == "apply" and dim == 3:
        n = rng.choice(SIZES_3D)
        prec = rng.choice(["c64", "c64", "c128"]) if n <= 96 else "c64"
        most = {256: 1, 128: 4, 96: 4}.get(n, 32)
        op = rng.choice(["A", "QA"]) if n <= 96 else "A"
        return dict(kind=kind, dim=3, n=n, prec=prec, nrhs=_log_int(rng, 1, most), op=op)
    if kind == "apply":
        n, prec = _log_int(rng, 16, 1024), rng.choice(["c64", "c128"])
        return dict(kind=kind, dim=2, n=n, prec=prec, nrhs=_log_int(rng, 1, 8 if n <= 512 else 1), op=rng.choice(["A", "QA"]))
    if kind == "precond" and dim == 3:
        return dict(kind=kind, dim=3, n=rng.choice([8, 16, 32]), prec="c64", nrhs=_log_int(rng, 1, 24))
    if kind == "precond":
        return dict(kind=kind, dim=2, n=_log_int(rng, 31, 300), prec="c128", nrhs=_log_int(rng, 1, 8))
    if kind == "solve" and dim == 3:
        return dict(kind=kind, dim=3, n=rng.choice([8, 16, 32]), prec=rng.choice(["c64", "c64", "c128"]), nrhs=_log_int(rng, 1, 4))
    if kind == "solve":
        return dict(kind=kind, dim=2, n=_log_int(rng, 31, 160), prec="c128", nrhs=_log_int(rng, 1, 4))
    return dict(kind="setup", dim=2, n=_log_int(rng, 31, 119), prec="c128", nrhs=1)


# ------------------------------------------------------------------ inputs


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _gen(seed):
    g = torch.Generator(device=_device())
    g.manual_seed(int(seed) % (1 << 62))
    return g


def _taper(t, delta=0.15):
    """s(t), s'(t): 1 in the middle of (0, 1), smooth to 0 at the ends."""
    def step(u):
        inside = (u > 0) & (u < 1)
        v = torch.where(inside, u, torch.full_like(u, 0.5))
        a, b = torch.exp(-1 / v), torch.exp(-1 / (1 - v))
        s = a / (a + b)
        ds = a * b / (a + b) ** 2 * (1 / v ** 2 + 1 / (1 - v) ** 2)
        zero = torch.zeros_like(u)
        return torch.where(inside, s, (u >= 1).to(u.dtype)), torch.where(inside, ds, zero)
    s0, d0 = step(t / delta)
    s1, d1 = step((1 - t) / delta)
    return s0 * s1, (d0 * s1 - s0 * d1) / delta


def _medium(case, seed):
    """(k, eps, grad eps): seeded tapered Gaussian bumps, numpy complex128."""
    n, dim, dev = case["n"], case["dim"], _device()
    rng = np.random.default_rng([int(seed), n, dim])
    x = torch.arange(1, n + 1, dtype=torch.float64, device=dev) / (n + 1)
    s, ds = _taper(x)
    f = torch.zeros((n,) * dim, dtype=torch.float64, device=dev)
    df = [torch.zeros_like(f) for _ in range(dim)]
    line = [tuple(n if a == dim - 1 - d else 1 for a in range(dim)) for d in range(dim)]  # axis d is dimension dim - 1 - d
    for _ in range(8):
        a, w = rng.uniform(0.1, 0.4 if dim == 3 else 0.3), rng.uniform(0.05, 0.12)
        c = rng.uniform(0.2, 0.8, dim)
        e = [torch.exp(-(x - c[d]) ** 2 / (2 * w * w)) for d in range(dim)]
        for g in range(dim + 1):  # g = dim: the bump; g < dim: its derivative along g
            t = torch.full((1,) * dim, float(a), dtype=torch.float64, device=dev)
            for d in range(dim):
                v = s * e[d] if g != d else (ds - s * (x - c[d]) / (w * w)) * e[d]
                t = t * v.reshape(line[d])
            if g == dim:
                f += t
            else:
                df[g] += t
    k = math.pi * n / 4 if dim == 3 else 2 * math.pi * (n + 1) / 6
    eps = (1 + f).cpu().numpy().astype(np.complex128)
    return k, eps, torch.stack(df).cpu().numpy().astype(np.complex128)


def _dtype(case):
    return torch.complex64 if case["prec"] == "c64" else torch.complex128


def _fields(case, seed, dtype):
    """nrhs random complex normal fields."""
    n, dim = case["n"], case["dim"]
    g = _gen(seed * 1000003 + 17)
    shape = (case["nrhs"], dim) + (n,) * dim
    re = torch.randn(shape, dtype=torch.float64, device=_device(), generator=g)
    im = torch.randn(shape, dtype=torch.float64, device=_device(), generator=g)
    return torch.complex(re, im).to(dtype)


def _plane_waves(case, k, seed):
    """nrhs incident plane waves E = pol exp(i k dir.x), complex128."""
    n, dim = case["n"], case["dim"]
    rng = np.random.default_rng([int(seed), 29])
    x = torch.arange(1, n + 1, dtype=torch.float64, device=_device()) / (n + 1)
    out = torch.empty((case["nrhs"], dim) + (n,) * dim, dtype=torch.complex128, device=_device())
    for b in range(case["nrhs"]):
        u = rng.standard_normal(dim)
        u /= np.linalg.norm(u)
        v = rng.standard_normal(dim)
        v -= (v @ u) * u
        v /= np.linalg.norm(v)
        ph = sum((float(u[d]) * x).reshape(tuple(n if a == dim - 1 - d else 1 for a in range(dim))) for d in range(dim))
        w = torch.exp(1j * k * ph)
        for d in range(dim):
            out[b, d] = float(v[d]) * w
    return out


def _classes(dim):
    """Per class of points: offsets per axis (lo, hi) of its neighbourhood."""
    span = ((0, 1), (-1, 1), (-1, 0))
    return [[span[(c // 3 ** d) % 3] for d in range(dim)] for c in range(3 ** dim)]


def _offsets(cls):
    """Neighbourhood offsets (o1, o2[, o3]), the last axis outermost."""
    out = [()]
    for lo, hi in reversed(cls):
        out = [(o,) + t for t in out for o in range(lo, hi + 1)]
    return out


def _seeded_tables(case, seed):
    """Stencil tables of Q A: orthonormal columns of the class's shape."""
    dim = case["dim"]
    rng = np.random.default_rng([int(seed), 31])
    nt = 3 ** dim
    alpha = np.zeros((nt, dim * nt, dim), np.complex128)
    beta = np.zeros((nt, (dim + 1) * nt, dim), np.complex128)
    for c, cls in enumerate(_classes(dim)):
        T = len(_offsets(cls))
        a = rng.standard_normal((dim * T, dim)) + 1j * rng.standard_normal((dim * T, dim))
        alpha[c, :dim * T] = np.linalg.qr(a)[0]
        beta[c, :(dim + 1) * T] = 1e-3 * (rng.standard_normal(((dim + 1) * T, dim)) + 1j * rng.standard_normal(((dim + 1) * T, dim)))
    return alpha, beta


def _factor_prec(case):
    return spm.SPM_C64 if case["prec"] == "c64" else spm.SPM_C128


def prepare(case, seed):
    """The problem handle a program keeps for its medium, and this pass's inputs and outputs."""
    k, eps, grad = _medium(case, seed)
    P = (spm.Problem if case["dim"] == 3 else spm.Problem2D)(case["n"], k, eps, grad)
    st = dict(kind=case["kind"], P=P, op=case.get("op"))
    if case["kind"] == "apply":
        if case["op"] == "QA":
            P.set_stencils(*_seeded_tables(case, seed))
        st["x"] = _fields(case, seed, _dtype(case))
        st["y"] = torch.zeros_like(st["x"])
    elif case["kind"] == "precond":
        P.build_stencils(_factor_prec(case))
        st["x"] = _fields(case, seed, _dtype(case))
        st["t"], st["y"] = torch.zeros_like(st["x"]), torch.zeros_like(st["x"])
    elif case["kind"] == "solve":
        P.build_stencils(_factor_prec(case))
        e = _plane_waves(case, k, seed)
        st["g"], st["y"] = torch.zeros_like(e), torch.zeros_like(e)
        P.rhs_from_incident(e, st["g"])
        st["prec"] = spm.SPM_MIXED if case["prec"] == "c64" else spm.SPM_C128
    else:
        st["factor"] = _factor_prec(case)
        st["x"] = _fields(case, seed, _dtype(case))
        st["t"], st["y"] = torch.zeros_like(st["x"]), torch.zeros_like(st["x"])
    return st


def run(st):
    P, y = st["P"], st["y"]
    if st["kind"] == "apply":
        (P.apply_QA if st["op"] == "QA" else P.apply_A)(st["x"], y)
        return y
    if st["kind"] == "solve":
        y.zero_()
        P.solve(st["g"], y, prec=st["prec"], tol=1e-10, maxit=200)
        return y
    sv = None
    if st["kind"] == "setup":
        P.build_stencils(st["factor"])
        sv = P.get_stencils()[2]
    P.apply_Q(st["x"], st["t"])
    P.solve_S(st["t"], y)
    return y if sv is None else {"sv": sv, "y": y}


# ------------------------------------------------------------------ work


def _dissect(dim, lo, hi):
    """(own, boundary) unknowns of every front of a middle-cut nested dissection."""
    n = hi  # the grid is [0, n)^dim
    out, todo = [], [(lo, hi)]
    while todo:
        a, b = todo.pop()
        size = [b[d] - a[d] for d in range(dim)]
        grown = [min(b[d] + 1, n[d]) - max(a[d] - 1, 0) for d in range(dim)]
        bnd = math.prod(grown) - math.prod(size)
        ax = max(range(dim), key=lambda d: (size[d], -d))
        if size[ax] > 5:
            cut = a[ax] + size[ax] // 2
            own = math.prod(size) // size[ax]
            todo.append((a, tuple(cut if d == ax else b[d] for d in range(dim))))
            todo.append((tuple(cut + 1 if d == ax else a[d] for d in range(dim)), b))
        else:
            own = math.prod(size)
        out.append((dim * own, dim * bnd))
    return out


def _apply_work(dim, n, el, nrhs, with_q):
    N = n ** dim
    if dim == 3:
        L = 2 * n
        flops = 7 * 5 * L ** 3 * math.log2(L ** 3) * 7 / 12 + 48 * L ** 3 + (1944 * N if with_q else 0)
        spectra = 4 * (n + 1) ** 3
    else:
        L = 1 << max(3, math.ceil(math.log2(2 * n - 1)))
        flops = 5 * L * math.log2(L) * (3 * n + 5 * L + 2 * n) + 32 * L * L + (288 * N if with_q else 0)
        spectra = 3 * (L // 2 + 1) ** 2
    return el * (spectra + (1 + dim) * N + 2 * dim * N * nrhs), flops * nrhs


def _precond_work(dim, n, el, nrhs):
    fronts = _dissect(dim, (0,) * dim, (n,) * dim)
    entries = sum(o * o + 2 * o * b for o, b in fronts)
    N = n ** dim
    flops = 8 * nrhs * (entries + dim * dim * 3 ** dim * N)
    return el * (entries + 2 * dim * N * nrhs), flops


def work(case):
    dim, n, nrhs = case["dim"], case["n"], case["nrhs"]
    el = 8 if case["prec"] == "c64" else 16
    if case["kind"] == "apply":
        b, f = _apply_work(dim, n, el, nrhs, case["op"] == "QA")
    elif case["kind"] == "precond":
        b, f = _precond_work(dim, n, el, nrhs)
    elif case["kind"] == "solve":
        # about ten iterations of A, Q and S^-1 to 1e-10, three FP64 residuals
        ab, af = _apply_work(dim, n, el, nrhs, True)
        pb, pf = _precond_work(dim, n, el, nrhs)
        rb, rf = _apply_work(dim, n, 16, nrhs, False)
        b, f = 10 * (ab + pb) + 3 * rb, 10 * (af + pf) + 3 * rf
    else:
        fronts = _dissect(dim, (0,) * dim, (n,) * dim)
        f = sum(8 * (o ** 3 + 2 * o * o * v + o * v * v) for o, v in fronts)
        b = el * (sum(o * o + 2 * o * v for o, v in fronts) + dim * dim * 3 ** dim * n ** dim)
        pb, pf = _precond_work(dim, n, el, nrhs)
        b, f = b + pb, f + pf
    return {"bytes": float(b), "flops": float(f)}


# ------------------------------------------------------------------ exact values
# The same maps in 64 bits by plain torch: Toeplitz entries of the corrected
# trapezoidal rule, zero-padded library FFTs, stencils from a library eigensolver,
# S eliminated layer by layer, A x = g by GMRES without restart.


def _lattice_z3():
    s = -3.0
    for a in range(-7, 8):
        for b in range(-7, 8):
            for c in range(-7, 8):
                r2 = a * a + b * b + c * c
                if r2:
                    s += math.erfc(math.sqrt(math.pi * r2)) / math.sqrt(r2) + math.exp(-math.pi * r2) / (math.pi * r2)
    return s


def _hankel(x):
    """H_0^(1)(x), H_1^(1)(x) for x >= 1, from K_nu(z) = e^-z int_0^inf e^(-z s) T_nu(1 + s) / sqrt(s (s + 2)) ds
    (DLMF 10.32.8 with s = cosh t - 1) at z = -i x, along s = i w^2 / x: a Gaussian times a smooth even
    function of w, so the trapezoidal rule converges geometrically (torch's own Bessel functions reach 1e-7)."""
    k0, k1 = torch.zeros_like(x, dtype=torch.complex128), torch.zeros_like(x, dtype=torch.complex128)
    step = 0.14
    for j in range(46):
        s = torch.complex(torch.zeros_like(x), (j * step) ** 2 / x)
        f = (step if j else step / 2) * math.exp(-((j * step) ** 2)) * 2j / torch.sqrt(1j * (2 + s) * x)
        k0 += f
        k1 += f * (1 + s)
    e = torch.exp(1j * x)
    return -2j / math.pi * e * k0, -2 / math.pi * e * k1


def _entries(dim, n, k, t):
    """G and its gradient's entries at integer offsets t (a list of dim broadcastable tensors)."""
    h = 1.0 / (n + 1)
    r = h * torch.sqrt(sum((a * a).to(torch.float64) for a in t))
    zero = r == 0
    rs = torch.where(zero, torch.ones_like(r), r)
    if dim == 3:
        z = _lattice_z3()
        e = torch.exp(1j * k * rs) * (h ** 3 / (4 * math.pi))
        g = torch.where(zero, torch.full_like(e, complex(-h * h * z / (4 * math.pi), h ** 3 * k / (4 * math.pi))), e / rs)
        dr, shift = e * (1j * k * rs - 1) / rs ** 3, h * z / (24 * math.pi)
    else:
        zp = -0.5 * math.log(2 * math.pi) - (2 * math.lgamma(0.25) - math.log(2 * math.pi * math.sqrt(2)))
        h0, h1 = _hankel(k * rs)
        g0 = complex(-(math.log(k * h / 2) + 0.57721566490153286061 + zp) / (2 * math.pi), 0.25) * h * h
        g = h0 * (0.25j * h * h)
        g = torch.where(zero, torch.full_like(g, g0), g)
        dr, shift = h1 * (-0.25j * k * h * h) / rs, -h / (8 * math.pi)
    out = [g]
    for d in range(dim):
        v = torch.where(zero, torch.zeros_like(g), dr * (h * t[d].to(torch.float64)))
        axis = (sum(abs(a) for a in t) == 1) & (t[d] != 0)
        out.append(v + torch.where(axis, shift * t[d].to(torch.float64), torch.zeros_like(r)))
    return out


def _grid(dim, vals):
    """vals along every axis: tensors for axis 0 (the fastest dimension) to dim - 1."""
    return [vals.reshape(tuple(-1 if a == dim - 1 - d else 1 for a in range(dim))) for d in range(dim)]


class _Exact:
    def __init__(self, case, seed):
        self.dim, self.n = case["dim"], case["n"]
        self.k, eps, grad = _medium(case, seed)
        eps, grad = (torch.from_numpy(a).to(_device()) for a in (eps, grad))
        self.m, self.p = 1 - eps, -grad / eps
        self.spec = None

    def apply_A(self, x):
        dim, n = self.dim, self.n
        L = 2 * n
        dims = tuple(range(-dim, 0))
        if self.spec is None:
            v = torch.arange(L, device=_device())
            t = _grid(dim, torch.where(v < n, v, v - L))
            bad = sum((a == -n).to(torch.int8) for a in t) > 0
            self.spec = [torch.fft.fftn(torch.where(bad, torch.zeros_like(e), e)) for e in _entries(dim, n, self.k, t)]
        crop = (slice(0, n),) * dim
        y = torch.empty_like(x)
        for b in range(x.shape[0]):
            w4 = torch.fft.fftn((self.p * x[b]).sum(0), s=(L,) * dim, dim=dims)
            for d in range(dim):
                w = torch.fft.fftn(self.m * x[b, d], s=(L,) * dim, dim=dims)
                w = self.k ** 2 * self.spec[0] * w + self.spec[1 + d] * w4
                y[b, d] = x[b, d] + torch.fft.ifftn(w)[crop]
        return y

    def stencils(self):
        """alpha, beta tables and the singular values of every class."""
        dim, n, k, nt = self.dim, self.n, self.k, 3 ** self.dim
        dev = _device()
        alpha = torch.zeros((nt, dim * nt, dim), dtype=torch.complex128, device=dev)
        beta = torch.zeros((nt, (dim + 1) * nt, dim), dtype=torch.complex128, device=dev)
        sv = torch.zeros((nt, dim * nt), dtype=torch.float64, device=dev)

        def block(off, u):  # rows (d, o), columns (f, u): k^2 G on the diagonal, then G^d
            T, C = off.shape[0], u.shape[0]
            e = _entries(dim, n, k, [off[:, None, d] - u[None, :, d] for d in range(dim)])
            M = torch.zeros((dim, T, dim + 1, C), dtype=torch.complex128, device=dev)
            for d in range(dim):
                M[d, :, d] = k * k * e[0]
                M[d, :, dim] = e[1 + d]
            return M.reshape(dim * T, (dim + 1) * C)

        for c, cls in enumerate(_classes(dim)):
            off = torch.tensor(_offsets(cls), device=dev)
            box = [(0, n - 1) if lo == 0 else (-(n - 1), 0) if hi == 0 else (-(n - 2), n - 2) for lo, hi in cls]
            g = torch.meshgrid(*[torch.arange(a, b + 1, device=dev) for a, b in box], indexing="ij")
            u = torch.stack([a.reshape(-1) for a in g], 1)
            near = torch.ones(u.shape[0], dtype=torch.bool, device=dev)
            for d, (lo, hi) in enumerate(cls):
                near &= (u[:, d] >= lo) & (u[:, d] <= hi)
            u = u[~near]
            R = off.shape[0] * dim
            H = torch.zeros((R, R), dtype=torch.complex128, device=dev)
            for s in range(0, u.shape[0], 50000):
                M = block(off, u[s:s + 50000])
                H += M @ M.conj().T
            w, U = torch.linalg.eigh(H)
            a = U[:, :dim].conj()
            alpha[c, :R] = a
            beta[c, :R // dim * (dim + 1)] = block(off, off).T @ a
            sv[c, :R] = w.clamp_min(0).sqrt()
        return alpha, beta, sv

    def class_of(self):
        i = torch.arange(self.n, device=_device())
        c = torch.where(i == 0, 0, torch.where(i == self.n - 1, 2, 1))
        return sum(a * 3 ** d for d, a in enumerate(_grid(self.dim, c)))

    def spread(self, table, fields):
        """A packed table on all 3^dim offsets: [class][offset][field][c]."""
        dim, nt = self.dim, 3 ** self.dim
        out = torch.zeros((nt, nt, fields, dim), dtype=torch.complex128, device=_device())
        for c, cls in enumerate(_classes(dim)):
            offs = _offsets(cls)
            for i, o in enumerate(offs):
                out[c, sum((o[d] + 1) * 3 ** d for d in range(dim))] = table[c, torch.arange(fields, device=_device()) * len(offs) + i]
        return out

    def shifted(self, v, o):
        """v at i + o (zero outside the grid), over the last dim axes."""
        out = torch.zeros_like(v)
        dst = tuple(slice(max(0, -a), self.n - max(0, a)) for a in reversed(o))
        src = tuple(slice(max(0, a), self.n - max(0, -a)) for a in reversed(o))
        out[(Ellipsis,) + dst] = v[(Ellipsis,) + src]
        return out

    def all_offsets(self):
        return _offsets([(-1, 1)] * self.dim)

    def apply_Q(self, alpha, v):
        tab, cls = self.spread(alpha, self.dim), self.class_of()
        y = torch.zeros_like(v)
        for o in self.all_offsets():
            s = sum((o[d] + 1) * 3 ** d for d in range(self.dim))
            w = self.shifted(v, o)
            for d in range(self.dim):
                for c in range(self.dim):
                    y[:, c] += tab[:, s, d, c][cls] * w[:, d]
        return y

    def s_blocks(self, alpha, beta):
        """S as {offset: [c][f][point]}, the columns at i + offset."""
        dim, cls = self.dim, self.class_of()
        ta, tb = self.spread(alpha, dim), self.spread(beta, dim + 1)
        inside = torch.ones((self.n,) * dim, dtype=torch.complex128, device=_device())
        out = {}
        for o in self.all_offsets():
            s = sum((o[d] + 1) * 3 ** d for d in range(dim))
            m, p, one = self.shifted(self.m, o), self.shifted(self.p, o), self.shifted(inside, o)
            blk = torch.empty((dim, dim) + (self.n,) * dim, dtype=torch.complex128, device=_device())
            for c in range(dim):
                for f in range(dim):
                    blk[c, f] = ta[:, s, f, c][cls] * one + tb[:, s, f, c][cls] * m + tb[:, s, dim, c][cls] * p[f]
            out[o] = blk
        return out

    def solve_S(self, alpha, beta, b):
        """S^-1 b by block elimination over the lines (2-D) or planes (3-D) of the slowest axis."""
        n, dim, dev = self.n, self.dim, _device()
        blocks, M = self.s_blocks(alpha, beta), n ** (dim - 1)
        N, q = dim * M, b.shape[0]
        flat = torch.arange(M, device=dev).reshape((n,) * (dim - 1))
        pairs = {}  # in-layer offset -> (points with a neighbour there, those neighbours)
        for o in _offsets([(-1, 1)] * (dim - 1)):
            dst = tuple(slice(max(0, -a), n - max(0, a)) for a in reversed(o))
            src = tuple(slice(max(0, a), n - max(0, -a)) for a in reversed(o))
            pairs[o] = (flat[dst].reshape(-1), flat[src].reshape(-1))

        def dense(i, oz):  # the block of layer i's rows and layer i + oz's columns
            A = torch.zeros((dim, M, dim, M), dtype=torch.complex128, device=dev)
            for o, (r, c) in pairs.items():
                v = blocks[o + (oz,)][:, :, i].reshape(dim, dim, M)
                for a in range(dim):
                    for f in range(dim):
                        A[a, r, f, c] = v[a, f, r]
            return A.reshape(N, N)

        def below(i, X):  # layer i's rows times X on layer i - 1
            X, Y = X.reshape(dim, M, -1), torch.zeros((dim, M, X.shape[1]), dtype=torch.complex128, device=dev)
            for o, (r, c) in pairs.items():
                v = blocks[o + (-1,)][:, :, i].reshape(dim, dim, M)
                for a in range(dim):
                    Y[a, r] += sum(v[a, f, r, None] * X[f, c] for f in range(dim))
            return Y.reshape(N, -1)

        rhs = b.reshape(q, dim, n, M).permute(2, 1, 3, 0).reshape(n, N, q)
        upper, part = [], []
        for i in range(n):
            D, r = dense(i, 0), rhs[i]
            if i:
                t = below(i, torch.cat([upper[-1], part[-1]], 1))
                D, r = D - t[:, :N], r - t[:, N:]
            X = torch.linalg.solve(D, torch.cat([dense(i, 1), r], 1) if i < n - 1 else r)
            upper.append(X[:, :-q].contiguous())
            part.append(X[:, -q:].contiguous())
        for i in range(n - 2, -1, -1):
            part[i] = part[i] - upper[i] @ part[i + 1]
        return torch.stack(part).reshape(n, dim, M, q).permute(3, 1, 0, 2).reshape(b.shape).contiguous()


def _gmres_all(mul, b, tol=1e-13, most=700):
    """GMRES without restart, one right-hand side at a time; None if it does not converge."""
    out = torch.empty_like(b)
    for q in range(b.shape[0]):
        r = b[q].reshape(-1)
        norm = torch.linalg.norm(r).item()
        V = torch.empty((most + 1, r.numel()), dtype=r.dtype, device=r.device)
        V[0] = r / norm
        H = np.zeros((most + 1, most), np.complex128)
        y = None
        for j in range(most):
            w = mul(V[j].reshape(b[q].shape)).reshape(-1)
            for _ in range(2):
                h = V[:j + 1].conj() @ w
                w = w - h @ V[:j + 1]
                H[:j + 1, j] += h.cpu().numpy()
            H[j + 1, j] = torch.linalg.norm(w).item()
            V[j + 1] = w / H[j + 1, j].real
            if j % 10 == 9 or j == most - 1:
                e = np.zeros(j + 2, np.complex128)
                e[0] = norm
                y = np.linalg.lstsq(H[:j + 2, :j + 1], e, rcond=None)[0]
                if np.linalg.norm(H[:j + 2, :j + 1] @ y - e) <= tol * norm:
                    break
        else:
            return None
        out[q] = (torch.from_numpy(y).to(r.device) @ V[:len(y)]).reshape(b[q].shape)
    return out


def exact(case, seed):
    kind, dim, n = case["kind"], case["dim"], case["n"]
    E = _Exact(case, seed)
    if kind == "apply":
        x = _fields(case, seed, _dtype(case)).to(torch.complex128)
        y = E.apply_A(x)
        if case["op"] == "QA":
            y = E.apply_Q(torch.from_numpy(_seeded_tables(case, seed)[0]).to(_device()), y)
        return y
    if kind == "solve":
        e = _plane_waves(case, E.k, seed)
        return _gmres_all(lambda v: E.apply_A(v[None])[0], e - E.apply_A(e))
    x = _fields(case, seed, _dtype(case)).to(torch.complex128)
    alpha, beta, sv = E.stencils()
    y = E.solve_S(alpha, beta, E.apply_Q(alpha, x))
    return y if kind == "precond" else {"sv": sv, "y": y}
