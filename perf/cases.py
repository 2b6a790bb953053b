"""Timed cases of the library: what a program that uses it has it do.

Each case names one use through the public entry points (``runner.Problem``
with its solver, ``sgkiif.Operator``, ``sgkiif.Server``) at sizes of the
repository's own workloads, tests and benchmark:

  solve    the coefficients of the initial state are set, a few time steps
           taken and the new coefficients read back on the device;
  matvec   one application of the diffusion operator to a device vector;
  served   a group of whole solves submitted to a running server, each
           waited for and its coefficients read to the host.

``exact`` restates the method in 64 bits with torch and numpy alone: dense 1D
factors, Arnoldi with the exponential of the symmetric Hessenberg matrix, the
quadrature on the finest grid, Newton with GMRES.
"""
import functools
import itertools
import math

import numpy as np
import torch

from paper_1810_11111_gb300 import sgkiif
from paper_1810_11111_gb300.runner import Problem

SIGMA = 20.0  # penalty of the interior-penalty form (the library's default)

# ------------------------------------------------------------------ cases


def _solve(name, d, n, k, reaction, M, dt, steps, precision, **more):
    case = dict(kind="solve", d=d, n=n, k=k, reaction=reaction, M=M, dt=dt, steps=steps, precision=precision,
                form="quadrature", scheme=2, bc="periodic", tensor=False, source=False)
    case.update(more)
    if name:
        case["name"] = name
    return case


def listed():
    return [
        # the smallest solve: the paper's 2D heat runs, where the latency of
        # one step (launches, grid barriers, the small exponential) is all
        _solve("heat2d_fp64", 2, 4, 1, "heat", 20, 0.01, 10, "fp64"),
        # the benchmark: stiff cubic reaction in 3D, in the mixed mode that a
        # production run takes
        _solve("cubic3d_mixed", 3, 6, 2, "cubic", 30, 0.005, 3, "mixed"),
        # the same problem for a user who wants plain 64 bits
        _solve("cubic3d_fp64", 3, 6, 2, "cubic", 30, 0.005, 1, "fp64"),
        # two-species pattern formation in 2D on a fine grid: host-driven
        # GMRES, the M = 40 projection per species
        _solve("schnak2d_mixed", 2, 8, 2, "schnakenberg", 40, 0.05, 3, "mixed"),
        # the same system in 3D, as the served requests draw it
        _solve("schnak3d_mixed", 3, 6, 2, "schnakenberg", 30, 0.005, 1, "mixed"),
        # cubic elements in 3D, as the served requests draw them
        _solve("cubic3d_p3_mixed", 3, 6, 3, "cubic", 30, 0.005, 1, "mixed"),
        # four dimensions, as the batched instances draw them
        _solve("cubic4d_mixed", 4, 5, 1, "cubic", 30, 0.005, 2, "mixed"),
        # the paper's Example 3: zero Dirichlet data, quadratic reaction,
        # time-dependent source, the third-order scheme with its history
        _solve("dirichlet2d_iif3_mixed", 2, 7, 2, "quadratic", 25, 1.0 / 64, 4, "mixed", scheme=3,
               bc="dirichlet", source=True),
        # a full diffusion tensor (mixed derivatives)
        _solve("tensor3d_mixed", 3, 5, 2, "cubic", 30, 0.005, 2, "mixed", tensor=True),
        # a large 4D problem with the sparse-grid interpolation form of the
        # reaction, which needs no full grid
        _solve("interp4d_mixed", 4, 8, 2, "cubic", 30, 0.005, 1, "mixed", form="interp"),
        # the operator by itself at the largest served shape (6.8 M coefficients)
        dict(name="matvec4d_fp64", kind="matvec", d=4, n=9, k=3, precision="fp64", bc="periodic"),
        # whole solves through the server, arriving together: scalar requests
        # stepped in one batch, systems by the workers, set-up included
        dict(name="served", kind="served", requests="3:6:1:cubic 3:6:2:cubic 3:6:1:schnakenberg 3:7:1:cubic",
             M=30, dt=0.005, steps=10, precision="mixed"),
    ]


def _nodal(d, n, k):
    return ((k + 1) << n) ** d


def draw(rng):
    """A case of the ranges above: sizes over their logarithm (levels), every
    option drawn; the finest grid stays within that of the listed cases."""
    kind = rng.choice(["solve"] * 7 + ["matvec"] * 2 + ["served"])
    if kind == "matvec":
        while True:
            d, n, k = rng.randint(2, 4), rng.randint(3, 9), rng.randint(1, 3)
            if 500 <= _dof(d, n, k) <= 6815744:
                return dict(kind="matvec", d=d, n=n, k=k, precision=rng.choice(["fp64", "mixed"]),
                            bc=rng.choice(["periodic", "dirichlet"]))
    if kind == "served":
        shapes = []
        while len(shapes) < 3:
            d, n, k = rng.randint(3, 4), rng.randint(4, 6), rng.randint(1, 3)
            if _nodal(d, n, k) <= 8 << 20:
                shapes.append("%d:%d:%d:%s" % (d, n, k, rng.choice(["cubic", "schnakenberg"])))
        return dict(kind="served", requests=" ".join(shapes), M=30, dt=0.005, steps=rng.randint(3, 8),
                    precision="mixed")
    while True:
        d, n, k = rng.randint(2, 4), rng.randint(3, 8), rng.randint(1, 3)
        reaction = rng.choice(["heat", "cubic", "cubic", "cubic", "schnakenberg", "quadratic"])
        precision = rng.choice(["mixed", "mixed", "fp64"])
        form = rng.choice(["quadrature", "quadrature", "quadrature", "interp"])
        tensor = reaction != "schnakenberg" and form == "quadrature" and rng.random() < 0.15
        if reaction in ("heat", "quadratic"):
            form = "quadrature"
        cap = (4 << 20) if precision == "fp64" or reaction == "schnakenberg" or tensor else (17 << 20)
        if form == "interp":
            if not 200 <= _dof(d, n, k) <= 200000:
                continue
        elif not 2000 <= _nodal(d, n, k) <= cap or (tensor and _dof(d, n, k) > 6000):
            continue
        quadratic = reaction == "quadratic"
        return _solve(None, d, n, k, reaction, rng.choice([20, 25, 30, 40]), rng.choice([0.005, 0.0025]),
                      rng.randint(1, 3), precision, form=form, scheme=rng.choice([2, 2, 3]) if quadratic else 2,
                      bc="dirichlet" if quadratic else "periodic", source=quadratic, tensor=tensor)


# --------------------------------------------------------- a user's program


def _kappas(d, reaction):
    if reaction == "schnakenberg":
        return [[0.01] * d, [0.5] * d]
    if reaction == "quadratic":
        return [[1.0 / (4 * math.pi ** 2 * d)] * d]
    if reaction == "heat":
        return [[1.0] * d]
    return [[1.0, 0.5, 0.1, 0.7][:d]]


def _tensor(d):
    """A rotated anisotropic tensor: the diagonal of the scalar runs with
    off-diagonal entries (diagonally dominant, so positive definite)."""
    K = np.diag([1.0, 0.5, 0.4, 0.7][:d])
    for i in range(d - 1):
        K[i, i + 1] = K[i + 1, i] = 0.1 * (1 + i)
    return K


def _terms(reaction):
    return {"heat": [[]],
            "cubic": [[(-100.0, (3,))]],
            "quadratic": [[(1.0, (2,))]],
            "schnakenberg": [[(0.1, (0, 0)), (-1.0, (1, 0)), (1.0, (2, 1))],
                             [(0.9, (0, 0)), (-1.0, (2, 1))]]}[reaction]


def _init(rng, d, reaction):
    """Initial data: seeded Fourier modes, or for the two-species system its
    seeded noise on every coefficient."""
    if reaction == "schnakenberg":
        seed = int(rng.integers(0, 2 ** 31))
        return [dict(noise_seed=seed, base=1.0, species=0), dict(noise_seed=seed, base=0.9, species=1)]
    if reaction == "quadratic":  # vanishes on the boundary
        modes = 4
        return [dict(amp=np.concatenate([[1.0], 0.1 * rng.uniform(-1.0, 1.0, modes - 1)]),
                     wavenum=np.concatenate([np.ones((1, d)), rng.integers(1, 4, (modes - 1, d))]).astype(np.int32),
                     kind=np.zeros((modes, d), np.int32), const=0.0)]
    modes = 8
    return [dict(amp=rng.uniform(-1.0, 1.0, modes), wavenum=rng.integers(1, 4, (modes, d)).astype(np.int32),
                 kind=rng.integers(0, 2, (modes, d)).astype(np.int32), const=0.0)]


def _sources(d):
    """u_t = Lap u / (4 pi^2 d) + u^2 - e^{-2t} prod sin^2(2 pi x_i), whose
    solution is e^{-t} prod sin(2 pi x_i) for the unperturbed initial data."""
    amp, wave, kind = [], [], []
    for on in itertools.product((0, 1), repeat=d):  # prod (1/2 - 1/2 cos(4 pi x_i))
        amp.append(-(0.5 ** d) * (-1.0) ** sum(on))
        wave.append([2 * o for o in on])
        kind.append([1] * d)
    return [[dict(lam=-2.0, amp=np.array(amp), wavenum=np.array(wave, np.int32), kind=np.array(kind, np.int32),
                  const=0.0)]]


def _config(case, seed):
    d = case["d"]
    rng = np.random.default_rng(seed)
    cfg = dict(d=d, n=case["n"], k=case["k"], kappas=_kappas(d, case["reaction"]), reaction=_terms(case["reaction"]),
               M=case["M"], dt=case["dt"], steps=case["steps"], init=_init(rng, d, case["reaction"]),
               scheme=case.get("scheme", 2), reaction_form=case.get("form", "quadrature"))
    if case.get("tensor"):
        cfg["kappas"] = [_tensor(d)]
    if case.get("source"):
        cfg["sources"] = _sources(d)
    return cfg


def _requests(case, seed):
    out = []
    for i, shape in enumerate(case["requests"].split()):
        d, n, k, reaction = shape.split(":")
        out.append(dict(case, kind="solve", d=int(d), n=int(n), k=int(k), reaction=reaction))
    return [_config(c, seed * 1000 + i) for i, c in enumerate(out)], out


def _precision(case):
    return sgkiif.SGK_FP64 if case["precision"] == "fp64" else sgkiif.SGK_MIXED


def _bc(case):
    return sgkiif.SGK_DIRICHLET0 if case.get("bc") == "dirichlet" else sgkiif.SGK_PERIODIC


class _State:
    """What the program holds; its library handles are closed with it."""

    def __init__(self, case, **held):
        self.case = case
        self.__dict__.update(held)

    def __del__(self):
        for name in ("problem", "server", "op", "index", "ctx"):
            handle = self.__dict__.pop(name, None)
            if handle is not None:
                handle.close()


def prepare(case, seed):
    if case["kind"] == "solve":
        return _State(case, problem=Problem(_config(case, seed), _precision(case), bc=_bc(case)))
    if case["kind"] == "served":
        configs, _ = _requests(case, seed)
        return _State(case, configs=configs, server=sgkiif.Server(workers=4, mem_budget_bytes=32 << 30))
    ctx = sgkiif.Context(0, torch.cuda.current_stream().cuda_stream, _precision(case))
    index = sgkiif.IndexSet(ctx, case["d"], case["n"], case["k"])
    op = sgkiif.Operator(ctx, index, _kappas(case["d"], "cubic")[0], _bc(case))
    return _State(case, ctx=ctx, index=index, op=op, x=_matvec_input(case, seed))


def _matvec_input(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.randn(_dof(case["d"], case["n"], case["k"]), dtype=torch.float64, device="cuda", generator=g)
    return x if case["precision"] == "fp64" else x.float()


def run(state):
    case = state.case
    if case["kind"] == "solve":
        p = state.problem
        p.reset()
        p.solver.step(case["steps"])
        out = []
        for s in range(p.nspecies):
            u = torch.empty(p.dof, dtype=torch.float64, device=p.device)
            p.solver.get_state(s, dev_ptr=u.data_ptr())
            out.append(u)
        return out
    if case["kind"] == "served":
        tickets = [state.server.submit(cfg, _precision(case)) for cfg in state.configs]
        return [state.server.wait(t, cap=len(cfg["kappas"]) * sgkiif.dof_of(cfg["d"], cfg["n"], cfg["k"]))[0]
                for t, cfg in zip(tickets, state.configs)]
    y = torch.empty_like(state.x)
    state.op.matvec(state.x.data_ptr(), y.data_ptr(), _precision(case))
    return y


# -------------------------------------------------------------------- work


def _tuples(d, n):
    return [l for l in itertools.product(range(n + 1), repeat=d) if sum(l) <= n]


def _size(l, k):
    return (k + 1) << (l - 1) if l else k + 1


def _dof(d, n, k):
    count = [1] + [0] * n  # coefficients by |l|_1, one direction after the other
    for _ in range(d):
        count = [sum(count[m - l] * _size(l, k) for l in range(m + 1)) for m in range(n + 1)]
    return sum(count)


@functools.lru_cache(None)
def _row_entries(n, k, periodic):
    """Entries of the 1D operator from level l to levels up to m, [l][m]."""
    S = np.abs(_operator_1d(n, k, periodic))
    S = S > 1e-12 * np.sqrt(np.outer(S.diagonal(), S.diagonal())) + 1e-14 * S.max()
    at = [0] + [(k + 1) << m for m in range(n + 1)]
    by = [[int(S[at[l]:at[l + 1], at[m]:at[m + 1]].sum()) for m in range(n + 1)] for l in range(n + 1)]
    return [list(itertools.accumulate(row)) for row in by]


@functools.lru_cache(None)
def _madds(d, n, k, periodic):
    rows, total = _row_entries(n, k, periodic), 0
    for l in _tuples(d, n):
        size = math.prod(_size(m, k) for m in l)
        total += sum(size // _size(m, k) * rows[m][n - sum(l) + m] for m in l)
    return total


def _pass_madds(d, n, k, q):
    """Multiply-adds of one finest-grid pass: the two-scale transforms there
    and back, Gauss points and moments cell by cell."""
    H, kp1 = (k + 1) << n, k + 1
    pyramid = sum(2 * H ** (i + 1) * max(1, _dof(d - 1 - i, n, k) if i < d - 1 else 1) * 4 * kp1 for i in range(d))
    points = 2 * sum(q ** (i + 1) * kp1 ** (d - i) for i in range(d))
    return min(pyramid, 8 * kp1 * d * H ** d) + (1 << n) ** d * points


def _degree(reaction):
    return {"heat": 0, "quadratic": 2, "cubic": 3, "schnakenberg": 3}[reaction]


def _points(case):
    p, k = _degree(case["reaction"]), case["k"]
    return -(-(p * k + k + 1) // 2)


def work(case):
    if case["kind"] == "served":
        parts = [work(c) for c in _requests(case, 0)[1]]
        return {"bytes": sum(p["bytes"] for p in parts), "flops": sum(p["flops"] for p in parts)}
    d, n, k = case["d"], case["n"], case["k"]
    dof, madds = _dof(d, n, k), _madds(d, n, k, case["bc"] == "periodic" if "bc" in case else True)
    if case["kind"] == "matvec":
        return {"bytes": 2 * dof * (8 if case["precision"] == "fp64" else 4), "flops": 2 * madds}
    S, M = (2 if case["reaction"] == "schnakenberg" else 1), case["M"]
    projections = case.get("scheme", 2) - 1
    if case.get("tensor"):  # four pairs of rows per off-diagonal entry, both directions
        madds += 4 * (d - 1) * dof * (2 * k + 2) ** 2
    step = S * projections * (2 * M * madds + 4 * M * M * dof)
    if case["reaction"] != "heat":
        if case.get("form", "quadrature") == "interp":
            step += S * 3 * 2 * 2 * d * (k + 2) * dof
        else:  # one residual and one Jacobian product at least
            step += 2 * 2 * S * _pass_madds(d, n, k, _points(case))
    return {"bytes": 2 * S * dof * 8, "flops": case["steps"] * step}


# ------------------------------------------------------- 64 bits, from scratch


def _legendre(r, x):
    p0, p1 = np.ones_like(x), x
    if r == 0:
        return p0
    for m in range(1, r):
        p0, p1 = p1, ((2 * m + 1) * x * p1 - m * p0) / (m + 1)
    return p1


@functools.lru_cache(None)
def _two_scale(k):
    """(H, G), each 2 (k+1) x (k+1): the orthonormal Legendre polynomials of a
    cell, and Alpert's wavelets (most vanishing moments last; the first right
    half coefficient from degree k down is positive), over its two halves."""
    x, w = np.polynomial.legendre.leggauss(2 * k + 4)
    half = [math.sqrt(2 * s + 1) * _legendre(s, x) for s in range(k + 1)]

    def over_halves(i):  # polynomial i of the whole cell against the halves' bases
        g = [math.sqrt(2 * i + 1) * _legendre(i, (x + c) / 2) for c in (-1.0, 1.0)]
        return np.concatenate([[np.sum(w * gh * hs) / 2 / math.sqrt(2) for hs in half] for gh in g])

    H = np.stack([over_halves(r) for r in range(k + 1)], axis=1)
    wavelets = {}
    for p in range(k, -1, -1):
        rows = [over_halves(i) for i in range(p + k + 1)] + list(wavelets.values())
        v = np.linalg.svd(np.stack(rows))[2][-1]
        lead = next(v[k + 1 + s] for s in range(k, -1, -1) if abs(v[k + 1 + s]) > 1e-8)
        wavelets[p] = v * math.copysign(1.0, lead)
    return H, np.stack([wavelets[p] for p in range(k + 1)], axis=1)


@functools.lru_cache(None)
def _to_finest(n, k):
    """Hierarchical coefficients -> finest-cell Legendre coefficients."""
    H, G = _two_scale(k)
    T = np.eye(k + 1)
    for m in range(n):
        T = np.concatenate([np.kron(np.eye(1 << m), H) @ T, np.kron(np.eye(1 << m), G)], axis=1)
    return T


@functools.lru_cache(None)
def _forms_1d(n, k, periodic):
    """Hierarchical matrices: interior-penalty form S, and for the mixed
    derivatives P (test derivative against value) and E (jump against mean)."""
    kp1, cells, h = k + 1, 1 << n, 0.5 ** n
    x, w = np.polynomial.legendre.leggauss(k + 2)
    s = np.sqrt(2 * np.arange(kp1) + 1)
    val = np.stack([s[r] * _legendre(r, x) for r in range(kp1)])
    der = np.stack([s[r] * np.polynomial.Legendre.basis(r).deriv()(x) for r in range(kp1)]) * 2 / h
    right, left = s / math.sqrt(h), s * (-1.0) ** np.arange(kp1) / math.sqrt(h)
    r = np.arange(kp1)
    dright = s * r * (r + 1) / 2 * 2 / h / math.sqrt(h)
    dleft = dright * (-1.0) ** (r + 1)
    S = np.kron(np.eye(cells), (der * w / 2) @ der.T)
    P = np.kron(np.eye(cells), (der * w / 2) @ val.T)
    E = np.zeros_like(S)
    for f in range(cells if periodic else cells + 1):
        jump, mean, dmean = (np.zeros(cells * kp1) for _ in range(3))
        inner = periodic or 0 < f < cells
        part = 0.5 if inner else 1.0
        if periodic or f > 0:
            L = slice((f - 1) % cells * kp1, ((f - 1) % cells + 1) * kp1)
            jump[L] += right
            mean[L] += part * right
            dmean[L] += part * dright
        if periodic or f < cells:
            R = slice(f % cells * kp1, (f % cells + 1) * kp1)
            jump[R] -= left
            mean[R] += part * left
            dmean[R] += part * dleft
        at = np.flatnonzero((jump != 0) | (mean != 0) | (dmean != 0))
        ix = np.ix_(at, at)
        j, m, dm = jump[at], mean[at], dmean[at]
        S[ix] += SIGMA / h * np.outer(j, j) - np.outer(j, dm) - np.outer(dm, j)
        E[ix] += np.outer(j, m)
    T = _to_finest(n, k)
    return T.T @ S @ T, T.T @ P @ T, T.T @ E @ T


def _operator_1d(n, k, periodic):
    return _forms_1d(n, k, periodic)[0]


def _along(F, x, m):
    """The matrix F applied along axis m of x."""
    return torch.movedim(torch.tensordot(F, x, dims=([1], [m])), 0, m)


class _Grid:
    """A sparse grid in 64 bits: coefficients by level tuple (lexicographic),
    row-major within it, embedded in the full hierarchical array."""

    def __init__(self, d, n, k, periodic, full=True):
        self.d, self.n, self.k, self.H = d, n, k, (k + 1) << n
        self.tuples = _tuples(d, n)
        self.sizes = {l: tuple(_size(m, k) for m in l) for l in self.tuples}
        self.first, at = {}, 0
        for l in self.tuples:
            self.first[l] = at
            at += math.prod(self.sizes[l])
        self.dof = at
        self.dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
        self.S, self.P, self.E = (torch.from_numpy(f).to(self.dev) for f in _forms_1d(n, k, periodic))
        self.T = torch.from_numpy(_to_finest(n, k)).to(self.dev)
        self.levels = [slice(_size(l, k) if l else 0, 2 * _size(l, k) if l else k + 1) for l in range(n + 1)]
        if full:
            place = torch.arange(self.H ** d, device=self.dev).reshape((self.H,) * d)
            self.place = torch.cat([place[tuple(self.levels[m] for m in l)].reshape(-1) for l in self.tuples])

    def block(self, x, l):
        return x[self.first[l]:self.first[l] + math.prod(self.sizes[l])].reshape(self.sizes[l])

    def embed(self, x):
        out = torch.zeros(self.H ** self.d, dtype=torch.float64, device=self.dev)
        out[self.place] = x
        return out.reshape((self.H,) * self.d)

    def diffuse(self, x, kappa):
        y = torch.zeros_like(x)
        for l in self.tuples:
            out = self.block(y, l)
            for i in range(self.d):
                for m in range(self.n - sum(l) + l[i] + 1):
                    other = l[:i] + (m,) + l[i + 1:]
                    out -= kappa[i] * _along(self.S[self.levels[l[i]], self.levels[m]], self.block(x, other), i)
        return y

    def diffuse_full(self, x, K):
        X = self.embed(x)
        Y = torch.zeros_like(X)
        for i in range(self.d):
            Y -= float(K[i][i]) * _along(self.S, X, i)
            for j in range(i + 1, self.d):
                if K[i][j] == 0:
                    continue
                P, E = self.P, self.E
                for a, b, c in ((P, P.T, 1.0), (P.T, P, 1.0), (E, P.T, -1.0), (P.T, E, -1.0), (E.T, P, -1.0),
                                (P, E.T, -1.0)):
                    Y -= float(K[i][j]) * c * _along(b, _along(a, X, i), j)
        return Y.reshape(-1)[self.place]

    def project(self, g):
        """L2 projection of separable Fourier terms (12 points a cell)."""
        x, w = np.polynomial.legendre.leggauss(12)
        cells, h, kp1 = 1 << self.n, 0.5 ** self.n, self.k + 1
        at = (np.arange(cells)[:, None] + (x + 1) / 2) * h
        basis = np.stack([math.sqrt((2 * r + 1) / h) * _legendre(r, x) for r in range(kp1)])
        T = _to_finest(self.n, self.k)

        def one(wave, kind):
            v = (np.sin if kind == 0 else np.cos)(2 * math.pi * wave * at)
            return torch.from_numpy(T.T @ ((v * w * h / 2) @ basis.T).reshape(-1)).to(self.dev)

        out = torch.zeros(self.dof, dtype=torch.float64, device=self.dev)
        out[0] += g.get("const", 0.0)
        for amp, waves, kinds in zip(g["amp"], g["wavenum"], g["kind"]):
            f = [one(int(wv), int(kd)) for wv, kd in zip(waves, kinds)]
            for l in self.tuples:
                term = f[0][self.levels[l[0]]]
                for m in range(1, self.d):
                    term = term[..., None] * f[m][self.levels[l[m]]]
                self.block(out, l).add_(term, alpha=float(amp))
        return out


class _Method:
    """The time stepping of one problem in 64 bits."""

    def __init__(self, case, cfg):
        self.case, self.cfg = case, cfg
        self.g = _Grid(cfg["d"], cfg["n"], cfg["k"], case.get("bc", "periodic") == "periodic")
        self.S = len(cfg["kappas"])
        self.terms = cfg["reaction"]
        self.sources = [[(t["lam"], self.g.project(t)) for t in terms] for terms in cfg.get("sources", [[]] * self.S)]
        self.heat = case["reaction"] == "heat"
        if case.get("form") == "interp":
            self._interpolation()
        elif not self.heat:
            self._quadrature()

    def _quadrature(self):
        g, q = self.g, _points(self.case)
        x, w = np.polynomial.legendre.leggauss(q)
        h = 0.5 ** g.n
        B = np.stack([math.sqrt((2 * r + 1) / h) * _legendre(r, x) for r in range(g.k + 1)], axis=1)
        V = np.kron(np.eye(1 << g.n), B) @ _to_finest(g.n, g.k)
        self.V = torch.from_numpy(V).to(g.dev)
        self.VW = torch.from_numpy((V * np.tile(w * h / 2, 1 << g.n)[:, None]).T.copy()).to(g.dev)

    def _interpolation(self):
        """Values at nested points: the fixed sets of reading x -> 2x mod 1,
        each level adding those points of its cells that are new."""
        g, k = self.g, self.g.k
        base = {1: [(1, 3), (2, 3)], 2: [(0, 1), (1, 3), (2, 3)], 3: [(1, 5), (2, 5), (3, 5), (4, 5)]}[k]
        values = [a / b for a, b in base]
        new = [(c + v) / 2 for c in (0, 1) for v in values]
        new = sorted(v for v in new if min(abs(v - u) for u in values) > 1e-12)
        points = list(values)
        for n in range(1, g.n + 1):
            cells = 1 << (n - 1)
            points += [(j + v) / cells for j in range(cells) for v in new]
        points = np.array(points) + 1e-13  # a point on a breakline belongs to the cell that it begins
        h = 0.5 ** g.n
        cell = np.floor(points / h).astype(int)
        xi = 2 * (points / h - cell) - 1
        B = np.stack([math.sqrt((2 * r + 1) / h) * _legendre(r, np.where(np.abs(xi + 1) < 1e-9, -1.0, xi))
                      for r in range(k + 1)], axis=1)
        T = _to_finest(g.n, k).reshape(1 << g.n, k + 1, g.H)
        V = torch.from_numpy(np.einsum("pr,pra->pa", B, T[cell])).to(g.dev)
        where = g.place
        ax = [(where // g.H ** (g.d - 1 - m)) % g.H for m in range(g.d)]
        C = V[ax[0][:, None], ax[0][None, :]]
        for m in range(1, g.d):
            C = C * V[ax[m][:, None], ax[m][None, :]]
        self.C, self.lu = C, torch.linalg.lu_factor(C)

    def f(self, u, s):
        out = torch.zeros_like(u[0])
        for c, e in self.terms[s]:
            out += c * functools.reduce(lambda a, b: a * b, [v ** p for v, p in zip(u, e)])
        return out

    def df(self, u, s, r):
        out = torch.zeros_like(u[0])
        for c, e in self.terms[s]:
            if e[r]:
                low = [p - (i == r) for i, p in enumerate(e)]
                out += c * e[r] * functools.reduce(lambda a, b: a * b, [v ** p for v, p in zip(u, low)])
        return out

    def values(self, x):
        if self.case.get("form") == "interp":
            return self.C @ x
        x = self.g.embed(x)
        for m in range(self.g.d):
            x = _along(self.V, x, m)
        return x

    def back(self, v):
        if self.case.get("form") == "interp":
            return torch.linalg.lu_solve(*self.lu, v[:, None])[:, 0]
        for m in range(self.g.d):
            v = _along(self.VW, v, m)
        return v.reshape(-1)[self.g.place]

    def F(self, U, t):
        u = [self.values(x) for x in U]
        out = [self.back(self.f(u, s)) for s in range(self.S)]
        return [o + sum((math.exp(lam * t) * S for lam, S in self.sources[s]), torch.zeros_like(o))
                for s, o in enumerate(out)], u

    def A(self, x, s):
        kap = self.cfg["kappas"][s]
        return self.g.diffuse_full(x, kap) if np.ndim(kap) == 2 else self.g.diffuse(x, kap)

    def expv(self, v, tau, s):
        M, gamma = self.cfg["M"], float(v.norm())
        if gamma == 0:
            return v
        V, H, m = [v / gamma], torch.zeros(M + 1, M, dtype=torch.float64), M
        for j in range(M):
            w = self.A(V[j], s)
            basis = torch.stack(V)
            for _ in range(2):
                h = basis @ w
                w = w - basis.T @ h
                H[:j + 1, j] += h.cpu()
            H[j + 1, j] = w.norm().cpu()
            if H[j + 1, j] <= 1e-12 * H[:j + 2, :j + 1].norm():
                m = j + 1
                break
            V.append(w / H[j + 1, j].item())
        sym = (H[:m, :m] + H[:m, :m].T) / 2
        lam, Q = torch.linalg.eigh(sym)
        y = Q @ (torch.exp(tau * lam) * Q[0])
        return gamma * (torch.stack(V[:m]).T @ y.to(v.device))

    def stage(self, W, c, t):
        """U - c F(U) = W."""
        if self.heat:
            return W
        U, scale, best = list(W), float(torch.cat(W).norm()), math.inf
        for _ in range(40):
            F, u = self.F(U, t)
            G = torch.cat([U[s] - c * F[s] - W[s] for s in range(self.S)])
            off = float(G.norm())
            if off <= 2e-15 * scale or (off <= 1e-12 * scale and off > 0.3 * best):
                break
            best = off
            d = [[self.df(u, s, r) for r in range(self.S)] for s in range(self.S)]

            def J(x):
                parts = x.split(self.g.dof)
                w = [self.values(p) for p in parts]
                return x - c * torch.cat([self.back(sum(d[s][r] * w[r] for r in range(self.S)))
                                          for s in range(self.S)])

            step = _gmres(J, -G)
            U = [a + b for a, b in zip(U, step.split(self.g.dof))]
        return U

    def run(self, U, steps):
        dt, t, past = self.cfg["dt"], 0.0, None
        for _ in range(steps):
            F = None if self.heat else self.F(U, t)[0]
            three = self.cfg["scheme"] == 3 and past is not None
            a = (5 / 12, 8 / 12, -1 / 12) if three else (0.5, 0.5)
            W = []
            for s in range(self.S):
                w = self.expv(U[s] if self.heat else U[s] + a[1] * dt * F[s], dt, s)
                if three:
                    w = w + a[2] * dt * self.expv(past[s], 2 * dt, s)
                W.append(w)
            U, past, t = self.stage(W, a[0] * dt, t + dt), F, t + dt
        return U


def _gmres(A, b, tol=1e-6, most=40):
    beta = float(b.norm())
    V, H = [b / beta], torch.zeros(most + 1, most, dtype=torch.float64)
    for j in range(most):
        w = A(V[j])
        basis = torch.stack(V)
        for _ in range(2):
            h = basis @ w
            w = w - basis.T @ h
            H[:j + 1, j] += h.cpu()
        H[j + 1, j] = w.norm().cpu()
        rhs = torch.zeros(j + 2, 1, dtype=torch.float64)
        rhs[0] = beta
        y = torch.linalg.lstsq(H[:j + 2, :j + 1], rhs).solution
        if float((H[:j + 2, :j + 1] @ y - rhs).norm()) <= tol * beta or H[j + 1, j] <= 1e-14 * beta:
            break
        V.append(w / H[j + 1, j].item())
    return torch.stack(V[:j + 1]).T @ y[:, 0].to(b.device)


def _solved(case, seed, cfg):
    method = _Method(case, cfg)
    if case["reaction"] == "schnakenberg":  # seeded noise on every coefficient, one stream for both species
        noise, U = np.random.default_rng(cfg["init"][0]["noise_seed"]), []
        for init in cfg["init"]:
            u = 0.01 * noise.standard_normal(method.g.dof)
            u[0] += init["base"]
            U.append(torch.from_numpy(u).to(method.g.dev))
    else:
        U = [method.g.project(init) for init in cfg["init"]]
    return method.run(U, cfg["steps"])


def exact(case, seed):
    """What run() returns, in 64 bits; None where the dense factors, the full
    grid or the number of steps would take too long."""
    if case["kind"] == "matvec":
        grid = _Grid(case["d"], case["n"], case["k"], case["bc"] == "periodic", full=False)
        x = _matvec_input(case, seed).double().to(grid.dev)
        return grid.diffuse(x, _kappas(case["d"], "cubic")[0])
    if case["kind"] == "served":
        out = []
        for cfg, c in zip(*_requests(case, seed)):
            small = _nodal(c["d"], c["n"], c["k"]) * (4 if c["reaction"] == "schnakenberg" else 1) <= 9 << 20
            out.append(torch.cat(_solved(c, seed, cfg)).cpu().numpy() if small else None)
        return out
    if case["form"] == "interp":
        if _dof(case["d"], case["n"], case["k"]) > 20000 or _nodal(case["d"], case["n"], case["k"]) > 1 << 28:
            return None
    return _solved(case, seed, _config(case, seed))
