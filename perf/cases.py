"""The calls a user of the library makes, as cases to be timed: single steps of
the method through the kernel-level entry points, and whole solves through the
drivers.

Every matrix is separable (a Kronecker sum of 1D operators, or a trilinear
finite-element stiffness matrix with lumped mass built from them), with random
1D coefficients made from the seed.  Its eigenpairs are products of 1D ones,
so the start blocks, the search intervals and the 64-bit reference values come
from small dense eigenproblems, while the sparse matrices handed to the library
have the patterns, sizes and kinds of values of its workloads (5-, 7- and
27-point stencils with random coefficients).
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2002_04807_gb300 as feast
from paper_2002_04807_gb300 import _lib
from paper_2002_04807_gb300.autograd import feast_eigenvalues

F64 = torch.float64
MASS = 1.0 / 6.0  # M = D - MASS * K: the consistent mass matrix of linear elements on a uniform grid


# --------------------------------------------------------------------------
# the cases
# --------------------------------------------------------------------------
def _filter(a, b, c, m, points=7, ne=8, ratio=200, mixed=True, tol=2, maxit=80, batch=1, noise=1e-7):
    return {"kind": "filter", "a": a, "b": b, "c": c, "m": m, "points": points, "ne": ne, "ratio": ratio,
            "mixed": mixed, "tol": tol, "maxit": maxit, "batch": batch, "noise": noise}


def listed():
    return [
        # a residual-inverse contour pass of the headline workload (64^3, 150 columns,
        # 8 nodes, one node per batch): where a solve spends nine tenths of its time
        {"name": "filter_7pt_64", **_filter(64, 64, 64, 150)},
        # the same step for a generalized problem with 27 points per row and a diagonal
        # B, many columns and nodes, half the side of the 96^3 workload
        {"name": "filter_27pt_48", **_filter(48, 48, 48, 300, points=27, ne=16, ratio=100)},
        # FP64 shifted solves (fpm(42) = 0), for callers that do not want mixed precision
        {"name": "filter_f64_32", **_filter(32, 32, 32, 64, mixed=False)},
        # a small ragged 2D problem with the library's default inner solver and node
        # batch (fpm(45) = 1, fpm(46) = 40, fpm(50) = 0): launches and latency count
        {"name": "filter_2d_ragged", **_filter(97, 61, 1, 37, points=5, tol=1, maxit=40, batch=0, noise=1e-8)},
        # the projections A_Q = Q^T A Q and B_Q = Q^T Q of one Rayleigh-Ritz step
        {"name": "project_64", "kind": "project", "a": 64, "b": 64, "c": 64, "m": 150},
        # the Ritz vectors X = Q V and their residuals, of the same step
        {"name": "ritz_64", "kind": "ritz", "a": 64, "b": 64, "c": 64, "m": 150, "points": 7},
        # the reduced dense eigenproblem of that step, in a later loop (B_Q near I)
        {"name": "reduced_150", "kind": "reduced", "m": 150},
        # the backward step alone: the gradient over A's stored entries at the size of
        # the differentiation workload
        {"name": "grad_48", "kind": "grad", "a": 48, "b": 48, "c": 48, "m": 71, "points": 7},
        # forward and backward of the differentiable solver on the headline problem:
        # the lowest eigenvalues, and the gradient of their sum over the stored entries
        {"name": "eigenvalues_64", "kind": "autograd", "a": 64, "b": 64, "c": 64, "m": 150, "mixed": True},
        # a small host call (the 1D example, n = 1000, the guide's default stopping rule)
        {"name": "solve_1d", "kind": "host", "n": 1000, "m": 48},
        # a complex Hermitian solve (random gauge phases on every link), device buffers
        {"name": "hermitian_24", "kind": "hermitian", "a": 24, "b": 24, "c": 24, "m": 60},
        # a batch of uneven 2D problems from host buffers in one call
        {"name": "batched_2d", "kind": "batched", "count": 24, "lo": 32, "hi": 96},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["filter", "filter", "filter", "project", "ritz", "reduced", "grad", "autograd", "host",
                       "hermitian", "batched"])
    if kind == "filter":
        points = rng.choice([5, 7, 7, 27])
        if points == 5:
            a, b, c = rng.randint(24, 256), rng.randint(24, 256), 1
        else:
            a, b, c = (rng.randint(11, 56 if points == 7 else 40) for _ in range(3))
        mixed = rng.random() < 0.75
        m = _log_int(rng, 8, min(160, a * b * c // 16) if mixed else 48)
        tol = rng.choice([1, 2])
        return _filter(a, b, c, m, points, rng.choice([4, 8, 16]), rng.choice([100, 200]), mixed, tol,
                       40 if tol == 1 else 80, rng.choice([0, 1, 1]), 1e-8 if tol == 1 else 1e-7)
    if kind in ("project", "ritz", "grad"):
        a, b, c = (rng.randint(9, 64) for _ in range(3))
        case = {"kind": kind, "a": a, "b": b, "c": c, "m": min(_log_int(rng, 8, 200), a * b * c // 4)}
        if kind != "project":
            case["points"] = rng.choice([7, 27])
        return case
    if kind == "reduced":
        return {"kind": "reduced", "m": _log_int(rng, 8, 300)}
    if kind == "autograd":
        a, b, c = (rng.randint(10, 40) for _ in range(3))
        return {"kind": "autograd", "a": a, "b": b, "c": c, "m": rng.randint(18, 90),
                "mixed": rng.random() < 0.75}
    if kind == "host":
        return {"kind": "host", "n": _log_int(rng, 200, 1600), "m": rng.randint(12, 60)}
    if kind == "hermitian":
        a, b, c = (rng.randint(8, 24) for _ in range(3))
        return {"kind": "hermitian", "a": a, "b": b, "c": c, "m": rng.randint(15, 60)}
    lo = rng.randint(20, 40)
    return {"kind": "batched", "count": rng.randint(2, 24), "lo": lo, "hi": lo + rng.randint(1, 50)}


# --------------------------------------------------------------------------
# separable operators
# --------------------------------------------------------------------------
class Pencil:
    """A = sum over the axes of K_axis times the other axes' M, B = product of
    the lumped masses D (B = I and M = I for the 5- and 7-point operators)."""

    def __init__(self, dims, points, rng, vmax=0.5):
        self.dims = [int(d) for d in dims]
        self.points = points
        self.n = math.prod(self.dims)
        self.k, self.d, self.m, self.mu, self.v = [], [], [], [], []
        for s in self.dims:
            if points == 27:  # linear elements on a slightly stretched grid
                h = rng.uniform(0.9, 1.1, s + 1)
                K = np.diag(1 / h[:-1] + 1 / h[1:]) - np.diag(1 / h[1:-1], 1) - np.diag(1 / h[1:-1], -1)
                D = 0.5 * (h[:-1] + h[1:])
                M = np.diag(D) - MASS * K
            elif s == 1:  # the axis that a 2D grid does not have
                K, D, M = np.zeros((1, 1)), np.ones(1), np.eye(1)
            else:
                axes = sum(x > 1 for x in self.dims)
                K = np.diag(2.0 + rng.uniform(0.0, vmax / axes, s)) - np.eye(s, k=1) - np.eye(s, k=-1)
                D, M = np.ones(s), np.eye(s)
            q = 1 / np.sqrt(D)
            mu, u = np.linalg.eigh(q[:, None] * K * q)
            for name, x in (("k", K), ("d", D), ("m", M), ("mu", mu), ("v", q[:, None] * u)):
                getattr(self, name).append(x)
        mus, c = self.mu, MASS if points == 27 else 0.0
        g = np.meshgrid(*mus, indexing="ij")
        lev = sum(g[i] * math.prod((1 - c * g[j]) for j in range(len(g)) if j != i) for i in range(len(g)))
        self.levels = lev  # every eigenvalue, on the grid of mode numbers
        self.order = np.argsort(lev, axis=None, kind="stable")
        self.lam = lev.ravel()[self.order]

    def interval(self, count):
        """Emax between the count-th eigenvalue and the next."""
        return float(0.5 * (self.lam[count - 1] + self.lam[count]))

    def csr(self, device):
        """0-based full-storage CSR of A (int32, int32, float64), columns ascending."""
        nd = len(self.dims)
        strides = [math.prod(self.dims[i + 1:]) for i in range(nd)]
        idx = torch.arange(self.n, device=device)
        coord = [(idx // strides[i]) % self.dims[i] for i in range(nd)]
        kt = [torch.as_tensor(x, device=device) for x in self.k]
        mt = [torch.as_tensor(x, device=device) for x in self.m]
        cols, vals, oks = [], [], []
        offs = [[]]
        for s in self.dims:
            offs = [o + [e] for o in offs for e in ((-1, 0, 1) if s > 1 else (0,))]
        for o in offs:
            if self.points != 27 and sum(e != 0 for e in o) > 1:
                continue
            ok = torch.ones(self.n, dtype=torch.bool, device=device)
            to, step = [], 0
            for i in range(nd):
                t = coord[i] + o[i]
                ok &= (t >= 0) & (t < self.dims[i])
                to.append(t.clamp(0, self.dims[i] - 1))
                step += o[i] * strides[i]
            v = torch.zeros(self.n, dtype=F64, device=device)
            for i in range(nd):
                t = kt[i][coord[i], to[i]]
                for j in range(nd):
                    if j != i:
                        t = t * mt[j][coord[j], to[j]]
                v += t
            cols.append(idx + step)
            vals.append(v)
            oks.append(ok)
        ok = torch.stack(oks, 1)
        ia = torch.zeros(self.n + 1, dtype=torch.int32, device=device)
        ia[1:] = torch.cumsum(ok.sum(1), 0)
        return ia, torch.stack(cols, 1)[ok].to(torch.int32), torch.stack(vals, 1)[ok]

    def mass(self, device):
        """Diagonal of B."""
        d = torch.ones(1, dtype=F64, device=device)
        for x in self.d:
            d = (d[:, None] * torch.as_tensor(x, device=device)[None, :]).reshape(-1)
        return d

    def vectors(self, m, device):
        """The m lowest eigenvectors (B-orthonormal), n x m."""
        at = np.unravel_index(self.order[:m], self.dims)
        x = torch.ones((1, m), dtype=F64, device=device)
        for i in range(len(self.dims)):
            v = torch.as_tensor(self.v[i], device=device)[:, torch.as_tensor(at[i], device=device)]
            x = (x[:, None, :] * v[None, :, :]).reshape(-1, m)
        return x

    def along(self, mats, x):
        """The Kronecker product of the axes' matrices applied to the columns of x."""
        m = x.shape[1]
        for i, a in enumerate(mats):
            left = math.prod(self.dims[:i])
            x = torch.matmul(torch.as_tensor(a, device=x.device), x.reshape(left, self.dims[i], -1))
            x = x.reshape(-1, m)
        return x

    def apply(self, x):
        """A x."""
        y = torch.zeros_like(x)
        for i, s in enumerate(self.dims):
            if s == 1:
                continue
            y += self.along([self.k[j] if j == i else self.m[j] for j in range(len(self.dims))], x)
        return y

    def function(self, f, x):
        """V f(Lambda) V^T B x, V all eigenvectors."""
        b = self.mass(x.device)[:, None]
        y = self.along([v.T for v in self.v], b * x)
        y *= torch.as_tensor(f(self.levels).reshape(-1, 1), device=x.device)
        return self.along(self.v, y)


def _rng(seed):
    return np.random.default_rng([int(seed), 2002])


def _dims(case):
    return [case["a"], case["b"], case["c"]]


def _pencil(case, seed):
    return Pencil(_dims(case), case.get("points", 7), _rng(seed))


def _noise(seed, shape):
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    return torch.randn(shape, dtype=F64, device="cuda", generator=g)


def _wanted(case):
    return max(1, int(case["m"] / 1.5))  # the subspace is half as large again as the wanted space


def _fpm(ne, ratio, mixed, tol, maxit, batch, eps=10):
    f = feast.feast_init()
    f[1], f[2], f[3], f[17], f[41], f[44], f[45], f[49] = ne, eps, 60, ratio, int(mixed), tol, maxit, batch
    return f


# --------------------------------------------------------------------------
# one kind after the other: prepare, run, exact
# --------------------------------------------------------------------------
def _filter_state(case, seed):
    """Ritz pairs of a late refinement loop: eigenvectors off by `noise` (mostly
    the modes that a contour pass damps least, those not far above the interval),
    and their residual block as right-hand side."""
    p = _pencil(case, seed)
    m = case["m"]
    emax = p.interval(_wanted(case))
    b = p.mass("cuda")
    e = p.function(lambda lev: 1 / (1 + (lev / emax) ** 2), _noise(seed, (p.n, m)))
    x = p.vectors(m, "cuda") + case["noise"] * e / (b[:, None] * e * e).sum(0).sqrt()
    lam = torch.as_tensor(p.lam[:m].copy(), device="cuda")
    r = p.apply(x) - b[:, None] * x * lam
    return p, x, lam, b, r


def prepare_filter(case, seed):
    p, x, lam, b, r = _filter_state(case, seed)
    st = {"n": p.n, "m": case["m"], "R": r, "X": x, "lam": lam, "emax": p.interval(_wanted(case)),
          "fpm": _fpm(case["ne"], case["ratio"], case["mixed"], case["tol"], case["maxit"], case["batch"]),
          "Q": torch.zeros_like(x), "ib": None, "jb": None, "b": None}
    st["ia"], st["ja"], st["a"] = p.csr("cuda")
    if case["points"] == 27:
        st["ib"] = torch.arange(p.n + 1, dtype=torch.int32, device="cuda")
        st["jb"] = st["ib"][:-1].clone()
        st["b"] = b
    return st


def run_filter(s):
    _lib.feast_filter_dev(s["n"], s["ia"], s["ja"], s["a"], s["ib"], s["jb"], s["b"], s["m"], s["R"], s["X"], s["lam"],
                          1, s["fpm"], 0.0, s["emax"], s["Q"])
    return {"Q": s["Q"]}


def exact_filter(case, seed):
    """The filter with exact solves is a function of the matrix."""
    p, x, _, _, _ = _filter_state(case, seed)
    ne, a = case["ne"], case["ratio"] / 100.0
    t, w = np.polynomial.legendre.leggauss(ne)
    th = 0.5 * math.pi * (1 - t)
    r = 0.5 * p.interval(_wanted(case))
    z = r + r * np.cos(th) + 1j * a * r * np.sin(th)
    w = 0.5 * w * r * (a * np.cos(th) + 1j * np.sin(th))
    return {"Q": p.function(lambda lev: sum((we / (ze - lev)).real for ze, we in zip(z, w)), x)}


def _block(p, m, seed, size):
    x = p.vectors(m, "cuda")
    return x + size / math.sqrt(p.n) * _noise(seed, x.shape)


def prepare_project(case, seed):
    p = _pencil(case, seed)
    m = case["m"]
    q = _block(p, m, seed, 1e-2)
    return {"n": p.n, "m": m, "Q": q, "AQ": p.apply(q), "A": torch.zeros((m, m), dtype=F64, device="cuda"),
            "B": torch.zeros((m, m), dtype=F64, device="cuda")}


def run_project(s):
    _lib.feast_gram_oz_dev(s["n"], s["m"], s["Q"], s["AQ"], s["A"])
    _lib.feast_gram_oz_dev(s["n"], s["m"], s["Q"], s["Q"], s["B"])
    return {"A": s["A"], "B": s["B"]}


def exact_project(case, seed):
    s = prepare_project(case, seed)
    out = {}
    for name, y in (("A", s["AQ"]), ("B", s["Q"])):
        c = torch.triu(s["Q"].t() @ y)
        out[name] = c + torch.triu(c, 1).t()
    return out


def prepare_ritz(case, seed):
    p = _pencil(case, seed)
    m = case["m"]
    q = _block(p, m, seed, 1e-1)
    v, _ = torch.linalg.qr(_noise(seed + 1, (m, m)))
    st = {"pencil": p, "n": p.n, "m": m, "Q": q, "V": v.contiguous(), "lam": torch.as_tensor(p.lam[:m].copy(), device="cuda"),
          "X": torch.zeros_like(q), "R": torch.zeros_like(q), "res": torch.zeros(m, dtype=F64, device="cuda"),
          "ib": None, "jb": None, "b": None, "alpha": float(p.lam[m - 1])}
    st["ia"], st["ja"], st["a"] = p.csr("cuda")
    if case["points"] == 27:
        st["ib"] = torch.arange(p.n + 1, dtype=torch.int32, device="cuda")
        st["jb"] = st["ib"][:-1].clone()
        st["b"] = p.mass("cuda")
    return st


def run_ritz(s):
    _lib.feast_gemm_oz_dev(s["n"], s["m"], s["m"], s["Q"], s["V"], s["X"])
    _lib.feast_residual_dev(s["n"], s["ia"], s["ja"], s["a"], s["ib"], s["jb"], s["b"], s["m"], s["X"], s["lam"],
                            s["alpha"], s["R"], s["res"])
    return {"X": s["X"], "R": s["R"], "res": s["res"]}


def exact_ritz(case, seed):
    s = prepare_ritz(case, seed)
    p = s["pencil"]
    x = s["Q"] @ s["V"]
    bx = p.mass("cuda")[:, None] * x
    r = p.apply(x) - bx * s["lam"]
    return {"X": x, "R": r, "res": r.norm(dim=0) / (s["alpha"] * bx.norm(dim=0))}


def _symmetric(seed, m):
    e = _noise(seed, (m, m)) / math.sqrt(m)
    return 0.5 * (e + e.t())


def prepare_reduced(case, seed):
    """Projections in the basis of the last Ritz vectors: eigenvalues of a 3D
    Laplacian on the diagonal, coupled by what the last contour pass changed."""
    m = case["m"]
    side = max(8, int(round((8 * m) ** (1 / 3))) + 2)
    lam = torch.as_tensor(Pencil([side] * 3, 7, _rng(seed)).lam[:m].copy(), device="cuda")
    a = torch.diag(lam) + 1e-3 * _symmetric(seed, m)
    b = torch.eye(m, dtype=F64, device="cuda") + 1e-2 * _symmetric(seed + 1, m)
    return {"m": m, "A": a.contiguous(), "B": b.contiguous(), "lam": torch.zeros(m, dtype=F64, device="cuda"),
            "V": torch.zeros((m, m), dtype=F64, device="cuda")}


def _fix_signs(v):
    """Eigenvectors are known up to their sign: the first component positive."""
    return v * torch.where(v[0] < 0, -1.0, 1.0).to(v.dtype)


def run_reduced(s):
    mk = _lib.feast_reduced_eig_dev(s["m"], s["A"], s["B"], s["lam"], s["V"])
    return {"live": mk, "lam": s["lam"], "V": _fix_signs(s["V"])}


def exact_reduced(case, seed):
    s = prepare_reduced(case, seed)
    a, b = s["A"].cpu(), s["B"].cpu()
    g = torch.linalg.cholesky(b)
    c = torch.linalg.solve_triangular(g, torch.linalg.solve_triangular(g, a, upper=False).t(), upper=False)
    lam, w = torch.linalg.eigh(0.5 * (c + c.t()))
    return {"live": None, "lam": lam, "V": _fix_signs(torch.linalg.solve_triangular(g.t(), w, upper=True))}


def prepare_grad(case, seed):
    p = _pencil(case, seed)
    st = {"n": p.n, "m": case["m"], "X": p.vectors(case["m"], "cuda"), "w": _noise(seed, case["m"])}
    st["ia"], st["ja"], a = p.csr("cuda")
    st["grad"] = torch.zeros_like(a)
    return st


def run_grad(s):
    _lib.feast_eig_grad_dev(s["n"], s["ia"], s["ja"], s["m"], s["X"], s["w"], s["grad"])
    return {"grad": s["grad"]}


def _pattern_gradient(ia, ja, x, w):
    rows = torch.repeat_interleave(torch.arange(len(ia) - 1, device=ia.device), (ia[1:] - ia[:-1]).long())
    g = [((x[r] * w) * x[c]).sum(1) for r, c in zip(rows.split(1 << 20), ja.long().split(1 << 20))]
    return torch.cat(g)


def exact_grad(case, seed):
    s = prepare_grad(case, seed)
    return {"grad": _pattern_gradient(s["ia"], s["ja"], s["X"], s["w"])}


def prepare_autograd(case, seed):
    p = _pencil(case, seed)
    ia, ja, a = p.csr("cuda")
    return {"n": p.n, "m": case["m"], "ia": ia, "ja": ja, "a": a.requires_grad_(), "emax": p.interval(_wanted(case)),
            "fpm": _fpm(8, 200, case["mixed"], 2, 80, 1)}


def run_autograd(s):
    s["a"].grad = None
    lam = feast_eigenvalues(s["a"], s["ia"], s["ja"], s["n"], 0.0, s["emax"], s["m"], s["fpm"])
    lam.sum().backward()
    return {"lam": lam.detach(), "grad": s["a"].grad}


def exact_autograd(case, seed):
    p = _pencil(case, seed)
    k = _wanted(case)
    ia, ja, _ = p.csr("cuda")
    return {"lam": torch.as_tensor(p.lam[:k].copy()),
            "grad": _pattern_gradient(ia, ja, p.vectors(k, "cuda"), torch.ones(k, dtype=F64, device="cuda"))}


def prepare_host(case, seed):
    """tridiag(-1, 2, -1) with a weak random potential on the host."""
    p = Pencil([case["n"]], 7, _rng(seed), vmax=4.0 / case["n"])
    ia, ja, a = (t.numpy() for t in p.csr("cpu"))
    return {"pencil": p, "n": p.n, "m": case["m"], "ia": ia, "ja": ja, "a": a, "emax": p.interval(_wanted(case)),
            "fpm": _fpm(8, 30, True, 2, 400, 1, eps=12)}


def run_host(s):
    r = feast.feast_scsr_solve("F", s["n"], s["a"], s["ia"], s["ja"], fpm=s["fpm"], emin=0.0, emax=s["emax"], m0=s["m"])
    if r.info not in (0, 3):
        raise RuntimeError(f"info {r.info}")
    x = r.X[:, :r.M]
    return {"count": r.M, "E": r.E[:r.M], "X": x * np.where(x[0] < 0, -1.0, 1.0)}


def exact_host(case, seed):
    s = prepare_host(case, seed)
    p = s["pencil"]
    k = _wanted(case)
    x = p.vectors(k, "cpu")
    return {"count": None, "E": torch.as_tensor(p.lam[:k].copy()), "X": _fix_signs(x)}


def prepare_hermitian(case, seed):
    """D A D^H with random phases D: every off-diagonal entry complex, A's spectrum."""
    p = _pencil(case, seed)
    ia, ja, a = p.csr("cuda")
    theta = torch.as_tensor(_rng(seed + 1).uniform(0.0, 2 * math.pi, p.n), device="cuda")
    rows = torch.repeat_interleave(torch.arange(p.n, device="cuda"), (ia[1:] - ia[:-1]).long())
    ph = theta[rows] - theta[ja.long()]
    m = case["m"]
    return {"n": p.n, "m": m, "ia": ia, "ja": ja, "a": torch.complex(a * torch.cos(ph), a * torch.sin(ph)),
            "emax": p.interval(_wanted(case)), "fpm": _fpm(8, 200, True, 2, 80, 1),
            "x": torch.zeros((m, p.n), dtype=torch.complex128, device="cuda")}


def run_hermitian(s):
    r = feast.feast_hcsr_solve_dev(s["n"], s["ia"], s["ja"], s["a"], fpm=s["fpm"], emin=0.0, emax=s["emax"], m0=s["m"],
                                   x=s["x"])
    if r.info not in (0, 3):
        raise RuntimeError(f"info {r.info}")
    v = torch.view_as_real(r.X[:r.M])
    return {"count": r.M, "E": r.E[:r.M], "density": (v * v).sum((0, 2))}  # |x|^2 needs no choice of phases


def exact_hermitian(case, seed):
    p = _pencil(case, seed)
    k = _wanted(case)
    return {"count": None, "E": torch.as_tensor(p.lam[:k].copy()), "density": p.vectors(k, "cuda").square().sum(1)}


def _batch_sizes(case):
    """(side, wanted eigenvalues) of every problem: part of the case, whatever the seed."""
    rng = np.random.default_rng([case["count"], case["lo"], case["hi"]])
    out = []
    for _ in range(case["count"]):
        side = int(math.exp(rng.uniform(math.log(case["lo"]), math.log(case["hi"] + 1))))
        out.append((side, int(rng.integers(8, 65))))
    return out


def _batch_pencils(case, seed):
    rng = _rng(seed)
    return [(Pencil([side, side, 1], 5, rng, vmax=1.0), k) for side, k in _batch_sizes(case)]


def prepare_batched(case, seed):
    problems = []
    for p, k in _batch_pencils(case, seed):
        ia, ja, a = (t.numpy() for t in p.csr("cpu"))
        emax = p.interval(k)
        problems.append({"n": p.n, "a": a, "ia": ia, "ja": ja, "emin": float(p.lam[0] - 0.05 * (emax - p.lam[0])),
                         "emax": emax, "m0": int(math.ceil(1.5 * k))})
    return {"problems": problems, "fpm": _fpm(8, 200, True, 2, 80, 0)}


def run_batched(s):
    st, res = feast.feast_scsr_solve_batched(s["problems"], s["fpm"])
    if st != 0 or any(r.info not in (0, 3) for r in res):
        raise RuntimeError(f"status {st}, info {[r.info for r in res]}")
    return {"counts": np.array([r.M for r in res]), "E": np.concatenate([r.E[:r.M] for r in res]),
            "density": np.concatenate([np.einsum("ij,ij->i", r.X[:, :r.M], r.X[:, :r.M]) for r in res])}


def exact_batched(case, seed):
    e, d = [], []
    for p, k in _batch_pencils(case, seed):
        e.append(torch.as_tensor(p.lam[:k].copy()))
        d.append(p.vectors(k, "cpu").square().sum(1))
    return {"counts": None, "E": torch.cat(e), "density": torch.cat(d)}


# --------------------------------------------------------------------------
# the measured interface
# --------------------------------------------------------------------------
def prepare(case, seed):
    s = globals()["prepare_" + case["kind"]](case, int(seed))
    s["kind"] = case["kind"]
    return s


def run(state):
    return globals()["run_" + state["kind"]](state)


def exact(case, seed):
    return globals()["exact_" + case["kind"]](case, int(seed))


def _nnz(dims, points):
    if points == 27:
        return math.prod(3 * s - 2 for s in dims)
    n = math.prod(dims)
    return n + 2 * sum(n // s * (s - 1) for s in dims)


def work(case):
    """Bytes of the inputs and outputs, once each; operations of the sums that
    define the outputs (iterative solves: one product with the matrix per
    contour node and column, one Rayleigh-Ritz step)."""
    kind = case["kind"]
    if kind == "reduced":
        m = case["m"]
        return {"bytes": 8.0 * (3 * m * m + m), "flops": 9.0 * m ** 3}
    if kind == "host":
        n, m = case["n"], case["m"]
        return {"bytes": 12.0 * 3 * n + 8.0 * n * m, "flops": 8.0 * 8 * m * 3 * n + 6.0 * n * m * m}
    if kind == "batched":
        nbytes = flops = 0.0
        for side, k in _batch_sizes(case):
            n, m = side * side, 1.5 * k
            nbytes += 12.0 * 5 * n + 8.0 * n * m
            flops += 8.0 * 8 * m * 5 * n + 6.0 * n * m * m
        return {"bytes": nbytes, "flops": flops}
    dims, m = _dims(case), case["m"]
    n, points = math.prod(dims), case.get("points", 7)
    nnz = _nnz(dims, points)
    csr, block = 12.0 * nnz + 4.0 * n, 8.0 * n * m
    if kind == "filter":
        return {"bytes": csr + 3 * block, "flops": 8.0 * case["ne"] * m * nnz}
    if kind == "project":
        return {"bytes": 2 * block + 16.0 * m * m, "flops": 4.0 * n * m * m}
    if kind == "ritz":
        return {"bytes": 3 * block + csr, "flops": 2.0 * n * m * m + 2.0 * nnz * m}
    if kind == "grad":
        return {"bytes": block + 12.0 * nnz + 4.0 * n, "flops": 2.0 * nnz * m}
    if kind == "autograd":
        return {"bytes": csr + 8.0 * nnz + block, "flops": 8.0 * 8 * m * nnz + 6.0 * n * m * m}
    return {"bytes": 20.0 * nnz + 2 * block, "flops": 16.0 * 8 * m * nnz + 24.0 * n * m * m}  # hermitian
