"""The contour filter of B = I problems from one Krylov space per column
(k_krylov.cu), against the CPU oracle's filter and against the per-node COCG
path (fpm(51) > 0), at the sizes where its tiling can go wrong: fewer rows than
one pass of a CTA, one row over, ragged tiles of columns, one node, more nodes
than a warp has lanes, rows longer than one packed chunk, empty and zero
columns, patterns that leave the CTAs' row ranges."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import feast_workloads as fw  # noqa: E402
import oracle as O  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import paper_2002_04807_gb300 as pkg

    pkg.library()
    return pkg


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), device="cuda")


def _grid(shape, seed):
    rng = np.random.default_rng(seed)
    return fw._grid_laplacian(shape, rng.uniform(0.0, 0.5, size=shape))


def _scattered(n, k, seed):
    """Symmetric, diagonally dominant, k random neighbours per row, one long row."""
    rng = np.random.default_rng(seed)
    r = np.concatenate([np.repeat(np.arange(n), k), np.zeros(min(n, 40), dtype=int)])
    c = np.concatenate([rng.integers(0, n, n * k), np.arange(min(n, 40))])
    keep = r != c
    r, c = r[keep], c[keep]
    v = -rng.uniform(0.2, 1.0, r.size)
    A = fw.csr_from_coo(n, np.concatenate([r, c]), np.concatenate([c, r]), np.concatenate([v, v]))
    row = np.repeat(np.arange(n), np.diff(A.indptr))
    d = np.bincount(row, np.abs(A.data), minlength=n) + 0.5
    i = np.arange(n)
    return fw.csr_from_coo(n, np.concatenate([row, i]), np.concatenate([A.indices, i]), np.concatenate([A.data, d]))


def _bipartite(n, seed):
    """Weighted chain whose rows store no diagonal entry."""
    w = np.random.default_rng(seed).uniform(0.5, 1.5, n - 1)
    i = np.arange(n - 1)
    return fw.csr_from_coo(n, np.concatenate([i, i + 1]), np.concatenate([i + 1, i]), np.concatenate([w, w]))


def _run(pkg, A, Y, ne, mixed, emax, rows=0, rii=0, X=None, lam=None, maxit=3000, ratio=100):
    n, m = Y.shape
    fpm = pkg.feast_init()
    fpm[1], fpm[17], fpm[41], fpm[50] = ne, ratio, mixed, rows
    fpm[44], fpm[45] = (6 if mixed else 12), maxit
    Q = torch.full((n, m), 7.0, dtype=torch.float64, device="cuda")
    it = pkg.feast_filter_dev(n, dev(A.indptr), dev(A.indices), dev(A.data), None, None, None, m, dev(Y),
                              dev(Y if X is None else X), dev(np.zeros(m) if lam is None else lam), rii, fpm, 0.0, emax, Q)
    return Q.cpu().numpy(), it


@pytest.mark.parametrize("mixed", [0, 1])
@pytest.mark.parametrize("shape,m,ne", [((1,), 1, 8), ((5,), 3, 1), ((63,), 17, 8), ((65,), 32, 4), ((8, 8), 33, 8),
                                        ((7, 9, 11), 16, 8), ((16, 16, 16), 40, 8), ((10, 10), 5, 40)])
def test_filter_matches_oracle(pkg, shape, m, ne, mixed):
    """Inner solves to 1e-12 (1e-6 in complex FP32) of the direct solves: the
    same bounds as the COCG filter's test."""
    A = _grid(shape, sum(shape) + m)
    m = min(m, A.n)
    emax = 1.0 + 2.0 * len(shape)
    Y = fw.gaussian_block(A.n, m, 3)
    Q, it = _run(pkg, A, Y, ne, mixed, emax)
    ref = O.filter_block(A, None, ne, 0.0, emax, 1.0, Y)
    assert it >= 1
    err = np.abs(Q - ref).max() / np.abs(ref).max()
    assert err < (1e-8 if not mixed else 2e-3), err


@pytest.mark.parametrize("mixed", [0, 1])
@pytest.mark.parametrize("kind", ["grid", "scattered", "dense_rows", "no_diagonal"])
def test_residual_form_matches_cocg_per_node(pkg, kind, mixed):
    """Residual-inverse form, a zero and a live column side by side: the iterates
    of the COCG path.  The reference is that path in FP64; the block may be as
    far from it as that path's own variants are (another order of summation,
    single precision), and no further, beside the COCG filter's own bound."""
    A = {"grid": lambda: _grid((13, 12, 11), 4), "scattered": lambda: _scattered(900, 3, 5),
         "dense_rows": lambda: fw.stencil27_spd(9, np.random.default_rng(6)),
         "no_diagonal": lambda: _bipartite(700, 7)}[kind]()
    m, ne = 37, 8
    R = fw.gaussian_block(A.n, m, 8)
    R[:, 5] = 0.0
    X = fw.gaussian_block(A.n, m, 9)
    emax = float(np.quantile(A.data[A.data > 0], 0.5))
    lam = np.linspace(0.1, 0.9, m) * emax
    kw = dict(rii=1, X=X, lam=lam, maxit=60)
    Q, it = _run(pkg, A, R, ne, mixed, emax, **kw)
    ref, it2 = _run(pkg, A, R, ne, 0, emax, rows=256, **kw)
    C, _ = _run(pkg, A, R, ne, mixed, emax, rows=128, **kw)
    assert abs(it - it2) <= 2 * ne, (it, it2)  # a step more or less where a residual meets the tolerance
    size = np.abs(ref).max()
    err, own = np.abs(Q - ref).max() / size, np.abs(C - ref).max() / size
    assert err < max(1e-8 if not mixed else 2e-3, 1.5 * own), (err, own)
    z, w = O.contour_gauss(ne, 0.0, emax, 1.0)
    rho = sum(np.real(we / (ze - lam[5])) for ze, we in zip(z, w))
    assert np.abs(Q[:, 5] - rho * X[:, 5]).max() <= 1e-12 * np.abs(rho * X[:, 5]).max()


def test_columns_with_infinities_do_not_reach_the_others(pkg):
    """A column that holds NaN contributes nothing, as on the COCG path, and its
    neighbours in the tile are untouched."""
    A = _grid((9, 9), 2)
    Y = fw.gaussian_block(A.n, 6, 1)
    ref, _ = _run(pkg, A, Y, 8, 1, 3.0)
    Y[4, 2] = np.nan
    Q, _ = _run(pkg, A, Y, 8, 1, 3.0)
    keep = [0, 1, 3, 4, 5]
    assert np.array_equal(Q[:, keep], ref[:, keep])
    assert np.array_equal(Q[:, 2], np.zeros(A.n))


def test_reruns_are_identical(pkg):
    A = _grid((20, 21, 19), 3)
    Y = fw.gaussian_block(A.n, 50, 2)
    a, _ = _run(pkg, A, Y, 8, 1, 2.0, maxit=40)
    b, _ = _run(pkg, A, Y, 8, 1, 2.0, maxit=40)
    assert np.array_equal(a, b)


@pytest.mark.parametrize("extreme", [False, True])
def test_smaller_workspace_goes_without_bases(pkg, monkeypatch, extreme):
    """A workspace that does not hold the Krylov bases is used for one COCG per node
    (launches of its streaming step in the profile); one that holds neither is refused."""
    from paper_2002_04807_gb300 import _lib

    p = fw.laplace3d_potential(side=16, count=16, m0=24, seed=4)
    ia, ja, av = dev(p.A.indptr), dev(p.A.indices), dev(p.A.data)
    ev = np.linalg.eigvalsh(p.A.to_dense())
    f = pkg.feast_init()
    f[1], f[2], f[3], f[17], f[41], f[44], f[45], f[52] = 8, 10, 40, 100, 1, 2, 200, 1
    f[39] = -1 if extreme else 0
    need = _lib.feast_scsr_workspace_bytes(p.n, av.numel(), 0, 24, f)
    for work, steps in ((need, False), (need - 1, True)):
        monkeypatch.setattr(_lib, "feast_scsr_workspace_bytes", lambda *a, w=work: w)
        if extreme:
            r = _lib.feast_scsr_extreme_dev(p.n, ia, ja, av, fpm=f.copy(), m0=24)
        else:
            r = _lib.feast_scsr_solve_dev(p.n, ia, ja, av, fpm=f.copy(), emin=p.emin, emax=p.emax, m0=24)
        assert r.info == 0 and r.M > 0
        want = ev[: r.M] if extreme else ev[(ev >= p.emin) & (ev <= p.emax)]
        assert r.M == len(want) and np.abs(r.E[: r.M] - want).max() <= 1e-9
        assert (pkg.feast_last_profile()["cocg_b_launches"] > 0) == steps
    monkeypatch.setattr(_lib, "feast_scsr_workspace_bytes", lambda *a: 1 << 20)
    if extreme:
        r = _lib.feast_scsr_extreme_dev(p.n, ia, ja, av, fpm=f.copy(), m0=24)
    else:
        r = _lib.feast_scsr_solve_dev(p.n, ia, ja, av, fpm=f.copy(), emin=p.emin, emax=p.emax, m0=24)
    assert r.info == -120


def test_smaller_workspace_hermitian(pkg):
    """The same for a complex Hermitian problem (BiCG per node)."""
    p = fw.laplace3d_gauge(side=12, count=12, m0=20, ratio=100)
    n = p.n
    args = (n, dev(p.A.indptr), dev(p.A.indices), dev(np.asarray(p.A.data, dtype=np.complex128)))
    f = pkg.feast_init()
    f[1], f[2], f[3], f[17], f[41], f[44], f[45] = 8, 10, 40, 100, 1, 2, 200
    need = pkg.feast_hcsr_workspace_bytes(n, args[3].numel(), 0, 20, f)
    got = []
    for work in (need, need - 1):
        r = pkg.feast_hcsr_solve_dev(*args, fpm=f.copy(), emin=p.emin, emax=p.emax, m0=20,
                                     work=torch.empty(work, dtype=torch.uint8, device="cuda"))
        assert r.info == 0 and r.M > 0
        got.append(r.E[: r.M])
    assert len(got[0]) == len(got[1]) and np.abs(got[0] - got[1]).max() <= 1e-9
    r = pkg.feast_hcsr_solve_dev(*args, fpm=f.copy(), emin=p.emin, emax=p.emax, m0=20,
                                 work=torch.empty(1 << 16, dtype=torch.uint8, device="cuda"))
    assert r.info == -120
