"""The contour filter of B = I problems (k_krylov.cu) does not depend on the units
of A: with A, the interval and the Ritz values multiplied by a power of two
every operation of a pass is multiplied by one, and the block must come out bit
for bit; a shifted spectrum must stop as the unshifted one does."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import feast_workloads as fw  # noqa: E402

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


def _filter(pkg, A, Y, mixed, emin, emax, scale=1.0, rii=0, X=None, lam=None, tol=None):
    n, m = Y.shape
    fpm = pkg.feast_init()
    fpm[1], fpm[17], fpm[41], fpm[49] = 8, 100, mixed, 1
    fpm[44], fpm[45] = (tol or (4 if mixed else 10)), 600
    Q = torch.full((n, m), 7.0, dtype=torch.float64, device="cuda")
    it = pkg.feast_filter_dev(n, dev(A.indptr), dev(A.indices), dev(A.data * scale), None, None, None, m,
                              dev(Y * (scale if rii else 1.0)), dev(Y if X is None else X),
                              dev(np.zeros(m) if lam is None else lam * scale), rii, fpm, emin * scale, emax * scale, Q)
    return Q.cpu().numpy(), it


@pytest.mark.parametrize("power", [-100, -77, 64, 100])
@pytest.mark.parametrize("kind,mixed,rii", [("line", 0, 0), ("grid", 0, 0), ("grid", 0, 1), ("long_rows", 0, 0),
                                            ("line", 1, 0), ("grid", 1, 0), ("long_rows", 1, 0)])
def test_filter_is_independent_of_units(pkg, kind, mixed, rii, power):
    """One CTA per tile, teams of CTAs, and rows of more than eight entries."""
    A = {"line": lambda: _grid((130,), 1), "grid": lambda: _grid((19, 17, 13), 2),
         "long_rows": lambda: fw.stencil27_spd(9, np.random.default_rng(3))}[kind]()
    Y = fw.gaussian_block(A.n, 21, 4)
    kw = dict(rii=rii)
    if rii:
        kw.update(X=fw.gaussian_block(A.n, 21, 5), lam=np.linspace(0.1, 0.9, 21))
    ref, it0 = _filter(pkg, A, Y, mixed, 0.0, 1.0, **kw)
    Q, it = _filter(pkg, A, Y, mixed, 0.0, 1.0, scale=2.0 ** power, **kw)
    assert it == it0 > 8
    assert np.array_equal(Q, ref)


def test_values_beyond_the_rows_are_not_read(pkg):
    """Arrays longer than ia[n], as a caller with room to spare passes them."""
    A = _grid((40,), 9)
    Y = fw.gaussian_block(A.n, 4, 10)
    ref, _ = _filter(pkg, A, Y, 1, 0.0, 1.0)
    A.indices = np.concatenate([A.indices, np.zeros(9, dtype=A.indices.dtype)])
    A.data = np.concatenate([A.data, np.full(9, 1e300)])
    Q, _ = _filter(pkg, A, Y, 1, 0.0, 1.0)
    assert np.array_equal(Q, ref)


def test_filter_of_a_shifted_spectrum_stops_alike(pkg):
    """A + s I with a shift of 2^26 on a spectrum of width 4 (both exact): the
    nodes are rounded to 7.5e-9, a quarter of a millionth of their distance (0.03)
    to the spectrum, and the FP64 recurrences keep 27 of their 53 bits, so a pair
    stops within a few steps of the unshifted one."""
    n, s = 300, 2.0 ** 26
    A = _grid((n,), 0)
    d = A.indices == np.repeat(np.arange(n), np.diff(A.indptr))
    A.data[d] = 2.0
    Y = fw.gaussian_block(n, 5, 6)
    ref, it0 = _filter(pkg, A, Y, 0, 0.0, 1.0, tol=8)
    A.data[d] += s
    Q, it = _filter(pkg, A, Y, 0, s, s + 1.0, tol=8)
    assert abs(it - it0) <= 5 * 8, (it, it0)
    assert np.abs(Q - ref).max() <= 1e-5 * np.abs(ref).max()


def _fpm(pkg):
    f = pkg.feast_init()
    f[1], f[2], f[3], f[17], f[41], f[44], f[45] = 8, 11, 30, 100, 0, 3, 400
    return f


def _same(r, r0, scale, emax):
    assert r0.info == 0 and r.info == 0 and r.M == r0.M > 0
    assert np.abs(r.E[: r.M] / scale - r0.E[: r0.M]).max() <= 1e-11 * emax


@pytest.mark.parametrize("power", [-100, 100])
def test_fp64_solves_are_independent_of_units(pkg, power):
    """Whole FP64 solves, real, batched and Hermitian, in units of 1e-30 and 1e30."""
    s = 2.0 ** power
    p = fw.laplace3d_potential(side=10, count=10, m0=18, seed=3)
    run = lambda c: pkg.feast_scsr_solve("F", p.n, p.A.data * c, p.A.indptr, p.A.indices, fpm=_fpm(pkg),  # noqa: E731
                                         emin=p.emin * c, emax=p.emax * c, m0=18)
    r0 = run(1.0)
    _same(run(s), r0, s, p.emax)
    one = lambda c: dict(n=p.n, a=p.A.data * c, ia=p.A.indptr, ja=p.A.indices, emin=p.emin * c,  # noqa: E731
                         emax=p.emax * c, m0=18)
    st, rs = pkg.feast_scsr_solve_batched([one(s), one(1.0)], _fpm(pkg))
    assert st == 0
    _same(rs[0], r0, s, p.emax)
    _same(rs[1], r0, 1.0, p.emax)
    h = fw.laplace3d_gauge(side=8, count=8, m0=14, ratio=100)
    runh = lambda c: pkg.feast_hcsr_solve("F", h.n, np.asarray(h.A.data) * c, h.A.indptr, h.A.indices,  # noqa: E731
                                          fpm=_fpm(pkg), emin=h.emin * c, emax=h.emax * c, m0=14)
    _same(runh(s), runh(1.0), s, h.emax)
