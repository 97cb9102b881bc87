"""The staged COCG step A (problems with a diagonal B) and the barrier of the
one-Krylov-space filter (B = I), each by the profile's own word: iteration caps
against the oracle's iterates, and waits that run out."""
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


def _case(pkg, diag_b, side=12):
    p = fw.laplace3d_potential(side=side, count=10, m0=18, seed=3)
    B = fw.diagonal_csr(np.random.default_rng(21).uniform(1.0, 2.0, p.n)) if diag_b else None
    return p, B


def _form(pkg, p, B, mixed):
    """Profile of a short solve of the same matrices."""
    f = pkg.feast_init()
    f[1], f[2], f[3], f[17], f[41], f[44], f[45], f[52] = 8, 3, 2, 100, mixed, 1, 60, 1
    kw = {} if B is None else dict(b=B.data, ib=B.indptr, jb=B.indices)
    pkg.feast_scsr_solve("F", p.n, p.A.data, p.A.indptr, p.A.indices, fpm=f, emin=p.emin, emax=p.emax, m0=18, **kw)
    return pkg.feast_last_profile()


def _filter(pkg, p, B, R, mixed, tol, maxit):
    n, m = R.shape
    f = pkg.feast_init()
    f[1], f[17], f[41], f[44], f[45] = 8, 100, mixed, tol, maxit
    b = (None,) * 3 if B is None else (dev(B.indptr), dev(B.indices), dev(B.data))
    Q = torch.zeros((n, m), dtype=torch.float64, device="cuda")
    it = pkg.feast_filter_dev(n, dev(p.A.indptr), dev(p.A.indices), dev(p.A.data), *b, m, dev(R), dev(R),
                              dev(np.zeros(m)), 0, f, p.emin, p.emax, Q)
    return Q.cpu().numpy(), it


@pytest.mark.parametrize("mixed", [0, 1])
@pytest.mark.parametrize("cap", [1, 6])
def test_staged_step_a_at_the_iteration_cap(pkg, mixed, cap):
    """As test_filter_iteration_cap_matches_capped_cocg, with its bounds, for a
    problem that runs the staged step."""
    p, B = _case(pkg, True)
    assert _form(pkg, p, B, mixed)["step_a_staged"] == 1
    Y = fw.gaussian_block(p.n, 18, 8)
    Q, it = _filter(pkg, p, B, Y, mixed, 16, cap)
    assert it == cap
    z, w = O.contour_gauss(8, p.emin, p.emax, 1.0)
    ref, scale = np.zeros(Y.shape), np.zeros(Y.shape)
    for ze, we in zip(z, w):
        Ye, its = O.shifted_solve(p.A, B, complex(ze), Y, method="cocg", tol=0.0, maxit=cap)
        assert (its == cap).all()
        ref += np.real(we * Ye)
        scale += np.abs(we * Ye)
    err = np.abs(Q - ref).max() / scale.max()
    assert err < (1e-12 if not mixed else 1e-4), err


@pytest.mark.parametrize("mixed", [0, 1])
def test_staged_step_a_wait_limit(pkg, mixed):
    """With a one-cycle limit a wait for staged copies sees them land within the
    hardware's own try-wait interval or gives up with -4; afterwards the call
    returns what it did before."""
    p, B = _case(pkg, True, side=16)
    assert _form(pkg, p, B, mixed)["step_a_staged"] == 1
    R = fw.gaussian_block(p.n, 18, 9)
    want, _ = _filter(pkg, p, B, R, mixed, 5, 400)
    pkg.feast_set_wait_limit(1)
    try:
        try:
            _filter(pkg, p, B, R, mixed, 5, 400)
        except pkg.FeastError as exc:
            assert "-4" in str(exc), exc
    finally:
        pkg.feast_set_wait_limit(0)
    torch.cuda.synchronize()
    assert np.array_equal(_filter(pkg, p, B, R, mixed, 5, 400)[0], want)


@pytest.mark.parametrize("mixed", [0, 1])
def test_krylov_barrier_wait_limit(pkg, mixed):
    """With a one-cycle limit a CTA that arrives before the others gives up: -4 and
    the filter's own message, and the call works again."""
    p, B = _case(pkg, False, side=16)
    prof = _form(pkg, p, B, mixed)
    assert prof["cocg_b_launches"] == 0 and prof["step_a_staged"] == 1 and prof["step_a_grid"] > 1
    R = fw.gaussian_block(p.n, 18, 9)
    want, _ = _filter(pkg, p, B, R, mixed, 5, 400)
    pkg.feast_set_wait_limit(1)
    try:
        with pytest.raises(pkg.FeastError, match="-4.*Krylov steps"):
            _filter(pkg, p, B, R, mixed, 5, 400)
    finally:
        pkg.feast_set_wait_limit(0)
    torch.cuda.synchronize()
    assert np.array_equal(_filter(pkg, p, B, R, mixed, 5, 400)[0], want)
