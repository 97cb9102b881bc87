"""Kernels at the sizes where their tiling changes form: the gradient (columns
in registers up to 128, in shared memory beyond; rows of 0 to 9 entries), the
sliced Ritz product (contractions up to 320 with resident row slices, longer
ones in pieces), the Jacobi teams (one thread's work up to many CTAs, odd
sizes, tiny and huge entries) and a batch whose problems fall into several
classes of rows."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import feast_workloads as fw  # noqa: E402

pytestmark = pytest.mark.gpu
EPS = 2.0 ** -53


@pytest.fixture(scope="module")
def pkg():
    import paper_2002_04807_gb300 as pkg

    pkg.library()
    return pkg


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), device="cuda")


@pytest.mark.parametrize("m", [1, 7, 8, 127, 128, 129, 131, 300])
def test_gradient_columns_and_row_lengths(pkg, m):
    """g_p = sum_k w_k x_ik x_jk over a pattern with rows of 0, 1, ... 9 entries."""
    rng = np.random.default_rng(m)
    n = 41
    lens = np.arange(n) % 10
    ia = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    ja = np.concatenate([np.sort(rng.choice(n, k, replace=False)) for k in lens]).astype(np.int32)
    X, w = rng.standard_normal((n, m)), rng.standard_normal(m)
    g = torch.zeros(ja.size, dtype=torch.float64, device="cuda")
    pkg.feast_eig_grad_dev(n, dev(ia), dev(ja), m, dev(X), dev(w), g)
    row = np.repeat(np.arange(n), lens)
    ref = np.einsum("pk,k,pk->p", X[row], w, X[ja])
    size = np.einsum("pk,k,pk->p", np.abs(X[row]), np.abs(w), np.abs(X[ja]))
    got = g.cpu().numpy()
    # (m + 2) roundings on either side, of at most the sum of the terms' sizes
    assert (np.abs(got - ref) <= 2 * (m + 2) * EPS * size).all()


@pytest.mark.parametrize("n,k,m", [(1, 1, 1), (31, 319, 9), (33, 320, 8), (33, 321, 8), (65, 15, 321), (64, 640, 16)])
def test_sliced_product_contraction_lengths(pkg, n, k, m):
    rng = np.random.default_rng(n + m + k)
    A, V = rng.standard_normal((n, k)), rng.standard_normal((k, m))
    C = torch.zeros((n, m), dtype=torch.float64, device="cuda")
    pkg.feast_gemm_oz_dev(n, k, m, dev(A), dev(V), C)
    ref = (A.astype(np.longdouble) @ V.astype(np.longdouble)).astype(np.float64)
    # k dropped terms of 2^-55 of the row's and the column's scale (up to twice their
    # largest entries) and an FP64 sum over at most k / 16 partial results
    tol = (k * 2.0 ** -53 + 4 * EPS) * np.abs(A).max(1)[:, None] * np.abs(V).max(0)[None, :] * 2
    assert (np.abs(C.cpu().numpy() - ref) <= tol).all()


@pytest.mark.parametrize("size", [1.0, 1e-170, 1e170])
@pytest.mark.parametrize("m", [1, 2, 3, 16, 33, 64, 129, 201])
def test_jacobi_sizes_and_scales(pkg, m, size):
    rng = np.random.default_rng(m)
    S = rng.standard_normal((m, m))
    S = (S + S.T) * 0.5
    lam, V = torch.zeros(m, dtype=torch.float64, device="cuda"), torch.zeros((m, m), dtype=torch.float64, device="cuda")
    pkg.feast_sym_eig_dev(m, dev(S * size), lam, V)
    ev = np.linalg.eigvalsh(S)
    v = V.cpu().numpy()
    # both sides are backward stable: a modest multiple of m eps of the norm
    tol = 20 * m * EPS * max(np.abs(ev).max(), 1e-300)
    assert np.abs(lam.cpu().numpy() / size - ev).max() <= tol
    assert np.abs(v.T @ v - np.eye(m)).max() <= 20 * m * EPS
    assert np.abs(S @ v - v * ev[None, :]).max() <= 2 * m ** 0.5 * tol


@pytest.mark.parametrize("mixed", [1, 0])
def test_batch_of_several_row_classes(pkg, mixed):
    """2D problems of 25 to 9,604 rows in one call, against the closed form
    4 - 2 cos(i pi / (s + 1)) - 2 cos(j pi / (t + 1))."""
    probs, want = [], []
    rng = np.random.default_rng(4)
    for s, t in ((5, 5), (98, 98), (17, 30), (64, 64), (86, 81)):
        A = fw._grid_laplacian((s, t), np.zeros((s, t)))
        ev = np.sort((4 - 2 * np.cos(np.arange(1, s + 1) * np.pi / (s + 1))[:, None]
                      - 2 * np.cos(np.arange(1, t + 1) * np.pi / (t + 1))[None, :]).ravel())
        k = 4 + int(np.argmax(np.diff(ev[4:9])))  # the widest gap after the 5th to 8th
        m0 = min(16, A.n)
        probs.append(dict(n=A.n, a=A.data, ia=A.indptr, ja=A.indices, emin=0.0, emax=0.5 * (ev[k] + ev[k + 1]), m0=m0,
                          x0=rng.standard_normal((A.n, m0))))
        want.append(ev[: k + 1])
    f = pkg.feast_init()
    f[1], f[2], f[3], f[4], f[17], f[41], f[44], f[45] = 8, 10, 40, 1, 100, mixed, 2, 200
    st, res = pkg.feast_scsr_solve_batched(probs, f)
    assert st == 0
    for r, ev in zip(res, want):
        assert r.info == 0 and r.M == len(ev)
        assert np.abs(r.E[: r.M] - ev).max() <= 1e-10  # no more than the residuals that the solve stops at
