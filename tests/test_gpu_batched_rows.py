"""Batches of matrices with rows of unlike lengths: each problem's eigenpairs,
against closed forms and dense references."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import feast_workloads as fw  # noqa: E402

pytestmark = pytest.mark.gpu


def _grid5(a, b, seed):
    rng = np.random.default_rng(seed)
    A = fw._grid_laplacian((a, b), rng.uniform(0, 0.3, (a, b)))
    return A, np.linalg.eigvalsh(A.to_dense())


def _chain(n, seed):
    """Weighted chain whose rows store no diagonal entry: with n odd, nnz + 7 n is odd."""
    w = np.random.default_rng(seed).uniform(0.5, 1.5, n - 1)
    i = np.arange(n - 1)
    A = fw.csr_from_coo(n, np.concatenate([i, i + 1]), np.concatenate([i + 1, i]), np.concatenate([w, w]))
    return A, np.linalg.eigvalsh(A.to_dense())


def _grid9(a, b, seed):
    """9-point stencil: K1 x I + I x K2 + 0.1 K1 x K2."""
    rng = np.random.default_rng(seed)
    K = [np.diag(2.0 + rng.uniform(0, 0.2, s)) - np.eye(s, k=1) - np.eye(s, k=-1) for s in (a, b)]
    rows, cols, vals = [], [], []
    for i1, j1 in zip(*np.nonzero(K[0])):
        for i2, j2 in zip(*np.nonzero(K[1])):
            rows.append(i1 * b + i2)
            cols.append(j1 * b + j2)
            vals.append(K[0][i1, j1] * (i2 == j2) + K[1][i2, j2] * (i1 == j1) + 0.1 * K[0][i1, j1] * K[1][i2, j2])
    mu = [np.linalg.eigvalsh(k) for k in K]
    ev = np.sort((mu[0][:, None] + mu[1] + 0.1 * mu[0][:, None] * mu[1]).ravel())
    return fw.csr_from_coo(a * b, np.array(rows), np.array(cols), np.array(vals)), ev


def _ring(n, seed):
    """Eight neighbours and no diagonal entry: nine packed entries."""
    w = np.random.default_rng(seed).uniform(0.5, 1.0, (4, n))
    i = np.arange(n)
    r = np.concatenate([i] * 4 + [(i + d) % n for d in range(1, 5)])
    c = np.concatenate([(i + d) % n for d in range(1, 5)] + [i] * 4)
    v = -np.concatenate([w.ravel()] * 2)
    A = fw.csr_from_coo(n, r, c, v)
    return A, np.linalg.eigvalsh(A.to_dense())


def _check(pkg, cases, mixed, rows=0, b=None):
    batch = []
    for A, ev in cases:
        k = 9 + int(np.argmax(np.diff(ev[9:16])))  # the edge in the widest gap after the tenth
        emax = 0.5 * (ev[k] + ev[k + 1])
        batch.append(dict(n=A.n, a=A.data, ia=A.indptr, ja=A.indices, emin=ev[0] - 0.05 * (emax - ev[0]), emax=emax,
                          m0=k + 12))
        if b is not None:
            B = b(A.n)
            batch[-1].update(b=B.data, ib=B.indptr, jb=B.indices)
    f = pkg.feast_init()
    f[1], f[2], f[3], f[17], f[41], f[44], f[45], f[50] = 8, 10, 40, 200, mixed, 2, 120, rows
    st, res = pkg.feast_scsr_solve_batched(batch, f)
    assert st == 0
    for (A, ev), q, r in zip(cases, batch, res):
        want = ev[(ev >= q["emin"]) & (ev <= q["emax"])]
        assert r.info == 0 and r.M == len(want)
        assert np.abs(r.E[: r.M] - want).max() <= 1e-9 * np.abs(want).max()
        X = r.X[:, : r.M]
        assert np.abs(X.T @ X - np.eye(r.M)).max() <= 1e-10
        assert r.res[: r.M].max() <= 1e-6  # stops on the trace


@pytest.mark.parametrize("mixed", [0, 1])
@pytest.mark.parametrize("rows", [0, 128])
@pytest.mark.parametrize("with_b", [False, True])
def test_problems_after_rows_without_diagonal_entries(rows, mixed, with_b):
    """The packed entries of a problem start on a 16-byte boundary whatever the
    problems before it store."""
    import paper_2002_04807_gb300 as pkg

    cases = [_chain(231, 1), _grid5(24, 19, 2), _chain(57, 3), _chain(400, 4), _grid5(13, 17, 5)]
    _check(pkg, cases, mixed, rows, (lambda n: fw.identity_csr(n)) if with_b else None)


@pytest.mark.parametrize("mixed", [0, 1])
@pytest.mark.parametrize("kinds", [("5", "9"), ("9", "ring"), ("ring", "5", "9", "9big", "5")])
def test_rows_of_different_lengths_in_a_batch(kinds, mixed):
    """Only the problems with rows of more than eight entries take the filter's cached form."""
    import paper_2002_04807_gb300 as pkg

    make = {"5": lambda s: _grid5(24, 19, s), "9": lambda s: _grid9(21, 17, s), "9big": lambda s: _grid9(87, 83, s),
            "ring": lambda s: _ring(331, s)}
    _check(pkg, [make[k](7 + q) for q, k in enumerate(kinds)], mixed)
