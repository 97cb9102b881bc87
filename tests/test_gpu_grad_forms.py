"""The gradient kernel's forms (lanes per row, entries in flight, chunks of
columns) at the rows and columns where one takes over from another, against the
sums in FP64 on the host."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import feast_workloads as fw  # noqa: E402

pytestmark = pytest.mark.gpu


def _matrix(n):
    """n rows of 1, 3, 5, 8 and 9 entries in turn, the columns around the row, one row empty."""
    rng = np.random.default_rng(n)
    ia, ja = [0], []
    for i in range(n):
        k = 0 if i == n // 2 else (1, 3, 5, 8, 9)[i % 5]
        ja.append(np.sort(rng.choice(np.arange(max(0, i - 40), min(n, i + 41)), size=min(k, n), replace=False)))
        ia.append(ia[-1] + len(ja[-1]))
    return np.array(ia, dtype=np.int32), np.concatenate(ja).astype(np.int32)


def _reference(ia, ja, X, w):
    row = np.repeat(np.arange(len(ia) - 1), np.diff(ia))
    return (np.einsum("pk,pk->p", X[row] * w, X[ja]), np.einsum("pk,pk->p", np.abs(X[row] * w), np.abs(X[ja])))


# 16 and 32 rows per SM: 2,432 and 4,864 rows on 152
@pytest.mark.parametrize("n,m", [(70, 63), (70, 64), (70, 257), (70, 2048), (2431, 65), (2432, 64), (2600, 128), (2600, 129),
                                 (2600, 256), (2600, 257), (2600, 512), (2600, 513), (4863, 897), (4864, 513), (4900, 600),
                                 (4900, 896), (4900, 897), (4900, 1030), (4900, 2048)])
def test_gradient_forms(n, m):
    import paper_2002_04807_gb300 as pkg

    ia, ja = _matrix(n)
    rng = np.random.default_rng(m)
    X, w = rng.standard_normal((n, m)), rng.standard_normal(m)
    dev = lambda v: torch.as_tensor(v, device="cuda")  # noqa: E731
    out = torch.full((len(ja),), 7.0, dtype=torch.float64, device="cuda")
    for _ in range(2):  # nothing is added to what the array held
        pkg.feast_eig_grad_dev(n, dev(ia), dev(ja), m, dev(X), dev(w), out)
    ref, size = _reference(ia, ja, X, w)
    # m products and sums, in any order: m eps of the sum of their sizes
    assert (np.abs(out.cpu().numpy() - ref) <= m * 2.0 ** -52 * size).all()


@pytest.mark.parametrize("n,m", [(90, 70), (3000, 300), (5000, 600)])
def test_gradient_forms_of_a_triangle_and_of_b(n, m):
    """Lower-triangle pattern (an off-diagonal value stands for two entries) and the
    weights -g lambda of B's entries."""
    import paper_2002_04807_gb300 as pkg

    A = fw.laplacian_1d(n)
    row = np.repeat(np.arange(n), np.diff(A.indptr))
    keep = A.indices <= row
    ia = np.concatenate([[0], np.cumsum(np.bincount(row[keep], minlength=n))]).astype(np.int32)
    ja = A.indices[keep]
    rng = np.random.default_rng(3)
    X, g, e = rng.standard_normal((n, m)), rng.standard_normal(m), rng.uniform(1, 2, m)
    ga, gb = pkg.feast_scsr_grad("L", n, ia, ja, X, g, ib=ia, jb=ja, e=e)
    two = np.where(np.repeat(np.arange(n), np.diff(ia)) == ja, 1.0, 2.0)
    for got, w in ((ga, g), (gb, -g * e)):
        ref, size = _reference(ia, ja, X, w)
        assert (np.abs(got - two * ref) <= (m + 2) * 2.0 ** -52 * two * size).all()
