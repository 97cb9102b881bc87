"""Error of the sliced products where it is one-sided and as large as it gets:
columns of one value whose digits below the first are all at an end of their
range, so that every term leaves the same pairs of digits out."""
from fractions import Fraction

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

# x = F 2^-55, F = 64 2^48 + digits of 2^40, 2^32, ... 1 (the last a multiple of 4: 53 bits)
LOW = [2 ** (8 * k) for k in range(1, 6)]
VALUES = {"high": 64 * 2 ** 48 + 127 * sum(LOW) + 124, "low": 66 * 2 ** 48 - 128 * sum(LOW) - 128}
# per term: 6 pairs of level 9 and what follows (6.03 2^14 2^-70), two roundings to 2^-56, the scale
# of both factors being 1: below 9 2^-56
TERM = Fraction(9, 2 ** 56)


def _bound(terms, exact, roundings=1):
    return terms * TERM + roundings * abs(exact) * Fraction(1, 2 ** 53)


@pytest.mark.parametrize("n,m", [(4096, 40), (1000, 3), (262144, 33)])
def test_projection_of_constant_columns(n, m):
    import paper_2002_04807_gb300 as pkg

    x = [(-1) ** j * list(VALUES.values())[j // 2 % 2] for j in range(m)]
    X = torch.as_tensor(np.array([v * 2.0 ** -55 for v in x])).to("cuda").expand(n, m).contiguous()
    C = torch.zeros((m, m), dtype=torch.float64, device="cuda")
    pkg.feast_gram_oz_dev(n, m, X, X, C)
    C = C.cpu().numpy()
    for i in range(m):
        for j in range(m):
            exact = n * Fraction(x[i] * x[j], 2 ** 110)
            # the row splits (at most 456, of 256 rows and more) are rounded one by one and summed
            splits = min(456, -(-n // 256))
            assert abs(Fraction(float(C[i, j])) - exact) <= _bound(n, exact, 2 * splits), (i, j)


@pytest.mark.parametrize("m", [7, 150, 320, 330])
def test_ritz_product_of_constant_rows(m):
    """Row slices in shared memory up to 320 terms, the tiled product beyond."""
    import paper_2002_04807_gb300 as pkg

    n, k = 70, 4
    v = list(VALUES.values())
    rows = [(-1) ** i * v[i // 2 % 2] for i in range(n)]
    cols = [v[0], v[1], -v[0], -v[1]]
    A = torch.as_tensor(np.array([r * 2.0 ** -55 for r in rows])).to("cuda")[:, None].expand(n, m).contiguous()
    V = torch.as_tensor(np.array([c * 2.0 ** -55 for c in cols])).to("cuda").expand(m, k).contiguous()
    C = torch.zeros((n, k), dtype=torch.float64, device="cuda")
    pkg.feast_gemm_oz_dev(n, m, k, A, V, C)
    C = C.cpu().numpy()
    for i in range(n):
        for j in range(k):
            exact = m * Fraction(rows[i] * cols[j], 2 ** 110)
            assert abs(Fraction(float(C[i, j])) - exact) <= _bound(m, exact), (i, j)
