"""COCG step A with a producer warp (cocg_step_ws): its entries carry no test for
padding and its warps share no barrier, so it is compared with the gather
through the caches (fpm(51) > 0) and with double precision where that can go
wrong: rows of fewer chunks than their neighbours, a last block that is not full
(down to one row), lines shorter and longer than a block, one column over a
group, B = I and diagonal."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import feast_workloads as fw  # noqa: E402

pytestmark = pytest.mark.gpu

STEPS = 20
# Every form computes the same 20 COCG iterates.  In single precision each step
# rounds three vectors a few times (some 4 eps of their largest entry), carried on
# by step lengths of order 10 at most: 20 * 4 * 10 * 2^-24 = 5e-5 of the largest value.
TOL = 1e-4


@pytest.mark.parametrize("shape,m", [((4, 4, 96), 33), ((6, 40, 97), 32), ((11, 41, 45), 5), ((3, 50, 61), 65),
                                     ((48, 48, 48), 8), ((1, 40, 64), 8)])
@pytest.mark.parametrize("diag_b", [True, False])
def test_staged_gather_agrees(shape, m, diag_b):
    import paper_2002_04807_gb300 as pkg

    rng = np.random.default_rng(5)
    A = fw.stencil27_spd(0, rng, shape=shape)
    n = A.n
    B = fw.diagonal_csr(rng.uniform(1.0, 2.0, n)) if diag_b else fw.diagonal_csr(np.ones(n))
    dev = lambda x: torch.as_tensor(np.ascontiguousarray(x), device="cuda")  # noqa: E731
    R = dev(rng.standard_normal((n, m)))
    a = [dev(A.indptr), dev(A.indices), dev(A.data), dev(B.indptr), dev(B.indices), dev(B.data)]
    out = {}
    for name, mixed, rows in (("staged", 1, 0), ("cached", 1, 256), ("fp64", 0, 256)):
        fpm = pkg.feast_init()
        fpm[1], fpm[17], fpm[41], fpm[50] = 2, 100, mixed, rows
        fpm[44], fpm[45], fpm[49] = 15, STEPS, 1
        Q = torch.zeros((n, m), dtype=torch.float64, device="cuda")
        pkg.feast_filter_dev(n, *a, m, R, R, dev(np.zeros(m)), 0, fpm, 0.0, 1.0, Q)
        out[name] = Q.cpu().numpy()
    scale = np.abs(out["fp64"]).max()
    assert np.isfinite(out["staged"]).all()
    assert np.abs(out["staged"] - out["cached"]).max() <= TOL * scale
    assert np.abs(out["staged"] - out["fp64"]).max() <= TOL * scale


def test_producer_wait_limit_is_bounded():
    """With a one-cycle limit each wait of the form either sees its copies land
    within the hardware's own try-wait interval or gives up: the call returns with
    the error (-4) or a result, and works again with the default limit."""
    import paper_2002_04807_gb300 as pkg

    rng = np.random.default_rng(7)
    A = fw.stencil27_spd(0, rng, shape=(12, 48, 48))
    B = fw.diagonal_csr(rng.uniform(1.0, 2.0, A.n))
    n, m = A.n, 16
    dev = lambda x: torch.as_tensor(np.ascontiguousarray(x), device="cuda")  # noqa: E731
    R = dev(rng.standard_normal((n, m)))
    a = [dev(A.indptr), dev(A.indices), dev(A.data), dev(B.indptr), dev(B.indices), dev(B.data)]
    fpm = pkg.feast_init()
    fpm[1], fpm[17], fpm[41], fpm[44], fpm[45], fpm[49] = 2, 100, 1, 15, STEPS, 1

    def call():
        Q = torch.zeros((n, m), dtype=torch.float64, device="cuda")
        pkg.feast_filter_dev(n, *a, m, R, R, dev(np.zeros(m)), 0, fpm, 0.0, 1.0, Q)
        return Q

    want = call()
    pkg.feast_set_wait_limit(1)
    try:
        try:
            call()
        except pkg.FeastError as exc:
            assert "-4" in str(exc), exc
    finally:
        pkg.feast_set_wait_limit(0)
    torch.cuda.synchronize()
    assert torch.equal(call(), want)
