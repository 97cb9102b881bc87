"""What feast_last_profile says of a contour filter from one Krylov space per column."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import feast_workloads as fw  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mixed", [0, 1])
@pytest.mark.parametrize("kind", ["line", "grid", "long_rows"])
def test_krylov_profile_describes_the_plan(kind, mixed):
    """Resident form: 512 threads per CTA, a thread per 16 bytes of a row, so a warp
    takes 32 / lanes rows at once, and the CTAs' ranges (multiples of 16 rows) cover
    the problem; rows of more than eight entries: blocks of 256 rows."""
    import paper_2002_04807_gb300 as pkg

    if kind == "grid":
        p = fw.laplace3d_potential(side=14, count=10, m0=18, seed=2)
        A, emax = p.A, p.emax
    else:
        A = fw.laplacian_1d(300) if kind == "line" else fw.stencil27_spd(10, np.random.default_rng(1))
        ev = np.linalg.eigvalsh(A.to_dense())
        emax = 0.5 * (ev[9] + ev[10])
    f = pkg.feast_init()
    f[1], f[2], f[3], f[17], f[41], f[44], f[45], f[52] = 8, 9, 30, 100, mixed, 2, 400, 1
    r = pkg.feast_scsr_solve("F", A.n, A.data, A.indptr, A.indices, fpm=f, emin=0.0, emax=emax, m0=18)
    assert r.info == 0 and r.M > 0
    pr = {k: int(v) for k, v in pkg.feast_last_profile().items()}
    assert pr["cocg_b_launches"] == 0 and pr["W"] == pr["mt"] and pr["groups"] == -(-18 // pr["W"])
    if kind == "long_rows":
        assert (pr["step_a_staged"], pr["step_a_rows_per_item"]) == (0, 256)
        return
    lanes = pr["W"] // (4 if mixed else 2)
    assert pr["step_a_staged"] == 1 and pr["step_a_rows_per_item"] == 32 // lanes
    assert pr["step_a_staged_rows"] % 16 == 0
    assert pr["step_a_grid"] * pr["step_a_staged_rows"] >= A.n
