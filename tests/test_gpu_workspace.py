"""Workspaces of the real device drivers as a Python caller passes them: sizes
between the least and the full one, and a device that does not hold the full one."""
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


def _case(pkg, entry):
    p = fw.laplace3d_potential(side=16, count=16, m0=24, seed=4)
    f = pkg.feast_init()
    f[1], f[2], f[3], f[17], f[41], f[44], f[45], f[52] = 8, 10, 40, 100, 1, 2, 400, 1
    f[39] = -1 if entry == "extreme" else 0
    csr = tuple(torch.as_tensor(v, device="cuda") for v in (p.A.indptr, p.A.indices, p.A.data))

    def solve(work=None):
        if entry == "extreme":
            r = pkg.feast_scsr_extreme_dev(p.n, *csr, fpm=f.copy(), m0=24, work=work)
        elif entry == "nodes":
            z, w = pkg.feast_contour_nodes(8, p.emin, p.emax, 100)
            r = pkg.feast_scsr_solve_dev_x(p.n, *csr, z, w, fpm=f.copy(), emin=p.emin, emax=p.emax, m0=24, work=work)
        else:
            r = pkg.feast_scsr_solve_dev(p.n, *csr, fpm=f.copy(), emin=p.emin, emax=p.emax, m0=24, work=work)
        assert r.info == 0
        # launches of COCG's streaming step: the solve went without bases
        return r.E[: r.M].copy(), pkg.feast_last_profile()["cocg_b_launches"] > 0

    sizes = [g(p.n, p.A.nnz, 0, 24, f) for g in (pkg.feast_scsr_workspace_min_bytes, pkg.feast_scsr_workspace_bytes)]
    return solve, sizes


@pytest.mark.parametrize("entry", ["interval", "nodes", "extreme"])
def test_a_callers_workspace_is_used(pkg, entry):
    solve, (least, full) = _case(pkg, entry)
    assert least < full
    ref, without = solve()
    assert not without
    for size, used in ((least, True), (full - 1, True), (full, False), (least - 1, False)):
        e, without = solve(torch.empty(size, dtype=torch.uint8, device="cuda"))
        assert without == used, size
        assert len(e) == len(ref) and np.abs(e - ref).max() <= 1e-9


@pytest.mark.parametrize("entry", ["interval", "nodes", "extreme"])
def test_a_device_without_room_for_the_bases(pkg, entry):
    """With torch's allocator limited to between the two sizes the calls run
    without bases instead of raising an out-of-memory error."""
    solve, (least, full) = _case(pkg, entry)
    ref, _ = solve()
    torch.cuda.empty_cache()
    total = torch.cuda.get_device_properties(0).total_memory
    room = torch.cuda.memory_reserved() + least + (full - least) / 2
    assert full - least > 64 << 20  # the allocator's own blocks do not matter
    torch.cuda.set_per_process_memory_fraction(room / total)
    try:
        e, without = solve()
    finally:
        torch.cuda.set_per_process_memory_fraction(1.0)
    assert without and len(e) == len(ref) and np.abs(e - ref).max() <= 1e-9


def test_batch_on_a_device_without_room_for_the_bases(pkg):
    """Most of the device is held by tensors: the 7 GB of Krylov bases of this
    batch do not fit, the 0.2 GB of its COCG do."""
    f = pkg.feast_init()
    f[1], f[2], f[3], f[17], f[41], f[44], f[45] = 8, 10, 40, 100, 1, 2, 4000
    probs = [fw.laplace3d_potential(side=16, count=16, m0=24, seed=s) for s in range(6)]
    batch = [dict(n=p.n, a=p.A.data, ia=p.A.indptr, ja=p.A.indices, emin=p.emin, emax=p.emax, m0=24) for p in probs]
    st, ref = pkg.feast_scsr_solve_batched(batch, f.copy())
    assert st == 0
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    hold = torch.empty(free - (3 << 30), dtype=torch.uint8, device="cuda")
    try:
        st, got = pkg.feast_scsr_solve_batched(batch, f.copy())
    finally:
        del hold
        torch.cuda.empty_cache()
    assert st == 0
    for r, r0 in zip(got, ref):
        assert r.info == r0.info == 0 and r.M == r0.M > 0
        assert np.abs(r.E[: r.M] - r0.E[: r0.M]).max() <= 1e-9


@pytest.mark.parametrize("mixed", [0, 1])
def test_a_cap_that_stands_for_none_takes_no_memory(pkg, mixed):
    """fpm(46) = 10^6 on a few hundred rows: the space has no more dimensions than
    rows, so neither the workspace nor a filter call's own grows with such a cap, and
    the block is that of a cap the pass does not meet."""
    A = fw.laplacian_1d(300)
    csr = [torch.as_tensor(v, device="cuda") for v in (A.indptr, A.indices, A.data)]
    R = torch.as_tensor(fw.gaussian_block(300, 12, 3), device="cuda")
    out = []
    for cap in (400, 1_000_000):
        f = pkg.feast_init()
        f[1], f[17], f[41], f[44], f[45] = 8, 100, mixed, (4 if mixed else 10), cap
        assert pkg.feast_scsr_workspace_bytes(300, A.nnz, 0, 12, f) < 256 << 20
        Q = torch.zeros_like(R)
        it = pkg.feast_filter_dev(300, *csr, None, None, None, 12, R, R, torch.zeros(12, dtype=torch.float64, device="cuda"),
                                  0, f, 0.0, 1.0, Q)
        assert it < 400
        out.append(Q.cpu().numpy())
    assert np.abs(out[0] - out[1]).max() <= 1e-3 * np.abs(out[0]).max()  # both solved to the tolerance
