"""The mixed form's PCG at the sizes where its inner product changes path: every row of A in shared memory
(384 sites), part of them (4,056 sites: 13 of 27 rows per block), all streamed because n is no multiple of
4 (486) or beyond the cached product's 4,096 sites (4,368).

Bounds.  The solve stops at ||r|| <= tol ||rhs||, checked against an FP64 residual of the projected
charges (a factor of 10 for the projection and its roundings); the charges differ from the direct solve's
by at most cond(A) tol, cond(A) < 1e3 at a site spacing of five Gaussian widths."""
import numpy as np
import pytest

from paper_2509_24742_gb300 import srbe, workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(8, 8), (9, 9), (26, 26), (28, 26)])
def test_mixed_pcg_reaches_the_direct_charges(nx, ny):
    tol = 1e-8
    s = wl.make_slab("pcg", (0.25 * nx, 0.25 * ny, 12.0), nx, ny, 60, 1, alpha=3.5, eta_inv=19.79, rc=1.0, P=30, M=2,
                     seed=7)
    with srbe.from_slab(s, precision=srbe.MIXED) as ctx:
        ctx.sample_k(3, 0)
        Q0, psi0, _ = ctx.solve_charges()
        ctx.set_solver(srbe.PCG, tol=tol, maxit=5000, warm=srbe.WARM_ZERO)
        Q1, psi1, _ = ctx.solve_charges()
        it, res = ctx.solver_stats()
        res64 = ctx.charge_residual()
    assert 0 < it < 5000 and res <= tol and res64 <= 10 * tol
    assert np.linalg.norm(Q1 - Q0) <= 1e3 * tol * np.linalg.norm(Q0)
    assert abs(psi1 - psi0) <= 1e3 * tol * abs(psi0)


@pytest.mark.parametrize("nx,ny,gone", [(3, 2, 0), (4, 3, 0), (17, 1, 2), (6, 3, 0), (7, 4, 0), (11, 3, 2)])
def test_mixed_pcg_on_small_electrodes(nx, ny, gone):
    """36, 72, 100, 108, 168 and 196 sites: the last of a block's eight column segments of the cached product
    start at or past the end of the row (100 and 196 also have blocks with fewer rows than others).  The
    bounds above: the sites are at least as far apart."""
    tol = 1e-8
    s = wl.make_slab("pcg", (max(1.5, 0.25 * nx), 1.5, 12.0), nx, ny, 40, 1, alpha=3.5, eta_inv=19.79, rc=1.0, P=30,
                     M=2, seed=7)
    keep = np.arange(gone, s.R.shape[0])
    s.R, s.side = s.R[keep], s.side[keep]
    with srbe.from_slab(s, precision=srbe.MIXED) as ctx:
        ctx.sample_k(3, 0)
        Q0, psi0, _ = ctx.solve_charges()
        ctx.set_solver(srbe.PCG, tol=tol, maxit=5000, warm=srbe.WARM_ZERO)
        for _ in range(3):
            Q1, psi1, _ = ctx.solve_charges()
            it, res = ctx.solver_stats()
            assert 0 < it < 5000 and res <= tol and ctx.charge_residual() <= 10 * tol
            assert np.linalg.norm(Q1 - Q0) <= 1e3 * tol * np.linalg.norm(Q0)
            assert abs(psi1 - psi0) <= 1e3 * tol * abs(psi0)
