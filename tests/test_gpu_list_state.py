"""Calls that change the Verlet lists' layout between two passes: what follows sees lists of the present layout."""
import copy

import numpy as np
import pytest

from paper_2509_24742_gb300 import srbe, workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [srbe.FP64, srbe.MIXED])
def test_descriptors_after_a_new_skin(precision):
    """A new skin gives the lists another capacity (here 160 entries, then 320 and 128); descriptors asked for before
    the next pass are those of the same configuration: sums of the same FP32 terms, up to 300 of one sign, in another
    order, within 300 x 6e-8."""
    s = wl.make_slab("skin", (2.26, 2.02, 12.0), 9, 8, 39, 3, alpha=3.5, eta_inv=19.79, rc=1.2, P=40, M=2, seed=3,
                     placement="lattice")
    with srbe.from_slab(s, precision=precision) as c:
        c.sample_k(1, 0)
        c.forces()
        D = c.descriptors()
        for skin in (0.6, 0.02, 1.0):
            c.set_skin(skin)
            E = c.descriptors()
            assert np.abs(E - D).max() <= 2e-5 * np.abs(D).max()


@pytest.mark.parametrize("precision,solver", [(srbe.FP64, srbe.DIRECT), (srbe.MIXED, srbe.DIRECT), (srbe.FP64, srbe.PCG),
                                              (srbe.MIXED, srbe.PCG)])
def test_another_electrode_on_the_same_context(precision, solver):
    """srbe_set_electrode again, with more and with fewer sites, over the same ions: the next pass is a fresh
    context's, bit for bit (lists built anew by both, an iterative solve from a zero start)."""
    a = wl.make_slab("first", (2.26, 2.02, 12.0), 9, 8, 39, 3, alpha=3.5, eta_inv=19.79, rc=1.2, P=40, M=2, seed=3,
                     placement="lattice")
    c = srbe.from_slab(a, precision=precision, alpha_A=1.7)
    for nx, ny, gone in ((9, 8, 0), (10, 9, 0), (6, 7, 1), (10, 9, 3)):
        s = wl.make_slab("next", a.box, nx, ny, 39, 3, alpha=3.5, eta_inv=19.79, rc=1.2, P=40, M=2, seed=3,
                         placement="lattice")
        s.r, s.q = a.r, a.q
        s.R, s.side = s.R[gone:], s.side[gone:]
        out = []
        for ctx in (c, srbe.from_slab(s, precision=precision, alpha_A=1.7)):
            if ctx is c:
                ctx.set_electrode(s.R, s.side)
            if solver == srbe.PCG and (ctx is not c or nx == 9):
                ctx.set_solver(srbe.PCG, tol=1e-10, maxit=4000, warm=srbe.WARM_ZERO)
            ctx.sample_k(5, 1)
            out.append(ctx.forces()[:2])
            if ctx is not c:
                ctx.close()
        assert all(np.array_equal(x, y) for x, y in zip(*out))
    with pytest.raises(srbe.SrbeError):
        c.set_electrode(s.R, np.zeros_like(s.side))          # one side empty: refused, the electrode stays
    assert np.array_equal(c.forces()[0], out[0][0])
    c.close()


def test_skin_beyond_the_stencil():
    """Cells are chosen for the default skin (0.1 nm): in a box of 4 nm they are 2/3 nm wide and two of them cover
    1.333 nm, so lists for rc + 0.3 nm lack some pairs.  Ions that start 1.34 to 1.49 nm apart and come within rc by
    moving less than half the skin each are seen all the same: a fresh context's forces."""
    rng = np.random.default_rng(4)
    s = wl.make_slab("skin", (4.0, 4.0, 12.0), 8, 8, 60, 1, alpha=2.0, eta_inv=19.79, rc=1.2, P=30, M=2, seed=3,
                     placement="lattice")
    s.r, s.q = s.r[:40].copy(), s.q[:40]
    s.r[:, 2] = 2.2 + 1.9 * (np.arange(40) // 20)
    for k in range(20):
        for h in (0, 1):
            s.r[2 * k + h, :2] = [(0.66 + (k % 5) * 0.79 + h * 0.0) % 4.0, (k % 4) + 0.01]
        d = rng.normal(size=2)
        s.r[2 * k + 1, :2] += (1.34 + 0.15 * rng.random()) * d / np.linalg.norm(d)
    far = s.r.copy()
    near = s.r.copy()
    for k in range(20):
        d = far[2 * k + 1] - far[2 * k]
        u = 0.145 * d / np.linalg.norm(d)
        near[2 * k] += u
        near[2 * k + 1] -= u
    with srbe.from_slab(s, alpha_A=1.7) as c:
        c.set_skin(0.3)
        c.sample_k(5, 1)
        c.forces()
        c.set_positions(near, s.q)             # the same ions: the lists are kept while they hold
        F, Q, _ = c.forces()
    t = copy.copy(s)
    t.r = near
    with srbe.from_slab(t, alpha_A=1.7) as c:
        c.sample_k(5, 1)
        F2, Q2, _ = c.forces()
    # the same pairs in another order: sums of a few hundred FP64 terms
    assert np.abs(F - F2).max() <= 1e-11 * np.abs(F2).max()
    assert np.abs(Q - Q2).max() <= 1e-11 * np.abs(Q2).max()


def test_autotune_after_another_electrode():
    """The tuners save and restore the state of trial steps.  The iterate of an iterative solve that is no longer
    selected is no part of it: it has the size of the electrode it was used with."""
    a, b = (wl.make_slab("tune", (2.26, 2.02, 12.0), nx, ny, 39, 3, alpha=3.5, eta_inv=19.79, rc=1.2, P=40, M=2, seed=3,
                         with_md=True, placement="lattice") for nx, ny in ((6, 5), (10, 9)))
    with srbe.from_slab(a, precision=srbe.MIXED, alpha_A=1.7, md=True) as c:
        c.minimize(10)
        c.set_solver(srbe.PCG, tol=1e-8, maxit=2000, warm=srbe.WARM_PREVIOUS)
        c.step(2, 3)
        c.set_solver(srbe.DIRECT)
        c.set_electrode(b.R, b.side)
        r, v = c.get_positions(velocities=True)
        c.autotune_skin(2, 3, skins=(0.05, 0.1))
        c.autotune_tiles(2, 3, occ=(4, 8))
        r2, v2 = c.get_positions(velocities=True)
    assert np.array_equal(r, r2) and np.array_equal(v, v2)
