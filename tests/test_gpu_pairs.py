"""The FP64 form's fixed-point pair sums where they change path: rc just below and at a power of two
(the coordinates' period doubles), wide and narrow Gaussians, boxes shorter than the cutoff (several
images), LJ and bonds, negative z, and pairs closer than the radial tables reach (R1 / 64).

Bound.  A force is a sum of up to a few thousand FP64 terms, each within a few units of 1.1e-16 of
its own size; terms of one sign of the size of the largest would give 1e-13 of it, so 1e-11 of the
ion's own force plus the rms force leaves a factor of 100."""
import numpy as np
import pytest

from paper_2509_24742_gb300 import srbe, workloads as wl

pytestmark = pytest.mark.gpu


def check(orc, s, md):
    samples = orc.sample_metropolis(s.box, s.alpha, s.M, s.P, 13, 0)
    ref = orc.System(s, alpha_A=1.9)
    m, c = ref.modes(samples)
    ev = ref.evaluate(m, c, with_lj=md)
    with srbe.from_slab(s, alpha_A=1.9, md=md) as ctx:
        ctx.set_k(samples)
        F, Q, _ = ctx.forces()
        F_plain = ctx.forces(energy=True)[0]
    # the pass with energies takes the plain pair functions on the same charges
    assert worst(F, F_plain) < 1e-11
    if s.eta < 0.1:          # wider Gaussians overlap: A's condition (6e10 at 1/3 nm) swamps the charges
        assert worst(F, ev["F"]) < 1e-11
        assert np.linalg.norm(Q - ev["Q"]) < 1e-10 * np.linalg.norm(ev["Q"])


def worst(F, ref):
    rms = np.sqrt((ref ** 2).mean())
    return (np.abs(F - ref).max(1) / (np.abs(ref).max(1) + rms)).max()


@pytest.mark.parametrize("rc,alpha,eta_inv,box", [
    (0.98, 3.0, 19.79, (2.0, 2.2, 12.0)),     # R1 = 1
    (0.99, 3.0, 19.79, (2.0, 2.2, 12.0)),     # R1 = 2 from here
    (1.98, 2.0, 3.0, (2.0, 2.0, 12.0)),       # R1 = 2, wide Gaussians, several images
    (2.0, 1.5, 40.0, (2.01, 2.02, 12.0)),     # R1 = 4, narrow ones (L != rc: an image at rc is a tie)
])
@pytest.mark.parametrize("md", [False, True])
def test_pair_sums_match_oracle(orc, rc, alpha, eta_inv, box, md):
    s = wl.make_slab("pairs", box, 8, 8, 60, 3, alpha=alpha, eta_inv=eta_inv, rc=rc, P=30, M=2, seed=3, with_md=md)
    check(orc, s, md)


def test_close_pairs_and_negative_z_match_oracle(orc):
    s = wl.make_slab("close", (2.0, 2.0, 12.0), 8, 8, 40, 1, alpha=3.0, eta_inv=19.79, rc=1.2, P=30, M=2, seed=4)
    s.r[1] = s.r[0] + [0.011, -0.007, 0.009]           # below R1 / 64 = 0.031
    s.r[3] = s.r[2] + [0.0, 0.031, 0.002]              # next to it
    s.r[5] = s.R[7] + [0.004, 0.003, -0.008]           # next to a site, negative z
    s.r[6] = [1.9999, 0.0001, 4.0]
    s.r[7] = [0.0002, 1.9998, 4.01]                    # across both periodic edges
    check(orc, s, False)


@pytest.mark.parametrize("d", [1e-8, 2e-10, 1e-11])
def test_ion_all_but_on_a_site(orc, d):
    """An ion 1e-8 to 1e-11 nm above a site, where r^2 rounds to zero in the pair sums' units: it still raises that
    site's potential (by -q 2 (1 / eta - alpha) / sqrt(pi), -19 q).  That term is (erfc(alpha r) - erfc(r / eta)) / r,
    a difference of numbers next to one: a few 1.1e-16 / r of it are rounding, 1e-4 at 1e-11 nm, 5e-6 of the term.
    The charges answer in proportion, so 1e-4 leaves a factor of 20."""
    s = wl.make_slab("on", (2.0, 2.0, 12.0), 8, 8, 40, 1, alpha=3.0, eta_inv=19.79, rc=1.2, P=30, M=2, seed=4)
    site = int(np.flatnonzero(s.R[:, 2] == 0.0)[9])
    s.r[0] = s.R[site] + [0.0, 0.0, d]
    samples = orc.sample_metropolis(s.box, s.alpha, s.M, s.P, 13, 0)
    ref = orc.System(s, alpha_A=1.9)
    ev = ref.evaluate(*ref.modes(samples), with_lj=False)
    with srbe.from_slab(s, alpha_A=1.9) as ctx:
        ctx.set_k(samples)
        Q, _, _ = ctx.solve_charges()
    assert np.linalg.norm(Q - ev["Q"]) < 1e-4 * np.linalg.norm(ev["Q"])
