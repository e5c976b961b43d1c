"""The neighbour rebuild where its paths change: cells of more than 32 ions (ranked through memory
instead of shuffles), runs of fewer and of more than 64 candidates, a box of one cell per dimension
with several images, and lists that overflow their capacity.  The mixed form's forces come from the
lists, the FP64 oracle's from brute sums over all images; their difference is FP32 rounding: per pair
a relative 1e-6 of its force (a few roundings and the 1.5e-7 erfc approximation), so 1e-5 of the
forces' norm leaves a factor of ten.  A missing or doubled pair would change it by more than 1e-3.
The dense region is compared in FP64 only: its separations (0.03 nm at z = 4 nm) lose 1e-5 to the
rounding of FP32 positions alone, whatever the lists hold."""
import numpy as np
import pytest

from paper_2509_24742_gb300 import srbe, workloads as wl

pytestmark = pytest.mark.gpu


def slab(n_pairs, box, rc, seed):
    return wl.make_slab("lists", box, 8, 8, n_pairs, 1, alpha=2.5, eta_inv=19.79, rc=rc, P=40, M=2, seed=seed,
                        placement="lattice")


@pytest.mark.parametrize("n_pairs,box,rc,clustered", [
    (3, (2.0, 2.0, 12.0), 1.2, False),        # a handful of ions: nearly every run is empty
    (400, (2.0, 2.2, 12.0), 1.2, False),      # few ions per run, both lateral images
    (900, (2.0, 2.0, 14.0), 2.2, False),      # cells of 30 to 60 ions, several images per axis
    (300, (2.0, 2.0, 12.0), 1.2, True),       # one dense region: long runs and overflowing lists
])
def test_forces_from_the_lists_match_oracle(orc, n_pairs, box, rc, clustered):
    s = slab(n_pairs, box, rc, 5)
    if clustered:
        rng = np.random.default_rng(3)
        s.r = np.c_[rng.uniform(0.2, 0.8, s.n_ion), rng.uniform(0.2, 0.8, s.n_ion), rng.uniform(3.4, 4.2, s.n_ion)]
    samples = orc.sample_metropolis(s.box, s.alpha, s.M, s.P, 11, 0)
    ref = orc.System(s, alpha_A=1.7)
    m, c = ref.modes(samples)
    ev = ref.evaluate(m, c, with_lj=False)
    for precision, bound in ((srbe.FP64, 1e-10), (srbe.MIXED, 1e-5))[:1 if clustered else 2]:
        with srbe.from_slab(s, precision=precision, alpha_A=1.7) as ctx:
            ctx.set_k(samples)
            F, Q, _ = ctx.forces()
        assert np.linalg.norm(F - ev["F"]) < bound * np.linalg.norm(ev["F"])
        assert np.linalg.norm(Q - ev["Q"]) < bound * np.linalg.norm(ev["Q"])
