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
