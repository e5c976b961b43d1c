"""srbe_step one step at a time, in runs and in both mixed: bitwise the trajectory of the ordinary launches, and a
single step is one graph with both its half kicks (as many kernels as the ordinary step and the one that stages the
mode list), nothing launched beside it."""
import numpy as np
import pytest

from paper_2509_24742_gb300 import srbe, workloads as wl

pytestmark = pytest.mark.gpu


def slab():
    return wl.make_slab("md_small", (2.0, 2.0, 12.0), 8, 8, 60, 3, alpha=3.5, eta_inv=19.79, rc=1.2, P=50, M=2, seed=21,
                        ax=0.25, ay=0.25, with_md=True)


@pytest.mark.parametrize("precision", [srbe.FP64, srbe.MIXED])
@pytest.mark.parametrize("device_sampler", [False, True])
@pytest.mark.parametrize("calls", [[1] * 12, [12], [5, 1, 1, 1, 4], [1, 1, 3, 1, 1, 1, 1, 2, 1]])
def test_single_steps_and_runs_give_the_same_trajectory(precision, device_sampler, calls):
    out = []
    for graphs in (False, True):
        with srbe.from_slab(slab(), precision=precision, alpha_A=1.7, md=True) as ctx:
            if device_sampler:
                ctx.set_sampler(srbe.EXACT)
                ctx.set_device_sampler(True)
            ctx.set_graphs(graphs)
            ctx.set_thermostat(5.0, 400.0, 5)
            seen = []
            for n in (calls if graphs else [1] * 12):
                ctx.step(n, 91)
                seen.append(ctx.get_positions(velocities=True))
        out.append((seen, np.cumsum(calls if graphs else [1] * 12)))
    ref = out[0][0]
    for (r, v), k in zip(*out[1]):
        assert np.array_equal(r, ref[k - 1][0]) and np.array_equal(v, ref[k - 1][1])


def test_a_single_step_is_one_graph():
    with srbe.from_slab(slab(), precision=srbe.MIXED, alpha_A=1.7, md=True) as ctx:
        ctx.step(1, 3)                     # captures
        ctx.set_graphs(False)
        ctx.step(1, 3)
        k0 = ctx.counters()[0]
        ctx.step(1, 3)
        ordinary = ctx.counters()[0] - k0
        ctx.set_graphs(True)
        ctx.step(1, 3)
        k0 = ctx.counters()[0]
        ctx.step(1, 3)
        assert ctx.graph_state() == (1, ordinary + 1)
        assert ctx.counters()[0] - k0 == ordinary + 1
