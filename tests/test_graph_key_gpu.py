"""Captured runs of sweeps are replayed only while everything that shapes their
launches is the same: a lattice whose options change between calls at one beta
and seed runs the chain of a lattice that captures nothing, bit for bit.  The
pairs of settings are those whose values meet in one word when they are packed
side by side with too few bits (rows 256 and the update rule, a period of 2^24
and fast math)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sm():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1107_5463_gb300 import spinmc
    return spinmc


def run(sm, L, n, settings, graph):
    lat = sm.Lattice(2, L, n=n, seed=4)
    lat.set_option(sm.SL_OPT_GRAPH, graph)
    for opts in settings:
        for name, value in opts:
            lat.set_option(getattr(sm, "SL_OPT_" + name), value)
        for _ in range(3):
            lat.sweep(0.7, 4, 9)
    got = lat.get_spins()
    lat.close()
    return got


@pytest.mark.parametrize("L,n,settings", [
    (512, 2, [[("UPDATE", 0)], [("ROWS", 256), ("UPDATE", 1)]]),
    (512, 2, [[("ROWS", 256), ("UPDATE", 0)], [("ROWS", 0), ("UPDATE", 1)]]),
    (512, 3, [[("ROWS", 256), ("UPDATE", 1)], [("ROWS", 0), ("UPDATE", 0)]]),
    (128, 3, [[("FAST_MATH", 1), ("RENORM_EVERY", 0)],
              [("FAST_MATH", 0), ("RENORM_EVERY", 1 << 24)]]),
])
def test_changed_options_take_effect(sm, L, n, settings):
    np.testing.assert_array_equal(run(sm, L, n, settings, 1), run(sm, L, n, settings, 0))
