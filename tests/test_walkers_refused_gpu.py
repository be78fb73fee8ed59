"""A configuration that sl_walkers_set_spins refuses leaves the walker as it was: spins,
level and the run that follows are those of walkers that were never asked."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sm():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1107_5463_gb300 import spinmc
    return spinmc


@pytest.mark.parametrize("L,klo,width", [(8, 20, 7), (16, 100, 4), (16, 120, 15)])
def test_a_refused_configuration_changes_nothing(sm, L, klo, width):
    lo = np.array([klo, klo + width], np.int32)
    runs = []
    for refuse in (False, True):
        w = sm.Walkers(L, lo, lo + width, 32, seed=3)
        w.wl(2, final_stage=20, seed=5)
        if refuse:
            for walker in (0, 17, 40):
                with pytest.raises(sm.SpinMCError, match="outside its window"):
                    sm.sl_walkers_set_spins(w.h, walker, np.ones(L * L, np.int8))  # level 0
        before = [w.spins(j) for j in range(w.nwalk)] + list(w.read())
        # one that is accepted, from another walker of the window
        sm.sl_walkers_set_spins(w.h, 1, w.spins(2))
        w.wl(3, final_stage=20, seed=6)
        runs.append(before + [w.spins(j) for j in range(w.nwalk)] + list(w.read()))
        w.close()
    for a, b in zip(*runs):
        np.testing.assert_array_equal(a, b)
