"""Batches whose packs are cut by sweeps and spread over the multiprocessors: the
same chains, bit for bit, as whole packs give (one sample per block), from run to
run and for runs of any length, with the state read back in between."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sm():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1107_5463_gb300 import spinmc
    return spinmc


@pytest.mark.parametrize("d,samples,sides,temps", [(3, 512, (8, 12, 16, 24, 32), 32),
                                                   (3, 512, (8, 12, 16, 24, 32), 8),
                                                   (3, 203, (4, 20), 5),
                                                   (2, 512, (4, 12, 32), 32)])
def test_pieces_give_the_chains_of_whole_packs(sm, d, samples, sides, temps):
    L = [sides[s % len(sides)] for s in range(samples)]
    betas = np.geomspace(0.5, 3.0, temps)
    b = sm.Batch(d, L, temps, betas, seed=11)
    w = sm.Batch(d, L, temps, betas, seed=11)
    w.set_option(sm.SL_BOPT_PACK, 1)
    for n in (4, 1, 7, 4, 13):
        E = [np.asarray(x.run(n, 5, series=True).cpu()) for x in (b, w)]
        np.testing.assert_array_equal(E[0], E[1])
        for s in (0, 3, samples // 2, samples - 1):
            for slot in (0, temps - 1):
                got, ref = b.get(s, slot), w.get(s, slot)
                np.testing.assert_array_equal(got[0], ref[0])
                assert got[1] == ref[1]
    b.close()
    w.close()


def test_batches_of_different_packs_take_turns(sm):
    """The kernel's shared-memory limit serves every batch of the process, whichever
    was set up last."""
    betas = np.geomspace(0.5, 3.0, 4)
    a, b = (sm.Batch(2, [32] * 8, 4, betas, seed=2) for _ in range(2))
    a.set_option(sm.SL_BOPT_PACK, 4)
    b.set_option(sm.SL_BOPT_PACK, 1)
    E = [np.asarray(x.run(3, 5, series=True).cpu()) for x in (a, b, a, b)]
    np.testing.assert_array_equal(E[0], E[1])
    np.testing.assert_array_equal(E[2], E[3])
    a.close()
    b.close()
