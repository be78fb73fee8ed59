"""Calls of few sweeps on byte lattices that fit the chip's shared memory.  Loading a
large one, above all its couplings, takes longer than a sweep, so such calls run on the
streaming kernel; the choice by the length of the call changes no chain, and a call of
one sweep takes no longer than on the streaming kernel (15% is allowed: equal launches
back to back can differ by a step of 2 us a call; the load took 20 to 33%)."""
import time

import numpy as np
import pytest

from paper_1107_5463_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sm():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1107_5463_gb300 import spinmc
    return spinmc


def lattice(sm, d, L, kernel):
    lat = sm.Lattice(d, L, J_bonds=inputs.ising_bonds(d, L, 9), seed=5)
    lat.set_option(sm.SL_OPT_KERNEL, kernel)
    return lat


@pytest.mark.parametrize("d,L", [(2, 512), (2, 2048), (3, 64), (3, 96), (3, 128)])
def test_any_mix_of_lengths_gives_the_same_chain(sm, d, L):
    got = []
    for kernel in (0, 2):
        lat = lattice(sm, d, L, kernel)
        series = [lat.sweep_series(0.8, n, 7)[0].cpu().numpy()
                  for n in (1, 12, 1, 2, 3, 4, 6, 9, 1, 20)]
        got.append((np.concatenate(series), lat.get_spins()))
        lat.close()
    np.testing.assert_array_equal(got[0][0], got[1][0])
    np.testing.assert_array_equal(got[0][1], got[1][1])


@pytest.mark.parametrize("d,L", [(2, 2048), (3, 96), (3, 128)])
def test_single_sweeps_cost_no_more_than_streaming(sm, d, L):
    import torch
    lats = [lattice(sm, d, L, kernel) for kernel in (0, 2)]
    took = [[], []]
    for rep in range(12):
        for k in range(2):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            for _ in range(100):
                lats[k].sweep(0.8, 1, 7)
            torch.cuda.synchronize()
            if rep > 1:
                took[k].append(time.perf_counter() - t0)
    for lat in lats:
        lat.close()
    assert min(took[0]) < 1.15 * min(took[1])
