"""Calls of several sweeps replay graphs of 2^i sweeps, which are kept from call to
call and take new arguments when beta, the seed or an option changes; whatever calls
came before, a call gives the chain and the series of plain launches, bit for bit (the
finishing kernels add the same partials in the same order).  To give the graphs of a
call new arguments takes less time than its plain launches do, on a lattice whose
sweeps are short."""
import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sm():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1107_5463_gb300 import spinmc
    return spinmc


CALLS = [(5, 1), (20, 1), (20, 1), (5, 1), (100, 1), (63, 1), (200, 1), (1, 1), (2, 2), (3, 2),
         (16, 2), (16, 2), (97, 3), (31, 3), (31, 3), (31, 3), (32, 4), (64, 4)]


@pytest.mark.parametrize("d,L,n,storage,rule", [(2, 256, 1, "SL_STORE_BITS", 0),
                                                (2, 8192, 1, None, 0), (3, 10, 1, None, 2),
                                                (2, 128, 2, None, 0), (2, 128, 2, None, 1),
                                                (3, 10, 2, None, 0), (2, 64, 3, None, 0),
                                                (3, 10, 3, None, 0), (3, 10, 3, None, 1)])
def test_every_call_gives_the_chain_of_plain_launches(sm, d, L, n, storage, rule):
    calls = CALLS if L < 1000 else CALLS[:6]
    out = []
    for graph in (0, 1):
        lat = sm.Lattice(d, L, n=n, seed=4, storage=getattr(sm, storage) if storage else None)
        lat.set_option(sm.SL_OPT_GRAPH, graph)
        lat.set_update(rule)
        series = []
        for k, seed in calls:
            E, m = lat.sweep_series(0.5, k, seed)
            series += [E.cpu().numpy(), m.cpu().numpy()]
        out.append((np.concatenate(series), lat.get_spins()))
        assert lat.state()[1] == sum(k for k, _ in calls)
        lat.close()
    np.testing.assert_array_equal(out[0][0], out[1][0])
    np.testing.assert_array_equal(out[0][1], out[1][1])


def test_a_new_seed_does_not_cost_new_graphs(sm):
    import torch
    lat = sm.Lattice(2, 1024, seed=4, storage=sm.SL_STORE_BITS)
    took = {}
    for graph in (0, 1):
        lat.set_option(sm.SL_OPT_GRAPH, graph)
        lat.sweep(0.44, 63, 1)
        t = []
        for seed in range(15):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            lat.sweep(0.44, 63, 100 + seed)
            torch.cuda.synchronize()
            t.append(time.perf_counter() - t0)
        took[graph] = np.median(t)
    lat.close()
    # (789 us of plain launches, 399, and 1056 with graphs made anew in the call)
    assert took[1] < 1.15 * took[0]
