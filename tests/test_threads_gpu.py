"""Two host threads, each with its own handle on its own stream, sizes chosen so
that the threads launch the same kernels with different amounts of shared memory.
A thread's launches depend on nothing the other one does: every call succeeds, and
each chain is the one that the thread's handle runs alone, bit for bit."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sm():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1107_5463_gb300 import spinmc
    return spinmc


def together(sm, make, step, read, n):
    """The results of handles make(0) and make(1) after n steps each: alone, and side by side."""
    import torch
    out, failed = [{}, {}], []

    def work(k, side):
        try:
            st = torch.cuda.Stream()
            with torch.cuda.stream(st):
                h = make(k, st)
                for _ in range(n):
                    step(h)
                out[side][k] = read(h)
                h.close()
        except Exception as e:  # a failed call shows in the main thread
            failed.append(e)

    for k in range(2):
        work(k, 0)
    ts = [threading.Thread(target=work, args=(k, 1)) for k in range(2)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not failed, failed[0]
    return out


@pytest.mark.parametrize("d,sides", [(2, (16, 64)), (2, (128, 1024)), (3, (32, 96))])
def test_resident_lattices(sm, d, sides):
    out = together(sm, lambda k, st: sm.Lattice(d, sides[k], seed=4, stream=st),
                   lambda h: h.sweep(0.4, 1, 9), lambda h: h.get_spins(), 3000)
    for k in range(2):
        np.testing.assert_array_equal(out[0][k], out[1][k])


def test_walkers(sm):
    klo = [np.array([40, 60], np.int32), np.arange(40, 140, 4).astype(np.int32)]

    def make(k, st):
        return sm.Walkers(16, klo[k], klo[k] + 4, 256, seed=3, stream=st)

    out = together(sm, make, lambda h: h.wl(1, final_stage=20, seed=5), lambda h: h.read(), 1500)
    for k in range(2):
        for a, b in zip(out[0][k], out[1][k]):
            np.testing.assert_array_equal(a, b)
