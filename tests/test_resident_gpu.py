"""GPU parity of the byte-Ising kernels that take one Philox group per thread:
lattices resident in shared memory (one block up to 2^14 sites, several
blocks with halo planes beyond) and the flat kernel for ragged rows, against
the oracle bit for bit, at row lengths W = L/2 that are multiples of 4, even
and odd, and planes whose entries leave the last Philox group short."""
import numpy as np
import pytest

import oracle
from paper_1107_5463_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sm():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1107_5463_gb300 import spinmc
    return spinmc


def check(sm, d, L, beta, nsw, J=1.0, Jb=None, heatbath=False, flat=False, calls=1):
    lat = sm.Lattice(d, L, J=J, J_bonds=Jb, seed=5, replica=3)
    if heatbath:
        lat.set_update(sm.SL_UPDATE_HEATBATH)
    if flat:
        lat.set_option(sm.SL_OPT_ROWS, 1)  # a streaming shape: not the resident kernel
    E, m = [], []
    for _ in range(calls):
        e, a = lat.sweep_series(beta, nsw, 77)
        E.append(e.cpu().numpy())
        m.append(a.cpu().numpy())
    s = oracle.ising_init(d, L, 5, 3)
    f = oracle.ising_heatbath_sweeps if heatbath else oracle.ising_sweeps
    Er, mr = f(d, L, s, beta, 77, 0, nsw * calls, J=J, Jb=Jb, replica=3)
    np.testing.assert_array_equal(np.concatenate(E), Er)
    np.testing.assert_array_equal(np.concatenate(m), mr)
    np.testing.assert_array_equal(lat.get_spins(), s)
    Em, M = lat.measure()
    assert Em == Er[-1] and abs(M[1] - mr[-1]) == 0.0
    assert lat.state()[1] == nsw * calls
    lat.close()


SIDES = [(2, 2), (2, 6), (2, 10), (2, 40), (2, 128), (2, 130), (2, 132), (2, 136), (2, 250),
         (2, 1000), (3, 2), (3, 6), (3, 20), (3, 24), (3, 26), (3, 28), (3, 32), (3, 50)]


@pytest.mark.parametrize("d,L", SIDES)
@pytest.mark.parametrize("J,heatbath", [(1.0, False), (-0.7, False), (1.0, True)])
def test_uniform_coupling(sm, d, L, J, heatbath):
    beta = inputs.BETA_C_2D_ISING if d == 2 else inputs.BETA_3D_ISING
    check(sm, d, L, beta, 4, J=J, heatbath=heatbath, calls=2)


@pytest.mark.parametrize("d,L", SIDES)
@pytest.mark.parametrize("heatbath", [False, True])
def test_pm_bonds(sm, d, L, heatbath):
    check(sm, d, L, 0.8, 4, Jb=inputs.ising_bonds(d, L, 9), heatbath=heatbath, calls=2)


@pytest.mark.parametrize("d,L", [(2, 2), (2, 6), (2, 24), (2, 250), (2, 1000), (3, 2), (3, 6),
                                 (3, 24), (3, 50)])
@pytest.mark.parametrize("J,heatbath", [(1.0, False), (-0.7, False), (1.0, True)])
def test_flat_kernel(sm, d, L, J, heatbath):
    check(sm, d, L, 0.4, 3, J=J, heatbath=heatbath, flat=True)


def test_more_sweeps_than_one_launch(sm):
    check(sm, 2, 16, inputs.BETA_C_2D_ISING, 1500)
    check(sm, 2, 136, inputs.BETA_C_2D_ISING, 1100)


def test_a_captured_call_replays(sm):
    import torch
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        lat = sm.Lattice(2, 136, seed=5)
        lat.sweep(0.4, 1, 7)
        st.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st, capture_error_mode="thread_local"):
            lat.sweep(0.4, 1, 7)
        for _ in range(3):
            g.replay()
        st.synchronize()
        lat.set_state(4)
        lat.sweep(0.4, 2, 7)
        s = oracle.ising_init(2, 136, 5, 0)
        oracle.ising_sweeps(2, 136, s, 0.4, 7, 0, 6)
        np.testing.assert_array_equal(lat.get_spins(), s)
        lat.close()
