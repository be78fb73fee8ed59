"""3D Swendsen-Wang updates on more than one 64 x 16 x 8 tile along x, against the
oracle bit for bit: L = 66 and 80 (a ragged second tile), 128 (two full ones), so that
clusters meet at the +x face of a tile and over the periodic boundary of another."""
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


@pytest.mark.parametrize("L,nsw", [(66, 5), (80, 5), (128, 3)])
@pytest.mark.parametrize("beta,J", [(inputs.BETA_3D_ISING, 1.0), (0.3, -0.9)])
def test_several_tiles_along_x(sm, L, nsw, beta, J):
    lat = sm.Lattice(3, L, n=1, J=J, seed=5)
    lat.set_update(sm.SL_UPDATE_SW)
    E, m = lat.sweep_series(beta, nsw, 55)
    got = lat.get_spins(), E.cpu().numpy(), m.cpu().numpy()
    lat.close()
    s = oracle.ising_init(3, L, 5)
    Er, mr = oracle.ising_sw_sweeps(3, L, s, beta, 55, 0, nsw, J=J)
    np.testing.assert_array_equal(got[0], s)
    np.testing.assert_array_equal(got[1], Er)
    np.testing.assert_array_equal(got[2], mr)
