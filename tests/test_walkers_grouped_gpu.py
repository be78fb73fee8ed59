"""Walkers against the oracle where the words of four attempts are fetched
together (sides at which most sweeps' site orders are clear of collisions, so
both paths run), in narrow windows (H worked out from the gain of ln g) and wide
ones (counted attempt by attempt)."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sm():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1107_5463_gb300 import spinmc
    return spinmc


# width 7: 8 levels; 15: 16 levels (the widest snapshot); 16 and 40: counted
@pytest.mark.parametrize("L,width,sweeps", [(16, 4, 12), (32, 7, 8), (32, 15, 6), (32, 16, 6),
                                            (64, 4, 5), (64, 40, 3), (128, 4, 2)])
@pytest.mark.parametrize("spins_smem", [0, 1])
def test_walkers_match_oracle(sm, L, width, sweeps, spins_smem):
    N = L * L
    klo = np.array([N // 4, N // 2 - width // 2], np.int32)
    khi = klo + width
    w = sm.Walkers(L, klo, khi, 32, seed=3)
    w.set_option(sm.SL_WOPT_SPINS_SMEM, spins_smem)
    pick = [0, 13, 31, 32, 50]
    refs = {j: oracle.Walker(L, int(klo[j // 32]), int(khi[j // 32]), 3, j) for j in pick}
    w.wl(sweeps, final_stage=3, flat_percent=70, seed=5)
    w.wl(2, final_stage=20, flat_percent=70, seed=6)
    S, H, lev, st, vis = w.read()
    for j, r in refs.items():
        assert r.wl(sweeps, 3, 70, tie_tol=1e-12, seed=5) == 0
        assert r.wl(2, 20, 70, tie_tol=1e-12, seed=6) == 0
        np.testing.assert_array_equal(w.spins(j), r.s)
        np.testing.assert_array_equal(S[j, :r.K], r.S)
        np.testing.assert_array_equal(H[j, :r.K], r.H)
        assert (lev[j], st[j], int(vis[j])) == (r.level, r.stage, r.visited)
    w.close()
