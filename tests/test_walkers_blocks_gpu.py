"""Walkers against the oracle where a block holds several warps: a last block with
idle warps, blocks in two turns and, beyond, single warps; warps whose walkers have
all passed the final stage stand beside others that go on."""
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


# 152 multiprocessors: 189 warps are blocks of 2, the last half idle; 1275 of windows
# that fit 8 to a block are blocks of 5 in two turns; 2575 are single
@pytest.mark.parametrize("L,width,wpw,windows,final", [(16, 4, 96, 63, 0), (16, 15, 128, 16, 1),
                                                       (64, 4, 128, 512, 20),
                                                       (32, 40, 1632, 25, 20),
                                                       (32, 40, 3296, 25, 20)])
def test_blocks_of_walkers_match_oracle(sm, L, width, wpw, windows, final):
    N = L * L
    klo = np.linspace(0, N - width, windows).astype(np.int32)
    khi = klo + width
    w = sm.Walkers(L, klo, khi, wpw, seed=3)
    pick = [0, wpw + 33, w.nwalk // 2 + 5, w.nwalk - 33, w.nwalk - 1]
    refs = {j: oracle.Walker(L, int(klo[j // wpw]), int(khi[j // wpw]), 3, j) for j in pick}
    sweeps = 30 if final < 2 else 2
    w.wl(sweeps, final_stage=final, flat_percent=40, seed=5)
    S, H, lev, st, vis = w.read()
    for j, r in refs.items():
        assert r.wl(sweeps, final, 40, tie_tol=1e-12, seed=5) == 0
        np.testing.assert_array_equal(w.spins(j), r.s)
        np.testing.assert_array_equal(S[j, :r.K], r.S)
        np.testing.assert_array_equal(H[j, :r.K], r.H)
        assert (lev[j], st[j], int(vis[j])) == (r.level, r.stage, r.visited)
    w.close()
