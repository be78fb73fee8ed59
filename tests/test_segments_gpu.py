"""Streaming kernels of continuous spins on segments of unequal length.

The automatic shape deals the rows out in segments of q and q + 1 rows.  Which
thread updates a site changes no decision, so the chain is that of one row per
thread: identical FP32 spins.  The FP64 totals gather FP32 partials of other
sites: a partial of up to 64 sites errs by at most 64 x 2d x 2^-24, so E agrees
within 1e-6 relative and |m| within 1e-7 (sizes where neither is near zero)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sm():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1107_5463_gb300 import spinmc
    return spinmc


def start(n, N):
    g = np.random.default_rng(N + n)
    if n == 2:
        return np.mod(g.normal(2.5, 0.7, N), 6.28).astype(np.float32)
    v = g.normal(size=(N, 3)) + np.array([0, 0, 1.5])
    return (v / np.linalg.norm(v, axis=1, keepdims=True)).astype(np.float32)


@pytest.mark.parametrize("rule", ["metropolis", "fast", "heatbath"])
@pytest.mark.parametrize("d,L,n", [(2, 1024, 2), (2, 1472, 2), (3, 96, 2),
                                   (2, 1024, 3), (2, 1120, 3), (3, 96, 3), (3, 128, 3)])
def test_uneven_segments_give_the_same_chain(sm, d, L, n, rule):
    beta = 1.12 if n == 2 else 1.5
    s0 = start(n, L ** d)
    got = []
    for rows in (0, 1):
        lat = sm.Lattice(d, L, n=n, seed=4)
        if rows:
            lat.set_option(sm.SL_OPT_ROWS, rows)
        if rule == "heatbath":
            lat.set_update(sm.SL_UPDATE_HEATBATH)
        elif rule == "fast":
            lat.set_option(sm.SL_OPT_FAST_MATH, 1)
        lat.set_spins(s0)
        E, m = lat.sweep_series(beta, 3, 8)
        got.append((lat.get_spins(), E.cpu().numpy(), m.cpu().numpy()))
        lat.close()
    np.testing.assert_array_equal(got[0][0], got[1][0])
    np.testing.assert_allclose(got[0][1], got[1][1], rtol=1e-6)
    np.testing.assert_allclose(got[0][2], got[1][2], rtol=0, atol=1e-7)
