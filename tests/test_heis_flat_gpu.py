"""Heisenberg sweeps on rows of any length against the per-site kernel: the same
arithmetic, rounding for rounding, so identical spins; their FP64 totals gather
FP32 terms of other sites, which err by 2^-24 of the sums of a thread (at most a few
hundred sites, |E| / N <= 3), so both agree within 1e-6 per site."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sm():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1107_5463_gb300 import spinmc
    return spinmc


def start(N):
    v = np.random.default_rng(N).normal(size=(N, 3)) + np.array([0, 0, 1.5])
    return (v / np.linalg.norm(v, axis=1, keepdims=True)).astype(np.float32)


@pytest.mark.parametrize("d,L", [(2, 2), (2, 6), (2, 20), (2, 250), (2, 514), (3, 2), (3, 4),
                                 (3, 10), (3, 24), (3, 62), (3, 70)])
@pytest.mark.parametrize("rule,fast,J", [("metropolis", 0, 1.0), ("metropolis", 0, -0.8),
                                         ("metropolis", 1, 1.0), ("heatbath", 0, 1.0),
                                         ("heatbath", 1, -0.8)])
def test_flat_equals_per_site_kernel(sm, d, L, rule, fast, J):
    s0 = start(L ** d)
    out = []
    for kernel in (0, 1):
        lat = sm.Lattice(d, L, n=3, J=J, seed=4, replica=2)
        lat.set_option(sm.SL_OPT_KERNEL, kernel)
        lat.set_option(sm.SL_OPT_FAST_MATH, fast)
        lat.set_option(sm.SL_OPT_RENORM_EVERY, 3)
        if rule == "heatbath":
            lat.set_update(sm.SL_UPDATE_HEATBATH)
        lat.set_spins(s0)
        E, m = lat.sweep_series(0.9, 6, 55)
        out.append((lat.get_spins(), E.cpu().numpy() / L ** d, m.cpu().numpy()))
        lat.close()
    np.testing.assert_array_equal(out[0][0], out[1][0])
    np.testing.assert_allclose(out[0][1], out[1][1], rtol=0, atol=1e-6)
    np.testing.assert_allclose(out[0][2], out[1][2], rtol=0, atol=1e-6)


@pytest.mark.parametrize("d,L,nsw", [(3, 150, 24), (2, 2002, 24)])
@pytest.mark.parametrize("J", [1.0, -0.8])
def test_no_decision_of_a_long_run_differs(sm, d, L, nsw, J):
    """Eighty million decisions: one rounding sequence apart would flip several."""
    out = []
    for kernel in (0, 1):
        lat = sm.Lattice(d, L, n=3, J=J, seed=4)
        lat.set_option(sm.SL_OPT_KERNEL, kernel)
        lat.sweep(0.6, nsw, 55)
        out.append(lat.get_spins())
        lat.close()
    assert np.count_nonzero(out[0] != out[1]) == 0
