"""The flat XY kernels against the per-site kernel (SL_OPT_KERNEL 1), whose
arithmetic they repeat rounding for rounding: equal spins after every rule, at
even, odd and single-column rows.  (The per-site kernel is compared with the
FP64 oracle elsewhere.)  The energy and |m| series differ only by the order in
which FP32 partials are added: per site they hold at most a few units of 2^-23
of terms of size 2d, far below 1e-6."""
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


@pytest.mark.parametrize("d,L", [(2, 2), (2, 6), (2, 20), (2, 250), (2, 300), (3, 2), (3, 4),
                                 (3, 10), (3, 24), (3, 64), (3, 70)])
@pytest.mark.parametrize("rule,fast,J", [("metropolis", 0, 1.0), ("metropolis", 0, -0.8),
                                         ("metropolis", 1, 1.0), ("heatbath", 0, 1.0),
                                         ("heatbath", 1, -0.8)])
def test_flat_equals_per_site_kernel(sm, d, L, rule, fast, J):
    a = inputs.angles(d, L, 3).astype(np.float32)
    out = []
    for kernel in (0, 1):
        lat = sm.Lattice(d, L, n=2, J=J, seed=4, replica=2)
        lat.set_option(sm.SL_OPT_KERNEL, kernel)
        lat.set_option(sm.SL_OPT_FAST_MATH, fast)
        if rule == "heatbath":
            lat.set_update(sm.SL_UPDATE_HEATBATH)
        lat.set_spins(a)
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
        lat = sm.Lattice(d, L, n=2, J=J, seed=4)
        lat.set_option(sm.SL_OPT_KERNEL, kernel)
        lat.sweep(0.6, nsw, 55)
        out.append(lat.get_spins())
        lat.close()
    assert np.count_nonzero(out[0] != out[1]) == 0
