"""The streaming kernels of continuous spins on automatic segments, whose lengths do
not divide the rows of these sides, against one row per thread: which thread updates a
site changes no decision, so the spins are identical.

The totals add the same FP32 terms, one per row and thread, with what rounding takes
carried along (an error below 2^-44 of a thread's sum), so E and |m| agree within 1e-12
of the sum of the terms' sizes, N times 2d and N.  The XY heat-bath folds up to 32 rows
of plain FP32 sums, 128 terms below 4 in size and a few more, at 2^-24 of their sum at
most per addition: within 1e-5 per site for E and |m|, and about a hundredth of that as
the errors of a million sites' sums are of either sign."""
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


# XY pairs; single Heisenberg columns (W % 64 == 32), 2D and 3D; Heisenberg pairs
@pytest.mark.parametrize("rule", ["metropolis", "fast", "heatbath"])
@pytest.mark.parametrize("d,L,n", [(2, 1152, 2), (2, 1408, 2), (2, 1088, 3), (3, 64, 3),
                                   (3, 192, 3), (2, 1152, 3), (3, 128, 3)])
def test_uneven_segments(sm, d, L, n, rule):
    N = L ** d
    s0 = start(n, N)
    got = []
    for rows in (0, 1):
        lat = sm.Lattice(d, L, n=n, seed=4)
        lat.set_option(sm.SL_OPT_KERNEL, 2)  # refused on rows that do not stream
        if rows:
            lat.set_option(sm.SL_OPT_ROWS, rows)
        if rule == "heatbath":
            lat.set_update(sm.SL_UPDATE_HEATBATH)
        elif rule == "fast":
            lat.set_option(sm.SL_OPT_FAST_MATH, 1)
        lat.set_spins(s0)
        E, m = lat.sweep_series(1.12 if n == 2 else 1.5, 3, 8)
        got.append((lat.get_spins(), E.cpu().numpy() / N, m.cpu().numpy()))
        lat.close()
    tol = 1e-7 if (n, rule) == (2, "heatbath") else 1e-12
    np.testing.assert_array_equal(got[0][0], got[1][0])
    np.testing.assert_allclose(got[0][1], got[1][1], rtol=0, atol=2 * d * tol)
    np.testing.assert_allclose(got[0][2], got[1][2], rtol=0, atol=tol)


# heis_flat with every spin normalised at each sweep, and with none ever
@pytest.mark.parametrize("d,L", [(2, 6), (2, 62), (2, 250), (3, 10), (3, 62)])
@pytest.mark.parametrize("renorm", [0, 1])
def test_flat_heisenberg_and_renormalisation(sm, d, L, renorm):
    out = []
    for kernel in (0, 1):
        lat = sm.Lattice(d, L, n=3, seed=4)
        lat.set_option(sm.SL_OPT_KERNEL, kernel)
        lat.set_option(sm.SL_OPT_RENORM_EVERY, renorm)
        lat.set_spins(start(3, L ** d))
        lat.sweep(0.9, 5, 55)
        out.append(lat.get_spins())
        lat.close()
    np.testing.assert_array_equal(out[0], out[1])
