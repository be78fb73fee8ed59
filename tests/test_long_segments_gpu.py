"""Measured totals of segments of any length.  A thread adds its rows' terms in FP32 and
carries on with what rounding took from the sum, so the totals are as good as the terms
whatever the segments.

The lattice is a uniform one whose terms make that visible: unit vectors (to 2^-19)
with components of 19 bits, of which FP32 holds every multiple up to 32 exactly, and
of longer sums only some.  At a huge beta no move is accepted but one in 10^7 that
lies within rounding of the spin itself.  M is then the sum of the spins read back:
exact but for those, 2^-24 of a thread's sum each, so within 1e-12 of the total, where
plain sums of 57 to 512 rows are off by 1e-9 to 1e-7.
  XY spins, whose cosines have no short form, are compared with the same lattice on one
row per thread, whose four terms are equal and so add up exactly.  At the angle taken
here a sum of up to 32 rows is off by 6e-8 at most, one of 40 to 512 rows by 2.6e-7 and
more (computed with its FP32 cosine and those beside it), so the two agree within 1e-7."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sm():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1107_5463_gb300 import spinmc
    return spinmc


def magnetisation(sm, d, L, n, s0, opts):
    import torch
    lat = sm.Lattice(d, L, n=n, seed=4)
    for name, value in opts:
        lat.set_option(getattr(sm, "SL_OPT_" + name), value)
    sm.sl_set_spins(lat.h, s0)
    E, m = lat.sweep_series(1e30, 1, 8)
    m = float(m.cpu().numpy()[0])
    out = torch.empty(s0.shape, dtype=torch.float32, device="cuda")
    sm.sl_get_spins(lat.h, out)
    lat.close()
    return m, out


@pytest.mark.parametrize("d,L,opts", [
    (3, 256, []), (3, 256, [("KERNEL", 3)]), (2, 4096, []), (2, 1088, [("ROWS", 272)]),
    (2, 512, [("ROWS", 512)]), (2, 512, [("ROWS", 256), ("KERNEL", 3)]),
    (2, 512, [("ROWS", 512), ("FAST_MATH", 1)]), (3, 128, [("ROWS", 128)])])
def test_heisenberg(sm, d, L, opts):
    import torch
    N = L ** d
    v = torch.round(torch.tensor([0.36, -0.48, 0.8]) * 2.0 ** 19) * 2.0 ** -19
    v += 2.0 ** -19 * (1 - torch.remainder(v * 2.0 ** 19, 2))  # odd: no shorter form
    s0 = v.to(torch.float32).repeat(N, 1).cuda()
    m, s = magnetisation(sm, d, L, 3, s0, opts)
    want = float(s.double().sum(0).norm()) / N
    assert abs(m - want) <= 1e-12 * want


@pytest.mark.parametrize("L,opts", [(4096, []), (512, [("ROWS", 512)]),
                                    (512, [("ROWS", 512), ("FAST_MATH", 1)])])
def test_xy(sm, L, opts):
    import torch
    s0 = torch.full((L * L,), 2.0 * np.pi * 712.0 / 65536.0, dtype=torch.float32, device="cuda")
    got = magnetisation(sm, 2, L, 2, s0, opts)
    want = magnetisation(sm, 2, L, 2, s0, [o for o in opts if o[0] != "ROWS"] + [("ROWS", 1)])
    assert torch.equal(got[1], want[1])
    assert abs(got[0] - want[0]) <= 1e-7 * want[0]


@pytest.mark.parametrize("d,L,n", [(3, 64, 3), (3, 128, 3), (2, 1408, 2)])
def test_couplings_of_any_size(sm, d, L, n):
    """At beta = 0 every move is accepted whatever J, and a power of two in J goes through
    every product and sum unchanged, as long as none leaves FP32's range: E / J is the same
    number.  (Above 2^100 the energy's bias stays where it is; plain sums' 1e-6 then.)"""
    E = {}
    for k in (0, 100, -100, 112):
        lat = sm.Lattice(d, L, n=n, J=2.0 ** k, seed=4)
        E[k] = lat.sweep_series(0.0, 2, 8)[0].cpu().numpy() * 2.0 ** -k
        lat.close()
    np.testing.assert_array_equal(E[100], E[0])
    np.testing.assert_array_equal(E[-100], E[0])
    np.testing.assert_allclose(E[112], E[0], rtol=0, atol=1e-6 * 2 * d * L ** d)
