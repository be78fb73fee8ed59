"""A call's energy and |m| series starts with its own first sweep, whichever sweep
the device has reached: after replays of a captured call, which the host does not
count, the values of the next n sweeps still fill the n places given and no others
(here the places after them are the test's own and stay as they were)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sm():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1107_5463_gb300 import spinmc
    return spinmc


@pytest.mark.parametrize("d,L,n,rule", [(2, 64, 1, 0), (2, 4096, 1, 0), (2, 64, 1, 2),
                                        (2, 256, 2, 0), (3, 30, 2, 0), (3, 32, 3, 0)])
def test_series_after_replays(sm, d, L, n, rule):
    import torch
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        ref = sm.Lattice(d, L, n=n, seed=5)
        ref.set_update(rule)
        E, m = ref.sweep_series(0.4, 8, 7)
        want = E.cpu().numpy()[4:], m.cpu().numpy()[4:]
        ref.close()
        lat = sm.Lattice(d, L, n=n, seed=5)
        lat.set_update(rule)
        lat.sweep(0.4, 1, 7)
        st.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st, capture_error_mode="thread_local"):
            lat.sweep(0.4, 1, 7)
        for _ in range(3):
            g.replay()
        out = torch.full((2, 64), -5.0, dtype=torch.float64, device="cuda")
        sm.sl_sweep_series(lat.h, 0.4, 4, 7, out[0], out[1])
        st.synchronize()
        got = out.cpu().numpy()
        lat.close()
    np.testing.assert_array_equal(got[0, :4], want[0])
    np.testing.assert_array_equal(got[1, :4], want[1])
    assert (got[:, 4:] == -5.0).all()
