"""GPU checks of the natural-order copies (sl_get_spins / sl_set_spins): the
chunk sizes of every row length, and host, device and unaligned device arrays,
against a plain numpy reading of the start configuration set by hand."""
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


# n, d, L, bits: W = L/2 a multiple of 8, of 4 only, odd, and one
CASES = [(1, 2, 64, 0), (1, 2, 40, 0), (1, 2, 6, 0), (1, 2, 2, 0), (1, 3, 16, 0), (1, 3, 24, 0),
         (1, 3, 10, 0), (1, 2, 128, 1), (1, 3, 64, 1), (2, 2, 22, 0), (2, 3, 18, 0),
         (3, 2, 34, 0), (3, 3, 20, 0), (3, 2, 2, 0)]


@pytest.mark.parametrize("n,d,L,bits", CASES)
def test_natural_order_copies(sm, n, d, L, bits):
    import torch
    if n == 1:
        a = inputs.ising_spins(d, L, 31)
    elif n == 2:
        a = inputs.angles(d, L, 31).astype(np.float32)
    else:
        a = inputs.unit_vectors(d, L, 31).astype(np.float32)
    tol = 1e-6 if n == 2 else 0.0  # angles pass through turns in FP32
    size = a.size
    dev = torch.zeros(size + 1, dtype=torch.from_numpy(a).dtype, device="cuda")
    flat = torch.from_numpy(a.reshape(-1)).cuda()
    for src in ("host", "device", "unaligned"):
        lat = sm.Lattice(d, L, n=n, seed=1, storage=sm.SL_STORE_BITS if bits else None)
        if src == "host":
            sm.sl_set_spins(lat.h, a)
        else:
            view = dev[1:] if src == "unaligned" else dev[:size]
            view.copy_(flat)
            torch.cuda.synchronize()
            sm.sl_set_spins(lat.h, view)
        np.testing.assert_allclose(lat.get_spins(), a, rtol=0, atol=tol)
        for off in (0, 1):
            out = torch.full((size + 2,), 9, dtype=dev.dtype, device="cuda")
            torch.cuda.synchronize()
            sm.sl_get_spins(lat.h, out[off:])
            got = out.cpu().numpy()
            np.testing.assert_allclose(got[off:off + size].reshape(a.shape), a, rtol=0, atol=tol)
            assert (got[off + size:] == 9).all() and (got[:off] == 9).all()
        E, M = lat.measure()
        lat.close()
        ref = sm.Lattice(d, L, n=n, seed=2, storage=sm.SL_STORE_BITS if bits else None)
        ref.set_spins(a)
        assert ref.measure()[0] == E
        ref.close()
