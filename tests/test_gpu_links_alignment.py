"""The link exchange with buffers aligned to 16 and only to 8 bytes: page-locked host memory (read and written
in place over the host link) and device memory, full and partial 32-site tiles.  A copy, so bit for bit."""
import ctypes

import numpy as np
import pytest

import lattice_inputs as LI
from paper_1311_1056_gb300 import cl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L", [(4, 4, 4, 4), (3, 5, 2, 1), (1, 1, 1, 1)])
@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("where", ["pinned", "device"])
def test_exchange_is_a_copy(L, offset, where):
    torch = pytest.importorskip("torch")
    V = LI.volume(L)
    U = LI.sl3c_lattice(L, 4, 0.1)
    n = V * 72
    kw = dict(pin_memory=True) if where == "pinned" else dict(device="cuda")
    a, b = (torch.zeros(n + 2, dtype=torch.float64, **kw) for _ in range(2))
    a[offset:offset + n] = torch.from_numpy(U.view(np.float64).reshape(-1).copy()).to(a.device)
    torch.cuda.synchronize()
    with cl.Lattice(L) as lat:
        pa, pb = a.data_ptr() + 8 * offset, b.data_ptr() + 8 * offset
        lib, dp = cl.load(), ctypes.POINTER(ctypes.c_double)
        if where == "pinned":
            assert lib.cl_set_links(lat.h, ctypes.cast(pa, dp)) == 0 and lib.cl_get_links(lat.h, ctypes.cast(pb, dp)) == 0
        else:
            cl.cl_set_links_device(lat.h, pa)
            cl.cl_get_links_device(lat.h, pb)
            lat.synchronize()
        assert np.array_equal(lat.links(), U)
    assert torch.equal(a, b)
