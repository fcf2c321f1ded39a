"""Sums at the edge of the 60-bit fixed-point range: each test puts one at or beyond the value where 64 bits
would wrap, with every operand inside its own bound, and compares with the oracle."""
import numpy as np
import pytest

import oracle as O
import lattice_inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cl():
    from paper_1311_1056_gb300 import cl as c
    return c


@pytest.mark.parametrize("prec", ["CL_FP64", "CL_DF64"])
@pytest.mark.parametrize("a", [1.0, 1.19])
def test_drift_of_large_trace(cl, prec, a):
    """One link diag(a, a, a^-2) exp(2 pi i / 3) among unit links: its six plaquettes add up to a drift close to a
    multiple of one, of trace 7.8 (a = 1) or 8.02 in the contributions' units, which the step has to remove.  K_max
    is a few tens of roundings of numbers of the drift's size, 1e-12 of it."""
    L, beta, eps, k_ref = (3, 4, 3, 5), 5.99, 0.01, 5.0
    U = np.zeros((I.volume(L), 4, 3, 3), complex)
    U[:] = np.eye(3)
    U[37, 2] = np.diag([a, a, a ** -2]) * np.exp(2j * np.pi / 3)
    ref, e, k = O.cl_step_adaptive(L, U, beta, 0.0, eps, k_ref, 7, 0)
    X = np.abs(O.drift(L, U, beta, 0.0)).max()
    with cl.Lattice(L, beta=beta, prec=getattr(cl, prec), seed=7) as lat:
        lat.set_links(U)
        lat.set_adaptive_step(k_ref)
        lat.step(eps)
        _, e_gpu, k_gpu = lat.langevin_time()
        err = np.abs(lat.links() - ref).max()
    assert abs(k_gpu - k) <= 1e-12 * X
    assert abs(e_gpu - e) <= 1e-12 * eps
    assert err <= 1e-12 * np.abs(ref).max()
