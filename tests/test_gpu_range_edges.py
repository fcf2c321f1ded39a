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


@pytest.mark.parametrize("p", [1.0, 2.4, 2.6, 2.9, 3.3])
def test_fp32_storage_observables_of_large_traces(cl, p):
    """The six plaquettes at one site are h = diag(p, p, p^-2): real traces of 3 to 6.7, whose sum passes 32 at
    p = 2.65 (at its neighbours, where h^-1 stands, earlier).  Entries of P and P^-1 reach p^2 = 11 and carry ~10 roundings of 6e-8 each: 1e-5 per trace, on 6 of
    the 6 V plaquettes and the ~30 that share a link with them."""
    L, beta = (3, 4, 3, 5), 6.0
    V = I.volume(L)
    x = I.coords(L)
    U = np.zeros((V, 4, 3, 3), np.complex64)
    U[:] = np.eye(3)
    base = np.array([1, 2, 0, 3])
    for mu in range(4):
        for nu in range(mu + 1, 4):
            y = base.copy()
            y[mu] = (y[mu] + 1) % L[mu]
            s = int(np.flatnonzero((x == y).all(1))[0])
            U[s, nu] = np.diag([p, p, p ** -2])
    U = U.astype(np.complex128)
    ref = O.observables(L, U, beta, 0.0)
    with cl.Lattice(L, beta=beta, prec=cl.CL_FP32_STORAGE) as lat:
        lat.set_links(U)
        obs = lat.observables()
    assert abs(obs["plaq_re"] - ref["plaq_re"]) <= 36 * 1e-5 / (18.0 * V)
    assert abs(obs["sw_re"] - ref["sw_re"]) <= beta / 6.0 * 36 * 2e-5


@pytest.mark.parametrize("prec,tol", [("CL_FP64", 1e-12), ("CL_DF64", 1e-12), ("CL_FP32_STORAGE", 1e-5)])
@pytest.mark.parametrize("h", [0.05, 0.12, 0.5, 0.8, 0.82, 0.84, 0.846, 0.86])
def test_cooling_exponents_whose_square_passes_two(cl, prec, tol, h):
    """One link B with B^2 = a + b J (J all ones): at its two ends H has a zero diagonal and +-h off it, so that the
    diagonal of H^2, 2 h^2, is in range up to h = 0.8478 while half its trace, 3 h^2, passes 2 at h = 0.8165.
    The result is three matrices of size up to e^(2 h); 1e-12 (1e-5) of it is hundreds of its roundings."""
    L, eps = (3, 4, 3, 5), 1.92  # a strength just below a power of two, so that f = H / eps is in range as well
    b = h / (4 * eps)
    a = min(r.real for r in np.roots([1.0, 3 * b, 0.0, -1.0]) if abs(r.imag) < 1e-12 and r.real > 0)
    w, v = np.linalg.eigh(a * np.eye(3) + b * np.ones((3, 3)))
    U = np.zeros((I.volume(L), 4, 3, 3), complex)
    U[:] = np.eye(3)
    U[37, 2] = (v * np.sqrt(w)) @ v.T
    kw = dict(eps=eps, alpha=1.0, forced_sweeps=1)
    if prec == "CL_FP32_STORAGE":
        U = U.astype(np.complex64).astype(complex)
    ref, _ = O.cool(L, U, O.cool_params(mode=O.D0, **kw))
    with cl.Lattice(L, prec=getattr(cl, prec)) as lat:
        lat.set_links(U)
        lat.cool(cl.make_cool(mode=cl.CL_D0, **kw))
        got = lat.links()
    assert np.abs(got - ref).max() <= tol * np.abs(ref).max()


@pytest.mark.parametrize("prec,tol", [("CL_FP64", 1e-14), ("CL_DF64", 1e-13), ("CL_FP32_STORAGE", 1e-6)])
@pytest.mark.parametrize("a", [0.0, 0.1, 0.5, 0.58, 0.6])
def test_norm_of_small_links(cl, prec, tol, a):
    """Links a U, off determinant one as a caller's may be: (1/3) Tr U U^+ = a^2.  A sum of V positive numbers."""
    L = (3, 4, 3, 5)
    U = a * I.su3_lattice(L, 4)
    if prec == "CL_FP32_STORAGE":
        U = U.astype(np.complex64).astype(complex)
    un = np.sum(np.abs(U) ** 2) / (12.0 * I.volume(L))
    with cl.Lattice(L, prec=getattr(cl, prec)) as lat:
        lat.set_links(U)
        obs = lat.observables()
    assert abs(obs["un"] - un) <= tol * max(un, 1.0)
    assert abs(obs["max_det_dev"] - np.abs(np.linalg.det(U) - 1.0).max()) <= max(tol, 1e-13)


@pytest.mark.parametrize("beta,theta", [(6.0, 1.0), (11.9, 0.0), (12.0, 0.0), (12.5, 2.0), (23.9, 0.0), (24.5, 0.0), (48.5, 0.0),
                                        (100.0, 1.0)])
@pytest.mark.parametrize("eps", [0.0027, 0.0056, 0.0057, 0.0112, 0.0113, 0.012, 0.0145, 0.05])
def test_update_on_both_sides_of_the_drift_constant(cl, beta, theta, eps):
    """The drift's constant 8 eps 2^cexp on both sides of the fixed-point bound, with the noise's inside and outside.
    The update is three products of matrices of size max |U| exp(|A|): 1e-12 of the result."""
    L = (4, 3, 2, 5)
    U = I.su3_lattice(L, 12)
    ref = O.cl_step(L, U, beta, theta, eps, 99, 4)
    with cl.Lattice(L, beta=beta, theta=theta, seed=99) as lat:
        lat.set_links(U)
        cl.cl_set_step(lat.h, 4)
        lat.step(eps)
        got = lat.links()
    assert np.abs(got - ref).max() <= 1e-12 * np.abs(ref).max()
