"""The FP64 form's fixed-point link algebra and its general path.

Fixed point holds numbers below 1.4375; links, plaquettes or contributions
beyond that are redone in FP64 by the threads that meet them.  Fields are taken
on both sides of that line and across it, with couplings that move the
contributions' scale, and compared with the oracle.

Tolerance: the drift is a sum of products of up to eight factors (links,
inverses, plaquettes, a dual field), a few hundred units of 2^-53 of max |X|
for links near SU(3); 1e-11 of max |X| leaves two decades for the cancellation
P - P^{-1} in fields of large links.  (Beyond |U| ~ 10 that cancellation alone
costs an FP64 evaluation more than this.)"""
import numpy as np
import pytest

import oracle as O
import lattice_inputs as I

pytestmark = pytest.mark.gpu

SHAPES = [(4, 4, 4, 4), (3, 5, 2, 4), (1, 4, 4, 2)]


@pytest.fixture(scope="module")
def cl():
    from paper_1311_1056_gb300 import cl as c
    return c


def field(L, spread, seed):
    """spread 0: SU(3), inside the bound; 0.1, 0.2: many sites inside; 0.4: most outside; "mixed": one wild site."""
    if spread == 0:
        return I.su3_lattice(L, seed)
    if spread == "mixed":
        U = I.su3_lattice(L, seed)
        U[I.volume(L) // 2] = I.sl3c_lattice((1, 1, 1, 1), seed + 1, 0.4)[0]
        return U
    return I.sl3c_lattice(L, seed, spread)


@pytest.mark.parametrize("L", SHAPES)
@pytest.mark.parametrize("spread", [0, 0.1, 0.2, 0.4, "mixed"])
@pytest.mark.parametrize("beta,theta", [(6.0, 1.0), (6.0, 0.0), (600.0, 40.0), (1e-3, 2.0), (0.0, 1.0 + 0.5j)])
def test_drift_inside_and_outside_the_fixed_point_range(cl, L, spread, beta, theta):
    U = field(L, spread, 11)
    ref = O.drift(L, U, beta, theta)
    with cl.Lattice(L, beta=beta, theta=theta) as lat:
        lat.set_links(U)
        X = lat.drift()
    assert np.abs(X - ref).max() <= 1e-11 * np.abs(ref).max()


@pytest.mark.parametrize("spread", [0, 0.1, 0.2, 0.4, "mixed"])
def test_observables_inside_and_outside_the_range(cl, spread):
    L = (3, 4, 2, 5)
    U = field(L, spread, 5)
    ref = O.observables(L, U, 6.0, 0.7)
    with cl.Lattice(L, beta=6.0, theta=0.7) as lat:
        lat.set_links(U)
        obs = lat.observables()
        q = lat.qdensity()
    scale = max(abs(ref["sw_re"]), 6.0 * 6 * I.volume(L))
    for k in ("plaq_re", "plaq_im", "un"):
        assert abs(obs[k] - ref[k]) <= 1e-12 * max(1.0, abs(ref[k])), k
    for k in ("q_re", "q_im", "sw_re", "sw_im"):
        assert abs(obs[k] - ref[k]) <= 1e-12 * scale, k
    assert abs(q.sum() - complex(obs["q_re"], obs["q_im"])) <= 1e-12 * max(1.0, np.abs(q).sum())


def test_non_finite_links_are_reported(cl):
    L = (4, 2, 3, 4)
    for bad in (np.nan, np.inf, -np.inf, 1e200):
        U = I.su3_lattice(L, 3)
        U[7, 2, 1, 1] = bad
        with cl.Lattice(L, beta=6.0, theta=1.0) as lat:
            lat.set_links(U)
            lat.step(0.01, 2)
            with pytest.raises(cl.CLError) as e:
                lat.observables()
            assert e.value.status == cl.CL_ERR_NONFINITE
