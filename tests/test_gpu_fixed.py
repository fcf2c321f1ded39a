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


@pytest.mark.parametrize("L", [(4, 4, 4, 4), (3, 5, 2, 4), (1, 4, 4, 2), (7, 3, 2, 5)])
@pytest.mark.parametrize("spread", [0, 0.05, 0.2, 0.4, "mixed"])
@pytest.mark.parametrize("mode", ["D0", "D1", "D2_MEANABS", "D2_RMS"])
def test_cooling_inside_and_outside_the_range(cl, L, spread, mode):
    """Two sweeps of a step small enough that no field blows up: a sweep multiplies each link by two
    matrices near 1, a few tens of roundings of the link's size; 1e-12 of max |U| is a hundred times that.
    (D_2 divides by <|f|>, at rounding level for SU(3) links: there the guard stops it on both sides.)"""
    U = field(L, spread, 21)
    kw = dict(eps=1e-3, alpha=1.0, forced_sweeps=2, d_guard=1e-9)
    ref, rep = O.cool(L, U, O.cool_params(mode=getattr(O, mode), **kw))
    with cl.Lattice(L) as lat:
        lat.set_links(U)
        got = lat.cool(cl.make_cool(mode=getattr(cl, "CL_" + mode), **kw))
        Ug = lat.links()
        f = lat.cool_gradient()
    assert got["sweeps"] == rep["sweeps"]
    assert np.abs(Ug - ref).max() <= 1e-12 * np.abs(ref).max()
    fr = O.cool_gradient(L, ref)
    assert np.abs(f - fr).max() <= 1e-11 * np.abs(ref).max() ** 2
    for k in ("un_before", "un_after"):
        assert abs(got[k] - rep[k]) <= 1e-12 * rep[k], k


def test_cooling_with_a_large_exponent(cl):
    """eps alpha |f| of order one: Omega leaves the fixed-point range and is formed in FP64."""
    L = (4, 2, 3, 4)
    U = field(L, 0.2, 9)
    kw = dict(eps=0.1, alpha=1.0, forced_sweeps=1)
    ref, _ = O.cool(L, U, O.cool_params(mode=O.D0, **kw))
    with cl.Lattice(L) as lat:
        lat.set_links(U)
        lat.cool(cl.make_cool(mode=cl.CL_D0, **kw))
        assert np.abs(lat.links() - ref).max() <= 1e-12 * np.abs(ref).max()


def test_a_cooling_call_without_a_sweep_keeps_the_links(cl):
    L = (4, 4, 2, 3)
    U = field(L, 0.2, 2)
    with cl.Lattice(L) as lat:
        lat.set_links(U)
        rep = lat.cool(cl.make_cool(0.01, mode=cl.CL_D1, n_min=0, n_max=5, d_floor=1e9))
        assert rep["sweeps"] == 0
        assert np.array_equal(lat.links(), U)


@pytest.mark.parametrize("spread", [0, 0.1, 0.4, "mixed"])
@pytest.mark.parametrize("eps", [1e-6, 1e-3, 0.0143, 0.0145, 0.05, 0.4])
@pytest.mark.parametrize("k_ref", [0.0, 3.0])
def test_update_over_step_sizes(cl, spread, eps, k_ref):
    """One CL step.  The step sizes put the exponent's norm below, next to and beyond the halvings of its
    series and the fixed-point range, and lie on both sides of the noise constant's (eps = 0.0144).  The update
    is three products of matrices of size max |U| exp(|A|); 1e-12 of the result is several hundred roundings.
    (The drift itself is off by up to 1e-11 of its size for links far from SU(3), times eps.)"""
    L = (4, 3, 2, 5)
    U = field(L, spread, 31)
    if k_ref:
        ref, _, _ = O.cl_step_adaptive(L, U, 6.0, 1.0, eps, k_ref, 99, 4)
    else:
        ref = O.cl_step(L, U, 6.0, 1.0, eps, 99, 4)
    if not np.isfinite(ref).all():
        pytest.skip("the reference step itself overflows")
    with cl.Lattice(L, beta=6.0, theta=1.0, seed=99) as lat:
        lat.set_links(U)
        cl.cl_set_step(lat.h, 4)
        lat.set_adaptive_step(k_ref)
        lat.step(eps)
        Ug = lat.links()
    assert np.abs(Ug - ref).max() <= 1e-12 * np.abs(ref).max() + 1e-11 * eps * np.abs(ref).max() ** 2


@pytest.mark.parametrize("eps", [1e-4, 0.02, 0.4])
def test_fp32_storage_update_over_step_sizes(cl, eps):
    """The FP32-storage exponential is rounded to float once; the product and the determinant's root are
    ~20 dependent roundings of 6e-8 on links of order one: 5e-6 of the result."""
    L = (4, 3, 2, 5)
    U = field(L, 0, 31).astype(np.complex64).astype(np.complex128)
    ref = O.cl_step(L, U, 6.0, 1.0, eps, 99, 0)
    with cl.Lattice(L, beta=6.0, theta=1.0, seed=99, prec=cl.CL_FP32_STORAGE) as lat:
        lat.set_links(U)
        lat.step(eps)
        assert np.abs(lat.links() - ref).max() <= 5e-6 * np.abs(ref).max()


def test_reprojection_of_links_off_determinant_one(cl):
    """det U away from 1 (beyond the fixed-point series): the principal cube root, as everywhere."""
    L = (2, 4, 3, 2)
    U = field(L, 0, 8) * (1.0 + 1e-6)
    U[3, 1] *= 1.01 * np.exp(0.2j)
    ref = O.cl_step(L, U, 0.0, 0.0, 1e-3, 5, 0)
    with cl.Lattice(L, beta=0.0, theta=0.0, seed=5) as lat:
        lat.set_links(U)
        lat.step(1e-3)
        assert np.abs(lat.links() - ref).max() <= 1e-12


@pytest.mark.parametrize("spread", [0, 0.1, 0.4, "mixed"])
@pytest.mark.parametrize("k_ref", [0.0, 3.0])
def test_df64_form_inside_and_outside_the_range(cl, spread, k_ref):
    """The same kernels on double-float links: drift, one step, observables.  Links and drift are rounded to 2^-48
    on their way out, below the FP64 form's bounds above."""
    L, eps = (4, 3, 2, 5), 1e-3
    w = field(L, spread, 31).view(np.float64)
    hi = w.astype(np.float32).astype(np.float64)
    U = (hi + (w - hi).astype(np.float32)).view(np.complex128)  # exact double-float numbers
    top = np.abs(U).max()
    if k_ref:
        ref, _, _ = O.cl_step_adaptive(L, U, 6.0, 1.0, eps, k_ref, 99, 0)
    else:
        ref = O.cl_step(L, U, 6.0, 1.0, eps, 99, 0)
    Xr, obs_r = O.drift(L, U, 6.0, 1.0), O.observables(L, U, 6.0, 1.0)
    with cl.Lattice(L, beta=6.0, theta=1.0, seed=99, prec=cl.CL_DF64) as lat:
        lat.set_links(U)
        assert np.array_equal(lat.links(), U)
        X, obs = lat.drift(), lat.observables()
        lat.set_adaptive_step(k_ref)
        lat.step(eps)
        Ug = lat.links()
    assert np.abs(X - Xr).max() <= 1e-11 * np.abs(Xr).max()
    scale = max(abs(obs_r["sw_re"]), 6.0 * 6 * I.volume(L))
    for k in ("plaq_re", "plaq_im", "un"):
        assert abs(obs[k] - obs_r[k]) <= 1e-12 * max(1.0, abs(obs_r[k])), k
    for k in ("q_re", "q_im", "sw_re", "sw_im"):
        assert abs(obs[k] - obs_r[k]) <= 1e-12 * scale, k
    assert np.abs(Ug - ref).max() <= 1e-12 * np.abs(ref).max() + 1e-11 * eps * top ** 2
