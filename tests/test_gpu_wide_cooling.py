"""Cooling and steps of links in and out of the fixed-point range where blocks take several groups of sites: odd
volumes above 24,576 sites (the wide shape) and above 65,536 (several rounds a block, a partial last group), and
fused FP64 batches.  Two sweeps multiply each link by four matrices near 1: 1e-12 of max |U| is hundreds of roundings
(DF64: links are stored to 2^-48 of their size)."""
import numpy as np
import pytest

import oracle as O
import lattice_inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cl():
    from paper_1311_1056_gb300 import cl as c
    return c


def field(L, kind, seed):
    """scattered: near SU(3) with one link in 200 far from it; rough: all of them some way off."""
    if kind == "rough":
        return I.sl3c_lattice(L, seed, 0.15)
    U = I.sl3c_lattice(L, seed, 0.02)
    r = I.rng(seed + 1)
    pick = r.random(U.shape[:2]) < 0.005
    U[pick] = I.random_sl3c(r, int(pick.sum()), 0.35)
    return U


@pytest.mark.parametrize("L", [(17, 13, 11, 11), (17, 16, 17, 16)])
@pytest.mark.parametrize("kind", ["scattered", "rough"])
@pytest.mark.parametrize("mode", ["D1", "D2_MEANABS"])
def test_wide_cooling_against_the_oracle(cl, L, kind, mode):
    U = field(L, kind, 3)
    kw = dict(eps=1e-3, alpha=1.0, forced_sweeps=2)
    ref, rep = O.cool(L, U, O.cool_params(mode=getattr(O, mode), **kw))
    top = np.abs(ref).max()
    for prec, tol in (("CL_FP64", 1e-12), ("CL_DF64", 1e-12)):
        with cl.Lattice(L, prec=getattr(cl, prec)) as lat:
            lat.set_links(U)
            got = lat.cool(cl.make_cool(mode=getattr(cl, "CL_" + mode), **kw))
            assert got["sweeps"] == 2
            assert np.abs(lat.links() - ref).max() <= tol * top
        for k in ("un_before", "un_after"):
            assert abs(got[k] - rep[k]) <= 1e-12 * rep[k], (prec, k)


@pytest.mark.parametrize("kind", ["scattered", "rough"])
def test_fused_fp64_batch_with_links_out_of_range(cl, kind):
    """Chains of uneven volumes: the fused launches give each the links of its lone run, bit for bit."""
    shapes = [(4, 4, 4, 4), (9, 7, 5, 6), (17, 13, 11, 11)]
    cp = cl.make_cool(1e-3, alpha=0.5, mode=cl.CL_D2_MEANABS, forced_sweeps=2)
    cp1 = cl.make_cool(1e-3, alpha=0.5, mode=cl.CL_D1, forced_sweeps=3)
    lone, lats = [], []
    for i, L in enumerate(shapes):
        U = field(L, kind, 10 + i)
        lat = cl.Lattice(L, beta=6.0, theta=0.5 * i, seed=5 + i, own_stream=True)
        lat.set_links(U)
        lats.append(lat)
        with cl.Lattice(L, beta=6.0, theta=0.5 * i, seed=5 + i) as one:
            one.set_links(U)
            for _ in range(2):
                one.step(1e-3)
                one.cool(cp1 if i == 1 else cp)
            lone.append(one.links())
    batch = cl.Batch(lats, 1e-3, [cp, cp1, cp])
    batch.run(2)
    for lat, ref in zip(lats, lone):
        lat.synchronize()
        assert np.array_equal(lat.links(), ref)
    batch.close()
    for lat in lats:
        lat.close()
