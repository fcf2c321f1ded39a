"""The chain kernel's fixed-point path and its FP64 fallback against the chain oracle: link counts at the edges of
a warp and of the path, starts inside the fixed-point range, just outside it (a product of links leaves it, the
links do not) and far outside, Langevin steps beyond its noise range, and links whose determinant is not one.

Tolerance: a link's error after a step is that of the cyclic product (n products, each 2^-53 of its factors' norms)
times eps |beta|, plus a few roundings of the link itself in the step and each sweep: with norms below M everywhere,
steps (n eps + 10 + 10 sweeps) M^2 2^-53; M^2 = 4 max|U|^4 covers the products."""
import numpy as np
import pytest

import oracle as O
from paper_1311_1056_gb300 import cl

pytestmark = pytest.mark.gpu


def _start(kind, n, seed):
    rng = np.random.default_rng(seed)
    if kind in ("near", "beyond"):
        return O.pc_random_gauge(O.pc_cold(n), seed, 0.05 if kind == "near" else 0.7)
    U = O.pc_random_gauge(O.pc_cold(n), seed, 0.05)
    if kind == "product":  # boosts along one axis that add up
        b = 0.6 / n
        return U @ np.diag([np.exp(b), np.exp(-b)]).astype(complex)
    return U * (1 + 0.05 * (rng.normal(size=(n, 1, 1)) + 1j * rng.normal(size=(n, 1, 1))))  # "det"


@pytest.mark.parametrize("mode", [cl.CL_D1, cl.CL_D2_RMS])
@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 512, 513])
@pytest.mark.parametrize("kind,eps", [("near", 0.005), ("product", 0.005), ("beyond", 0.005), ("det", 0.01),
                                      ("near", 0.1), ("near", 0.4)])
def test_chain_steps(kind, eps, n, mode):
    if n > 100 and (kind == "beyond" or eps > 0.05):
        pytest.skip("products of this many links run away in the oracle as well")
    steps, sweeps = 3, 4
    kw = dict(alpha=0.5, mode=mode, forced_sweeps=sweeps)
    betas, seeds = [1.2, 0.8 + 0.4j], [21, 22]
    U0 = np.stack([_start(kind, n, s) for s in seeds])
    with cl.PolyakovChains(2, n, betas, seeds) as pc:
        pc.set_links(U0)
        rec = pc.run(steps, eps, cl.make_cool(0.01, **kw), obs_every=1)
        U = pc.links()
        pc.set_links(U0)
    with cl.PolyakovChains(2, n, betas, seeds) as pc:  # a run split into calls
        pc.set_links(U0)
        for _ in range(steps):
            pc.run(1, eps, cl.make_cool(0.01, **kw), obs_every=0)
        assert np.array_equal(pc.links(), U, equal_nan=True)
    for c in range(2):
        ref, orec = O.pc_trajectory(U0[c], betas[c], eps, seeds[c], 0, steps, O.cool_params(0.01, **kw))
        if not np.isfinite(ref).all():
            continue
        m2 = 4 * max(np.abs(ref).max(), np.abs(U0[c]).max(), 1.0) ** 4
        tol = steps * (n * eps + 10 + 10 * sweeps) * m2 * 2.0 ** -53 * max(1.0, np.abs(orec[:, :2]).max())
        assert np.abs(U[c] - ref).max() < tol
        assert np.array_equal(rec[:, c, 4], orec[:, 4])
        assert np.abs(rec[:, c, :3] - orec[:, :3]).max() < n * tol
