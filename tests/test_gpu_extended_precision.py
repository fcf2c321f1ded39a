"""Drift and charge density of the FP64 form against extended precision (long double: 64 bits or more of significand).

Fixed point has one absolute error for numbers of any size, so a field kept too small for its range loses bits that
FP64 would keep.  The bounds are 1.5 times the rms error that an FP64 evaluation of the same formulas shows on these
links (of the result's rms: drift 2.7e-16 at spread 0.27 and 2.5e-16 at 0.1, charge density 4.5e-16 and 6.0e-16; of
smooth links 1.45e-15 and 3.8e-15 at 0.01, 1.8e-14 and 4.8e-14 at 0.001)."""
import numpy as np
import pytest

import lattice_inputs as I

pytestmark = pytest.mark.gpu

L = (4, 4, 3, 5)
V = I.volume(L)
PLANES = ((0, 1), (0, 2), (0, 3), (1, 2), (1, 3), (2, 3))
LD = np.clongdouble


@pytest.fixture(scope="module")
def cl():
    if np.finfo(np.longdouble).eps > 2e-19:
        pytest.skip("no extended precision here")
    from paper_1311_1056_gb300 import cl as c
    return c


def hop(f, mu, d):
    return np.roll(f.reshape((L[3], L[2], L[1], L[0]) + f.shape[1:]), -d, 3 - mu).reshape(f.shape)


def mm(*m):
    r = m[0]
    for b in m[1:]:
        r = (r[..., :, :, None] * b[..., None, :, :]).sum(-2)
    return r


def adj(m):
    r = np.empty_like(m)
    for i in range(3):
        for j in range(3):
            a, b = [k for k in range(3) if k != j]
            p, q = [k for k in range(3) if k != i]
            r[..., i, j] = (-1) ** (i + j) * (m[..., a, p] * m[..., b, q] - m[..., a, q] * m[..., b, p])
    return r


def tr(m):
    return m[..., 0, 0] + m[..., 1, 1] + m[..., 2, 2]


def com(a, b):
    return mm(a, b) - mm(b, a)


def fields(U):
    P = [mm(U[:, m], hop(U[:, n], m, 1), adj(mm(U[:, n], hop(U[:, m], n, 1)))) for m, n in PLANES]
    D = [p - adj(p) for p in P]
    F = []
    for (m, n), d in zip(PLANES, D):
        t = hop(mm(adj(U[:, m]), d, U[:, m]), m, -1)
        F.append(d + t + hop(mm(adj(U[:, n]), d + t, U[:, n]), n, -1))
    return P, D, F


KAPPA = np.longdouble(-1) / (256 * np.longdouble("3.14159265358979323846264338327950288") ** 2)


def density(F):
    return KAPPA * (tr(mm(F[0], F[5])) - tr(mm(F[1], F[4])) + tr(mm(F[2], F[3])))


def drift(U, P, D, F, beta, theta):
    b6, X = np.longdouble(beta) / 6, np.zeros((V, 4, 3, 3), LD)
    for p, (m, n) in enumerate(PLANES):
        G = (-1 if p in (1, 4) else 1) * LD(-1j) * LD(theta) * KAPPA * F[5 - p]
        a, u, d = U[:, m], U[:, n], D[p]
        ai, ui, Pi = adj(a), adj(u), adj(P[p])
        ab = mm(a, hop(u, m, 1))
        G1, G3r = mm(a, hop(G, m, 1), ai), mm(u, hop(G, n, 1), ui)
        Gh = G + G1 + mm(ab, hop(hop(G, m, 1), n, 1), adj(ab)) + mm(P[p], G3r, Pi)
        K = mm(Gh, P[p]) + mm(Pi, Gh)
        X[:, m] += K + com(d, G) - b6 * d
        X[:, n] += b6 * d - K
        X[:, n] += hop(mm(ai, K + com(d, G) + com(d, G1) - b6 * d, a), m, -1)
        X[:, m] += hop(mm(ui, com(d, G3r) - K + b6 * d, u), n, -1)
    return X


def links(spread, seed, rough=0.012):
    """SU(3) links exp(i spread h) with a non-unitary part of size rough, det = 1."""
    r = np.random.default_rng(seed)

    def gauss():
        z = r.normal(size=(V, 4, 3, 3)) + 1j * r.normal(size=(V, 4, 3, 3))
        return z - (tr(z) / 3)[..., None, None] * np.eye(3)

    def expm(A):
        E = np.eye(3) + A / 20
        for k in range(19, 0, -1):
            E = np.eye(3) + mm(A, E) / k
        return E

    h = gauss()
    h = expm(0.25j * spread * (h + h.conj().swapaxes(-1, -2)))
    U = mm(expm(rough * gauss()), h, h, h, h)
    return U * (np.linalg.det(U) ** (-1 / 3))[..., None, None]


def rms(err, ref):
    return float(np.sqrt((np.abs(err) ** 2).sum() / (np.abs(ref) ** 2).sum()))


@pytest.mark.parametrize("spread,drift_bound,density_bound", [(0.27, 4.0e-16, 6.8e-16), (0.1, 3.8e-16, 9.0e-16)])
def test_drift_and_charge_density_keep_double_precision(cl, spread, drift_bound, density_bound):
    U = links(spread, 1)
    P, D, F = fields(U.astype(LD))
    q = density(F)
    for beta, theta in ((6.0, 1.0), (5.9, 0.01), (6.2, 0.5 + 0.3j), (6.0, 0.0)):
        with cl.Lattice(L, beta=beta, theta=theta) as lat:
            lat.set_links(U)
            assert rms(lat.drift() - drift(U.astype(LD), P, D, F, beta, theta), drift(U.astype(LD), P, D, F, beta, theta)) <= drift_bound
            assert rms(lat.qdensity() - q, q) <= density_bound


@pytest.mark.parametrize("spread,rough,drift_bound,density_bound", [(0.01, 1e-4, 2.2e-15, 5.7e-15), (0.001, 1e-5, 2.7e-14, 7.2e-14)])
def test_smooth_links_keep_double_precision(cl, spread, rough, drift_bound, density_bound):
    U = links(spread, 1, rough)
    P, D, F = fields(U.astype(LD))
    X, q = drift(U.astype(LD), P, D, F, 6.0, 1.0), density(F)
    with cl.Lattice(L, beta=6.0, theta=1.0) as lat:
        lat.set_links(U)
        assert rms(lat.drift() - X, X) <= drift_bound
        assert rms(lat.qdensity() - q, q) <= density_bound


@pytest.mark.parametrize("spread,rough,fp64", [(1.0, 0.0, 4.41e-16), (0.27, 0.012, 4.58e-16), (0.03, 1e-3, 1.325e-15), (0.01, 1e-4, 3.705e-15)])
def test_charge_density_is_no_worse_than_fp64(cl, spread, rough, fp64):
    """Mean over eight sets of links against the same mean of kernels in FP64 arithmetic, on the same links.  The means
    of either scatter by 1.5 to 3 percent (4 to 8 percent a set): 5 percent between them."""
    err = []
    for seed in range(11, 19):
        U = links(spread, seed, rough)
        q = density(fields(U.astype(LD))[2])
        with cl.Lattice(L, beta=6.0, theta=1.0) as lat:
            lat.set_links(U)
            err.append(rms(lat.qdensity() - q, q))
    assert np.mean(err) <= 1.05 * fp64
