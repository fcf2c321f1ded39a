"""FP32 storage: the cooling gradient and the norms behind the stop rule, bit for bit.

The rule stops a call when the norm's decrease falls below tol_rel of its distance from one; chains meet that
threshold within FP32 rounding, so the order in which a site's floats are summed decides how many sweeps they take.
It is one order in every shape of the kernels: forward links mu = 0 .. 3, then the backward ones, each entry one chain
of fused multiply-adds.  Restated here with exact float32 multiply-adds.

Tolerance of the norms: the lattice's sum runs in FP64 over exact site numbers, below 100 dependent roundings of
1.1e-16; 2e-14 of the norm.  (Summed in another order they differ by 1e-7 / sqrt(V) > 1e-10.)"""
import numpy as np
import pytest

import lattice_inputs as I

pytestmark = pytest.mark.gpu

# narrow with whole and partial groups, extents of one; wide; wide with several rounds a block and a partial tail
SHAPES = [(4, 4, 4, 4), (5, 3, 7, 2), (1, 4, 4, 3), (16, 16, 12, 9), (17, 16, 17, 16)]


@pytest.fixture(scope="module")
def cl():
    from paper_1311_1056_gb300 import cl as c
    return c


def fma(a, b, c):
    """float32 a b + c, rounded once: the sum in double rounded to odd, then to float."""
    p, c = a.astype(np.float64) * b.astype(np.float64), c.astype(np.float64)
    s = p + c
    t = s - p
    err = (p - (s - t)) + (c - t)
    even = (s.view(np.int64) & 1) == 0
    s = np.where((err != 0) & even, np.nextafter(s, np.where(err > 0, np.inf, -np.inf)), s)
    return s.astype(np.float32)


def links(L, seed):
    return I.sl3c_lattice(L, seed, 0.02).astype(np.complex64)


def hop_back(L, mu):
    """Site index of x - e_mu for every site."""
    x = I.coords(L)
    x[:, mu] = (x[:, mu] - 1) % L[mu]
    return x[:, 0] + L[0] * (x[:, 1] + L[1] * (x[:, 2] + L[2] * x[:, 3]))


def site_sums(L, U):
    """The nine numbers of G_x and the sum of the diagonal after the forward links, in float32."""
    V = I.volume(L)
    re, im = np.ascontiguousarray(U.real), np.ascontiguousarray(U.imag)
    d = [np.zeros(V, np.float32) for _ in range(3)]
    o = {q: [np.zeros(V, np.float32), np.zeros(V, np.float32)] for q in ((0, 1), (0, 2), (1, 2))}
    for dir in range(8):
        mu = dir & 3
        site = np.arange(V) if dir < 4 else hop_back(L, mu)
        r, i = re[site, mu], im[site, mu]
        for k in range(3):
            row = [(r[:, j, k], i[:, j, k]) if dir < 4 else (r[:, k, j], i[:, k, j]) for j in range(3)]
            for j in range(3):
                a, b = row[j]
                sg = np.float32(1 if dir < 4 else -1)
                d[j] = fma(sg * a, a, fma(sg * b, b, d[j]))
            for (p, q), s in o.items():
                (ar, ai), (br, bi) = row[p], row[q]
                if dir < 4:  # + a conj(b)
                    s[0] = fma(ai, bi, fma(ar, br, s[0]))
                    s[1] = fma(ai, br, fma(ar, -bi, s[1]))
                else:        # - conj(a) b
                    s[0] = fma(-ai, bi, fma(-ar, br, s[0]))
                    s[1] = fma(ai, br, fma(-ar, bi, s[1]))
        if dir == 3:
            un = (d[0] + d[1]) + d[2]
    return d, o, un


def gradient(d, o):
    f = np.empty((8, d[0].size), np.float32)
    four, two, r3 = np.float32(4), np.float32(2), np.float32(0.57735026918962576451)
    f[0], f[1] = four * o[0, 1][0], -(four * o[0, 1][1])
    f[2] = two * (d[0] - d[1])
    f[3], f[4] = four * o[0, 2][0], -(four * o[0, 2][1])
    f[5], f[6] = four * o[1, 2][0], -(four * o[1, 2][1])
    f[7] = two * r3 * ((d[0] + d[1]) - two * d[2])
    return f


def norm_of(un):
    return un.astype(np.float64).sum() / (12.0 * un.size)


def link_norms(U):
    """norm2 of a link: one chain over its entries."""
    s = np.zeros(U.shape[:2], np.float32)
    for k in range(9):
        e = U[..., k // 3, k % 3]
        a, b = np.ascontiguousarray(e.real), np.ascontiguousarray(e.imag)
        s = fma(a, a, fma(b, b, s))
    return s


@pytest.mark.parametrize("L", SHAPES)
def test_gradient_and_norm_are_summed_in_one_order(cl, L):
    U = links(L, 7)
    d, o, un = site_sums(L, U)
    with cl.Lattice(L, prec=cl.CL_FP32_STORAGE) as lat:
        lat.set_links(U.astype(np.complex128))
        f = lat.cool_gradient()
        rep = lat.cool(cl.make_cool(0.01, alpha=1.0, mode=cl.CL_D2_MEANABS, forced_sweeps=1))
    want = gradient(d, o)
    assert np.array_equal(f, want.T.astype(np.float64))
    assert abs(rep["un_before"] - norm_of(un)) <= 2e-14 * norm_of(un)
    D = np.abs(want.astype(np.float64)).mean()
    assert abs(1.0 / rep["alpha_ad_last"] - D) <= 2e-14 * D


@pytest.mark.parametrize("L", SHAPES)
def test_norm_after_a_sweep_is_summed_in_one_order(cl, L):
    U = links(L, 9)
    with cl.Lattice(L, prec=cl.CL_FP32_STORAGE) as lat:
        lat.set_links(U.astype(np.complex128))
        rep = lat.cool(cl.make_cool(0.01, alpha=0.5, mode=cl.CL_D1, forced_sweeps=2))
        V = lat.links().astype(np.complex64)
    n = link_norms(V.reshape(-1, 4, 3, 3))
    un = ((n[:, 0] + n[:, 1]) + n[:, 2]) + n[:, 3]
    assert abs(rep["un_after"] - norm_of(un)) <= 2e-14 * norm_of(un)


def test_sites_of_any_size_reach_the_norm(cl):
    """A few sites of huge links beside ordinary ones (their norms leave the integers' range)."""
    L = (4, 4, 4, 4)
    U = links(L, 3)
    U[17] *= np.float32(40.0)
    U[200, 2] *= np.float32(1e6)
    with cl.Lattice(L, prec=cl.CL_FP32_STORAGE) as lat:
        lat.set_links(U.astype(np.complex128))
        rep = lat.cool(cl.make_cool(1e-20, alpha=1.0, mode=cl.CL_D1, forced_sweeps=1))
        V = lat.links().astype(np.complex64)
    n = link_norms(V.reshape(-1, 4, 3, 3))
    un = ((n[:, 0] + n[:, 1]) + n[:, 2]) + n[:, 3]
    assert abs(rep["un_after"] - norm_of(un)) <= 2e-14 * norm_of(un)
