"""What the framework is timed on: complex-Langevin work through its public entry points.

A case names one kind of work and its sizes.  The kinds are what a user's program does:

* traj     chains advanced by cl_trajectory: CL steps, each followed by cooling sweeps, the
           observables recorded after the last one.  The program holds its links in device
           tensors: it hands them in, and takes the new ones out.
* replay   one captured step (CL step with the adaptive step size, adaptive cooling) replayed
           as a CUDA graph: how long runs and the request server advance a chain.
* cool     gauge cooling alone, with the adaptive strength, of links handed in.
* obs      plaquette, unitarity norm, topological charge and action of links handed in.
* batch    chains of mixed sizes advanced by one fused launch per kernel family.
* host     links from page-locked host memory, one step with cooling, links back to the host.
* pchain   SU(2) Polyakov chains, CL steps with adaptive cooling.

`form` is the arithmetic form of the links: fp64, fp32 (FP32 storage) or df64 (double-float).
Links and observables of the fp32 form carry FP32 precision and are returned in it.
"""
import math

import numpy as np
import torch

from paper_1311_1056_gb300 import cl

PREC = {"fp64": cl.CL_FP64, "fp32": cl.CL_FP32_STORAGE, "df64": cl.CL_DF64}
MODE = {"d0": cl.CL_D0, "d1": cl.CL_D1, "d2": cl.CL_D2_MEANABS}
OBS = ("plaq_re", "plaq_im", "un", "q_re", "q_im", "sw_re", "sw_im", "s_re", "s_im")
DEV = "cuda" if torch.cuda.is_available() else "cpu"


def _case(kind, form, L, **more):
    return dict(kind=kind, form=form, L0=L[0], L1=L[1], L2=L[2], L3=L[3], **more)


def listed():
    return [
        # the smallest chain of the repository: 4^4, ten short steps with five D_0 sweeps each; launches count
        dict(_case("traj", "fp64", (4, 4, 4, 4), beta=6.0, theta=0.0, eps=0.01, mode="d0", sweeps=5, steps=10),
             name="traj_fp64_4x4_d0"),
        # the single-chain physics run: 16^4 with the theta term, adaptive D_2 strength, FP64 links
        dict(_case("traj", "fp64", (16, 16, 16, 16), beta=6.0, theta=1.0, eps=0.005, mode="d2", sweeps=4, steps=2),
             name="traj_fp64_16x4_d2"),
        # the throughput run: 32^4, one step and ten D_1 sweeps, FP64 links
        dict(_case("traj", "fp64", (32, 32, 32, 32), beta=6.2, theta=1.0, eps=0.005, mode="d1", sweeps=10, steps=1),
             name="traj_fp64_32x4_d1"),
        # the same run with FP32 link storage
        dict(_case("traj", "fp32", (32, 32, 32, 32), beta=6.2, theta=1.0, eps=0.005, mode="d1", sweeps=10, steps=1),
             name="traj_fp32_32x4_d1"),
        # double-float links, a medium lattice
        dict(_case("traj", "df64", (16, 16, 16, 16), beta=6.0, theta=1.0, eps=0.005, mode="d1", sweeps=5, steps=1),
             name="traj_df64_16x4_d1"),
        # odd extents, Wilson action only (theta = 0), FP64
        dict(_case("traj", "fp64", (13, 9, 11, 15), beta=5.9, theta=0.0, eps=0.01, mode="d0", sweeps=3, steps=2),
             name="traj_fp64_odd_wilson"),
        # one served request: 8^4, FP32 storage, captured step with adaptive step size and cooling
        dict(_case("replay", "fp32", (8, 8, 8, 8), beta=6.0, theta=1.0, eps=0.005, steps=8), name="replay_fp32_8x4"),
        # a cooling study on its own: 12^4 FP64 links, up to twenty adaptive D_2 sweeps
        dict(_case("cool", "fp64", (12, 12, 12, 12), eps=0.005, mode="d2", sweeps=20), name="cool_fp64_12x4_d2"),
        # measuring a stored configuration: observables of 24^4 FP64 links
        dict(_case("obs", "fp64", (24, 24, 24, 24), beta=6.1, theta=0.5), name="obs_fp64_24x4"),
        # the ensemble: twelve chains of 8^4, 12^4 and 16^4, FP32 storage, fused launches
        dict(kind="batch", form="fp32", chains=12, Lmin=8, Lmax=16, eps=0.005, steps=2, name="batch_fp32_12"),
        # links from and to the host around every step: FP32 storage, 24 x 24 x 24 x 32
        dict(_case("host", "fp32", (24, 24, 24, 32), beta=6.2, theta=1.0, eps=0.005, mode="d1", sweeps=2, steps=1),
             name="host_fp32_24x32"),
        # SU(2) Polyakov chains of 30 links: eight steps with adaptive cooling
        dict(kind="pchain", form="fp64", chains=512, links=30, eps=0.005, sweeps=5, steps=8, name="pchain_512x30"),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("traj", "traj", "traj", "traj", "replay", "cool", "obs", "batch", "host", "pchain"))
    eps = round(rng.uniform(0.003, 0.01), 5)
    if kind == "batch":
        lmin = rng.randint(4, 9)
        return dict(kind="batch", form=rng.choice(("fp32", "fp64")), chains=_logint(rng, 2, 16), Lmin=lmin,
                    Lmax=lmin + rng.randint(1, 6), eps=eps, steps=rng.randint(1, 2))
    if kind == "pchain":
        return dict(kind="pchain", form="fp64", chains=_logint(rng, 8, 1000), links=_logint(rng, 2, 60), eps=eps,
                    sweeps=rng.randint(1, 8), steps=rng.randint(2, 12))
    form = rng.choice(("fp64", "fp64", "fp32", "fp32", "df64")) if kind == "traj" else rng.choice(("fp64", "fp32"))
    top = 24 if form == "fp64" else 28
    if kind == "replay":
        top = 16
    L = [_logint(rng, 4, top) for _ in range(4)]
    if rng.random() < 0.15:
        L[rng.randrange(4)] = rng.randint(1, 3)
    beta, theta = round(rng.uniform(5.8, 6.2), 3), rng.choice((0.0, 0.5, 1.0, round(rng.uniform(0.1, 1.5), 3)))
    if kind == "replay":
        return _case(kind, form, L, beta=beta, theta=theta, eps=eps, steps=rng.randint(2, 8))
    if kind == "cool":
        return _case(kind, form, L, eps=eps, mode=rng.choice(("d0", "d1", "d2")), sweeps=rng.randint(1, 20))
    if kind == "obs":
        return _case(kind, form, L, beta=beta, theta=theta)
    if kind == "host":
        return _case(kind, form, L, beta=beta, theta=theta, eps=eps, mode=rng.choice(("d0", "d1", "d2")),
                     sweeps=rng.randint(0, 4), steps=1)
    return _case(kind, form, L, beta=beta, theta=theta, eps=eps, mode=rng.choice(("d0", "d1", "d2")),
                 sweeps=rng.randint(1, 10), steps=rng.randint(1, 2))


# ------------------------------------------------------------------ inputs
def _links(L, seed, tag=0):
    """Links such as a chain holds once it has thermalised: SU(3) matrices scattered around the identity
    (plaquette near 0.6), slightly off SU(3) (unitarity norm - 1 near 1e-3), det = 1.  AoS [site][mu][3][3]."""
    g = torch.Generator(device=DEV)
    g.manual_seed(1000003 * int(seed) + tag)
    n = 4 * math.prod(L)
    z = torch.randn((2, n, 3, 3, 2), generator=g, device=DEV, dtype=torch.float64)
    z = torch.view_as_complex(z)
    u = torch.eye(3, dtype=torch.complex128, device=DEV) + 0.27 * z[0]
    rows = []
    for i in range(3):
        r = u[:, i]
        for q in rows:
            r = r - (q.conj() * r).sum(-1, keepdim=True) * q
        rows.append(r / r.abs().square().sum(-1, keepdim=True).sqrt())
    u = torch.stack(rows, 1)
    u = u + 0.012 * _mm(z[1], u)
    u = u * torch.pow(_det(u), -1.0 / 3.0)[:, None, None]
    return u.reshape(math.prod(L), 4, 3, 3).contiguous()


def _shape(case):
    return (case["L0"], case["L1"], case["L2"], case["L3"])


def _cool_params(case, forced=True):
    return cl.make_cool(case["eps"], alpha=0.1 if case["mode"] == "d2" else 1.0, mode=MODE[case["mode"]], n_min=0,
                        n_max=case["sweeps"], tol_rel=0.01, forced_sweeps=case["sweeps"] if forced else -1)


def _served_cool(eps):
    """Cooling as the ensembles and the request server run it: up to ten sweeps of alpha / D_2, alpha = 0.1."""
    return cl.make_cool(eps, alpha=0.1, mode=cl.CL_D2_MEANABS, n_max=10, tol_rel=0.01, d_floor=1e-6)


K_REF = 12.0


def _members(case, seed):
    """The chains of a batch: extents spread over [Lmin, Lmax], couplings and seeds of their own."""
    rng = np.random.default_rng([int(seed), 77])
    out = []
    for i in range(case["chains"]):
        n = case["Lmin"] + (i * (case["Lmax"] - case["Lmin"])) // max(1, case["chains"] - 1)
        out.append(dict(L=(n,) * 4, beta=float(rng.uniform(5.8, 6.2)), theta=float(rng.choice([0.0, 0.5, 1.0])),
                        seed=int(rng.integers(1 << 40)), tag=i + 1))
    return out


class _State:
    pass


def prepare(case, seed):
    s = _State()
    s.case, kind = case, case["kind"]
    prec = PREC[case["form"]]
    if kind == "pchain":
        rng = np.random.default_rng([int(seed), 5])
        n = case["chains"]
        s.beta = rng.uniform(0.5, 1.5, n) + 1j * rng.uniform(-0.5, 0.5, n)
        s.seeds = rng.integers(1 << 40, size=n)
        s.u0 = _chain_links(case, seed)
        s.chains = cl.PolyakovChains(n, case["links"], s.beta, s.seeds)
        s.cp = cl.make_cool(case["eps"], alpha=1.0, mode=cl.CL_D1, n_max=case["sweeps"], tol_rel=0.01)
        return s
    if kind == "batch":
        s.lats, s.out = [], []
        for m in _members(case, seed):
            lat = cl.Lattice(m["L"], beta=m["beta"], theta=m["theta"], prec=prec, seed=m["seed"], own_stream=True)
            u = _links(m["L"], seed, m["tag"])
            torch.cuda.synchronize()
            cl.cl_set_links_device(lat.h, u.data_ptr())
            lat.set_adaptive_step(K_REF)
            lat.synchronize()
            s.lats.append(lat)
            s.out.append(torch.empty_like(u))
        s.batch = cl.Batch(s.lats, case["eps"], [_served_cool(case["eps"])] * len(s.lats))
        return s
    L = _shape(case)
    s.lat = cl.Lattice(L, beta=case.get("beta", 6.0), theta=case.get("theta", 0.0), prec=prec,
                       seed=int(seed) + 12345, own_stream=(kind == "replay"))
    s.u = _links(L, seed)
    if kind == "host":
        s.host_in, s.host_out = (torch.empty(s.u.shape, dtype=s.u.dtype, pin_memory=True) for _ in range(2))
        s.host_in.copy_(s.u)
        s.np_in, s.np_out = s.host_in.numpy(), s.host_out.numpy()
        s.u = None
    else:
        s.out = torch.empty_like(s.u)
        torch.cuda.synchronize()
        cl.cl_set_links_device(s.lat.h, s.u.data_ptr())
    if kind in ("traj", "host"):
        s.cp = _cool_params(case)
    elif kind == "cool":
        s.cp = _cool_params(case, forced=False)
    elif kind == "replay":
        s.lat.set_adaptive_step(K_REF)
        s.lat.capture_step(case["eps"], _served_cool(case["eps"]))
    s.lat.synchronize()
    return s


def _out_links(case, t):
    """Links of the fp32 form in the precision that they are stored in."""
    return torch.view_as_real(t).to(torch.float32 if case["form"] == "fp32" else torch.float64)


def _out_obs(case, o):
    return torch.tensor([o[k] for k in OBS], dtype=torch.float32 if case["form"] == "fp32" else torch.float64)


def run(s):
    case, kind = s.case, s.case["kind"]
    if kind == "traj":
        cl.cl_set_links_device(s.lat.h, s.u.data_ptr())
        obs, rep = s.lat.trajectory(case["eps"], case["steps"], s.cp, obs_every=case["steps"])
        cl.cl_get_links_device(s.lat.h, s.out.data_ptr())
        return {"links": _out_links(case, s.out), "obs": _out_obs(case, obs[0]), "sweeps": rep[0]["sweeps"]}
    if kind == "replay":
        s.lat.replay(case["steps"])
        cl.cl_get_links_device(s.lat.h, s.out.data_ptr())
        s.lat.synchronize()
        return {"links": _out_links(case, s.out)}
    if kind == "cool":
        cl.cl_set_links_device(s.lat.h, s.u.data_ptr())
        rep = s.lat.cool(s.cp)
        cl.cl_get_links_device(s.lat.h, s.out.data_ptr())
        return {"links": _out_links(case, s.out), "sweeps": rep["sweeps"]}
    if kind == "obs":
        cl.cl_set_links_device(s.lat.h, s.u.data_ptr())
        return {"obs": _out_obs(case, s.lat.observables())}
    if kind == "batch":
        s.batch.run(case["steps"])
        for lat, o in zip(s.lats, s.out):
            cl.cl_get_links_device(lat.h, o.data_ptr())
        for lat in s.lats:
            lat.synchronize()
        return {"links": [_out_links(case, o) for o in s.out]}
    if kind == "host":
        s.lat.set_links(s.np_in)
        obs, _ = s.lat.trajectory(case["eps"], case["steps"], s.cp, obs_every=case["steps"])
        cl.cl_get_links(s.lat.h, s.lat.V, out=s.np_out)
        return {"links": _out_links(case, s.host_out), "obs": _out_obs(case, obs[0])}
    s.chains.set_links(s.u0)
    rec = s.chains.run(case["steps"], case["eps"], s.cp, obs_every=case["steps"])
    return {"links": s.chains.links().view(np.float64), "traces": rec[0, :, :3], "sweeps": rec[0, :, 4].astype(np.int64)}


# -------------------------------------------------------------------- work
def _step_flops(theta):
    """Flops per site of one CL step: inverses, plaquettes, clover field, drift, update."""
    if theta:
        return 4 * 126 + 6 * (738 + 1296 + 4608) + 4 * 1321
    return 4 * 126 + 6 * (738 + 828) + 4 * 1321


SWEEP_FLOPS = 914 + 209 + 4 * 360


def work(case):
    kind = case["kind"]
    if kind == "pchain":
        n = case["chains"] * case["links"]
        per = 2 * math.ceil(math.log2(max(2, case["links"]))) * 56 + 400 + 200 * case["sweeps"]
        return {"bytes": 2 * 64 * n, "flops": n * case["steps"] * per}
    real = 4 if case["form"] == "fp32" else 8
    if kind == "batch":
        v = 0
        flops = 0
        for m in _members(case, 0):
            n = math.prod(m["L"])
            v += n
            flops += n * case["steps"] * (_step_flops(1.0) + 2 * SWEEP_FLOPS)
        return {"bytes": 2 * v * 72 * real, "flops": flops}
    v = math.prod(_shape(case))
    out = 1 if kind == "obs" else 2
    by = out * v * 72 * 8
    if kind == "obs":
        return {"bytes": by, "flops": v * (504 + 6 * (738 + 1296 + 700))}
    if kind == "cool":
        return {"bytes": by, "flops": v * SWEEP_FLOPS * max(1, case["sweeps"] // 2)}
    sweeps = 2 if kind == "replay" else case["sweeps"]
    return {"bytes": by, "flops": v * case["steps"] * (_step_flops(case["theta"]) + sweeps * SWEEP_FLOPS)}


# ------------------------------------------------- the same in plain torch
# The method as its definitions give it, in 64 bits: the drift by differentiating the action, the noise
# from the published Philox4x32-10, the exponentials by matrix_exp.

def _mm(a, b):
    return (a.unsqueeze(-1) * b.unsqueeze(-3)).sum(-2)


def _det(m):
    return (m[..., 0, 0] * (m[..., 1, 1] * m[..., 2, 2] - m[..., 1, 2] * m[..., 2, 1])
            - m[..., 0, 1] * (m[..., 1, 0] * m[..., 2, 2] - m[..., 1, 2] * m[..., 2, 0])
            + m[..., 0, 2] * (m[..., 1, 0] * m[..., 2, 1] - m[..., 1, 1] * m[..., 2, 0]))


def _inv(m):
    """Inverse of a matrix of determinant 1: its adjugate, cofactor by cofactor."""
    c = [[None] * 3 for _ in range(3)]
    for i in range(3):
        for j in range(3):
            a, b = [k for k in range(3) if k != j]
            p, q = [k for k in range(3) if k != i]
            c[i][j] = (-1) ** (i + j) * (m[..., a, p] * m[..., b, q] - m[..., a, q] * m[..., b, p])
    return torch.stack([torch.stack(r, -1) for r in c], -2)


def _tr(m):
    return m[..., 0, 0] + m[..., 1, 1] + m[..., 2, 2]


def _hop(f, L, mu, d):
    """The field f at x + d e_mu (x0 runs fastest in the site index)."""
    g = f.reshape((L[3], L[2], L[1], L[0]) + f.shape[1:])
    return torch.roll(g, -d, 3 - mu).reshape(f.shape)


PLANES = ((0, 1), (0, 2), (0, 3), (1, 2), (1, 3), (2, 3))


def _plaq(U, L, mu, nu):
    a, b = U[:, mu], _hop(U[:, nu], L, mu, 1)
    c, d = _hop(U[:, mu], L, nu, 1), U[:, nu]
    return _mm(_mm(a, b), _inv(_mm(d, c)))


def _q(U, L, P):
    """Topological charge density, kappa [Tr F01 F23 - Tr F02 F13 + Tr F03 F12], clover F."""
    F = []
    for (mu, nu), p in zip(PLANES, P):
        d = p - _inv(p)
        um, un = U[:, mu], U[:, nu]
        t = _hop(_mm(_mm(_inv(um), d), um), L, mu, -1)
        w = _mm(_mm(_inv(un), d + t), un)
        F.append(d + t + _hop(w, L, nu, -1))
    k = -1.0 / (256.0 * math.pi ** 2)
    return k * (_tr(_mm(F[0], F[5])) - _tr(_mm(F[1], F[4])) + _tr(_mm(F[2], F[3])))


def _measure(U, L, beta, theta):
    P = [_plaq(U, L, *pl) for pl in PLANES]
    tr = torch.stack([_tr(p) for p in P])
    tri = torch.stack([_tr(_inv(p)) for p in P])
    sw = beta * (tr.numel() - (tr.sum() + tri.sum()) / 6.0)
    q = _q(U, L, P).sum()
    s = sw - 1j * theta * q
    plaq = tr.sum() / (3.0 * tr.numel())
    un = U.abs().square().sum() / (3.0 * U.shape[0] * 4)
    v = [plaq.real, plaq.imag, un, q.real, q.imag, sw.real, sw.imag, s.real, s.imag]
    return torch.tensor([float(x) for x in v], dtype=torch.float64)


def _drift(U, L, beta, theta):
    """X with D_a S = i Tr(lambda_a X): U (dS/dU)^T, by reverse mode on the holomorphic S."""
    W = U.detach().clone().requires_grad_(True)
    P = [_plaq(W, L, *pl) for pl in PLANES]
    S = sum(-(beta / 6.0) * (_tr(p) + _tr(_inv(p))).sum() for p in P)
    if theta:
        S = S - 1j * theta * _q(W, L, P).sum()
    (g,) = torch.autograd.grad(S.real, W)
    return _mm(U, g.conj().transpose(-1, -2))


def _philox(c, key):
    """Philox4x32-10 on int64 tensors that hold 32-bit words."""
    m32 = 0xFFFFFFFF

    def mul(a, b):
        lo_part = b * (a & 0xFFFF)
        hi_part = b * (a >> 16)
        return ((hi_part + (lo_part >> 16)) >> 16) & m32, (((hi_part & 0xFFFF) << 16) + lo_part) & m32

    k0, k1 = key & m32, (key >> 32) & m32
    for _ in range(10):
        h0, l0 = mul(0xD2511F53, c[0])
        h1, l1 = mul(0xCD9E8D57, c[2])
        c = (h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0)
        k0, k1 = (k0 + 0x9E3779B9) & m32, (k1 + 0xBB67AE85) & m32
    return c


def _normals(seeds, step, site, slot, pairs):
    """Box-Muller pairs keyed by (seed, step, site, slot, j): shape site.shape + (2 pairs,)."""
    out = []
    for j in range(pairs):
        z = torch.zeros_like(site)
        w = _philox((site, z + step, slot + z, z + j), seeds)
        u1 = (((w[0] >> 6) << 26) + (w[1] >> 6)).double().add(0.5) * 2.0 ** -52
        u2 = (((w[2] >> 6) << 26) + (w[3] >> 6)).double().add(0.5) * 2.0 ** -52
        r = (-2.0 * torch.log(u1)).sqrt()
        out += [r * torch.cos(2 * math.pi * u2), r * torch.sin(2 * math.pi * u2)]
    return torch.stack(out, -1)


def _hermitian(h):
    """sum_a h_a lambda_a."""
    r3 = 1.0 / math.sqrt(3.0)
    c = torch.complex
    z = torch.zeros_like(h[..., 0])
    rows = [[c(h[..., 2] + r3 * h[..., 7], z), c(h[..., 0], -h[..., 1]), c(h[..., 3], -h[..., 4])],
            [c(h[..., 0], h[..., 1]), c(r3 * h[..., 7] - h[..., 2], z), c(h[..., 5], -h[..., 6])],
            [c(h[..., 3], h[..., 4]), c(h[..., 5], h[..., 6]), c(-2 * r3 * h[..., 7], z)]]
    return torch.stack([torch.stack(r, -1) for r in rows], -2)


def _expm(A):
    """Taylor series after halving the argument s times, squared back s times."""
    n = float(A.abs().square().sum((-1, -2)).max().sqrt())
    s = max(0, math.ceil(math.log2(max(n, 1e-300))) + 1)
    B = A * 2.0 ** -s
    one = torch.eye(3, dtype=A.dtype, device=A.device)
    E = one + B / 18.0
    for k in range(17, 0, -1):
        E = one + _mm(B, E) / k
    for _ in range(s):
        E = _mm(E, E)
    return E


def _step(U, L, beta, theta, eps, seed, step, k_ref=0.0):
    X = _drift(U, L, beta, theta)
    X = X - _tr(X)[..., None, None] / 3.0 * torch.eye(3, dtype=X.dtype, device=X.device)
    if k_ref > 0:
        eps = eps * min(1.0, k_ref / math.sqrt(2.0 * float(X.abs().square().sum((-1, -2)).max())))
    V = U.shape[0]
    site = torch.arange(V, device=U.device).repeat_interleave(4)
    mu = torch.arange(4, device=U.device).repeat(V)
    eta = math.sqrt(2.0) * _normals(seed, step, site, mu, 4).reshape(V, 4, 8)
    U = _mm(_expm(2.0 * eps * X + 1j * math.sqrt(eps) * _hermitian(eta)), U)
    return U * torch.pow(_det(U), -1.0 / 3.0)[..., None, None]


def _gradient(U, L):
    """f_ax = 2 Tr[lambda_a sum_mu (U U^+ - U^+_{x-mu} U_{x-mu})], shape [site][8]."""
    G = 0
    for mu in range(4):
        u = U[:, mu]
        h = u.conj().transpose(-1, -2)
        G = G + _mm(u, h) - _hop(_mm(h, u), L, mu, -1)
    r3 = 1.0 / math.sqrt(3.0)
    g = lambda i, j: G[:, i, j]  # noqa: E731
    f = [4 * g(0, 1).real, -4 * g(0, 1).imag, 2 * (g(0, 0) - g(1, 1)).real, 4 * g(0, 2).real, -4 * g(0, 2).imag,
         4 * g(1, 2).real, -4 * g(1, 2).imag, 2 * r3 * (g(0, 0) + g(1, 1) - 2 * g(2, 2)).real]
    return torch.stack(f, -1)


def _cool(U, L, cp, forced):
    """Cooling sweeps with the adaptive strength and the stop rule; returns links and sweeps."""
    k, prev = 0, 0.0
    while True:
        f = _gradient(U, L)
        un = float(U.abs().square().sum()) / (12.0 * U.shape[0])
        D = {cl.CL_D0: 1.0, cl.CL_D1: un}.get(cp.mode)
        D = float(f.abs().mean()) if D is None else D
        if forced >= 0:
            stop = k >= forced
        else:
            stop = k >= cp.n_max or un - 1 < cp.d_floor or (k and prev - un < cp.tol_rel * (prev - 1))
        if stop or D < cp.d_guard:
            return U, k
        Om, Omi = (_expm(_hermitian(s * cp.eps * cp.alpha / D * f)) for s in (-1.0, 1.0))
        U = torch.stack([_mm(_mm(Om, U[:, mu]), _hop(Omi, L, mu, 1)) for mu in range(4)], 1)
        k, prev = k + 1, un


def _stored(case, U):
    return U.to(torch.complex64).to(torch.complex128) if case["form"] == "fp32" else U


def exact(case, seed):
    kind = case["kind"]
    if kind == "pchain":
        return _exact_chains(case, seed)
    real = lambda U: torch.view_as_real(U.contiguous())  # noqa: E731
    if kind == "batch":
        out = []
        for m in _members(case, seed):
            U = _stored(case, _links(m["L"], seed, m["tag"]))
            for n in range(case["steps"]):
                U = _step(U, m["L"], m["beta"], m["theta"], case["eps"], m["seed"], n, K_REF)
                U, _ = _cool(U, m["L"], _served_cool(case["eps"]), -1)
            out.append(real(U))
        return {"links": out}
    L = _shape(case)
    U = _stored(case, _links(L, seed))
    if kind == "obs":
        return {"obs": _measure(U, L, case["beta"], case["theta"])}
    if kind == "cool":
        U, k = _cool(U, L, _cool_params(case, forced=False), -1)
        return {"links": real(U), "sweeps": k}
    for n in range(case["steps"]):
        if kind == "replay":
            U = _step(U, L, case["beta"], case["theta"], case["eps"], int(seed) + 12345, n, K_REF)
            U, _ = _cool(U, L, _served_cool(case["eps"]), -1)
        else:
            U = _step(U, L, case["beta"], case["theta"], case["eps"], int(seed) + 12345, n)
            U, k = _cool(U, L, _cool_params(case), case["sweeps"])
    if kind == "replay":
        return {"links": real(U)}
    if kind == "host":
        return {"links": real(U).cpu(), "obs": _measure(U, L, case["beta"], case["theta"])}
    return {"links": real(U), "obs": _measure(U, L, case["beta"], case["theta"]), "sweeps": k}


# ------------------------------------------------------ SU(2) Polyakov chains
def _chain_links(case, seed):
    """Unit quaternions near 1 with a small non-unitary part, det = 1: [chain][link][2][2]."""
    rng = np.random.default_rng([int(seed), 6])
    a = 0.3 * rng.normal(size=(case["chains"], case["links"], 3)) + 0.03j * rng.normal(size=(case["chains"], case["links"], 3))
    return _exp2(torch.from_numpy(1j * a)).numpy()


def _exp2(a):
    """exp(sum_a a_a sigma_a) = cosh r + (sinh r / r) a.sigma with r^2 = a.a."""
    r = torch.sqrt((a * a).sum(-1))
    sh = torch.where(r.abs() < 1e-9, torch.ones_like(r), torch.sinh(r) / torch.where(r.abs() < 1e-9, torch.ones_like(r), r))
    c, b = torch.cosh(r), a * sh[..., None]
    return torch.stack([torch.stack([c + b[..., 2], b[..., 0] - 1j * b[..., 1]], -1),
                        torch.stack([b[..., 0] + 1j * b[..., 1], c - b[..., 2]], -1)], -2)


def _sigma(m):
    """Tr(sigma_a m)."""
    return torch.stack([m[..., 0, 1] + m[..., 1, 0], 1j * (m[..., 0, 1] - m[..., 1, 0]), m[..., 0, 0] - m[..., 1, 1]], -1)


def _exact_chains(case, seed):
    rng = np.random.default_rng([int(seed), 5])
    n, N, eps = case["chains"], case["links"], case["eps"]
    beta = torch.from_numpy(rng.uniform(0.5, 1.5, n) + 1j * rng.uniform(-0.5, 0.5, n))
    seeds = torch.from_numpy(rng.integers(1 << 40, size=n))
    U = torch.from_numpy(_chain_links(case, seed))
    sweeps = torch.zeros(n, dtype=torch.int64)
    for step in range(case["steps"]):
        pre, suf = [torch.eye(2, dtype=U.dtype).expand(n, 2, 2)], [torch.eye(2, dtype=U.dtype).expand(n, 2, 2)]
        for k in range(N):
            pre.append(pre[-1] @ U[:, k])
            suf.append(U[:, N - 1 - k] @ suf[-1])
        W = torch.stack([suf[N - k] @ pre[k] for k in range(N)], 1)  # the chain cut open at link k
        K = 0.5j * beta[:, None, None] * _sigma(W)  # K_a = -D_a S = (i beta / 2) Tr(sigma_a W_k)
        site = torch.arange(N).expand(n, N)
        eta = _normals(seeds[:, None].expand(n, N), step, site, 3 << 8, 2)[..., :3] * math.sqrt(2.0)
        U = _exp2(1j * (eps * K + math.sqrt(eps) * eta)) @ U
        U = U / torch.sqrt(torch.linalg.det(U))[..., None, None]
        sweeps = torch.zeros(n, dtype=torch.int64)
        prev, live = torch.zeros(n, dtype=torch.float64), torch.ones(n, dtype=torch.bool)
        for k in range(case["sweeps"] + 1):
            un = U.abs().square().sum((-1, -2)).mean(-1) / 2.0
            live = live & (un >= 1.0) & (k < case["sweeps"])
            if k:
                live = live & ~(prev - un < 0.01 * (prev - 1))
            h = U.conj().transpose(-1, -2)
            f = 2.0 * _sigma(U @ h - torch.roll(h @ U, 1, 1)).real
            a = torch.where(live, -eps / un, torch.zeros_like(un))[:, None, None] * f + 0j
            U = _exp2(a) @ U @ torch.roll(_exp2(-a), -1, 1)
            sweeps += live
            prev = un
    P = U[:, 0]
    for k in range(1, N):
        P = P @ U[:, k]
    tr = 0.5 * (P[:, 0, 0] + P[:, 1, 1])
    un = U.abs().square().sum((-1, -2)).mean(-1) / 2.0
    return {"links": torch.view_as_real(U.contiguous()).reshape(n, N, 2, 4), "traces": torch.stack([tr.real, tr.imag, un], -1),
            "sweeps": sweeps}
