"""Performance cases: what a user of this package evaluates, through its public entry points.

A case is a dict of plain values.  ``kind`` selects the entry point and the input:

  free       Plan.eval on a free-space cloud (``cloud``: ball, plummer or jittered lattice)
  periodic   Plan.eval on a lattice of the periodic cube [0, 2 pi)^3 (``field``: taylor_green
             or spectrum)
  strengths  Plan.eval_strengths: new strengths on the tree a full evaluation left behind
  targets    Plan.eval_targets: the velocity of one cloud at points that are not particles
  batch      Plan.eval_batch: many independent free-space problems in one call
  direct     direct: all pairs of a cloud

Sizes and parameters are those of the package's workloads: problems of 1e3 to 1e6 blobs with
expansion orders 4, 8 and 12 at theta = 0.5 (ball and Plummer clouds; sigma = 1.5 mean spacings),
the 4096-blob jittered lattice (p = 6), periodic lattices up to 128^3 at p = 10, theta = 0.4
(sigma = 1.2 spacings).  Inputs are drawn on the GPU from the seed alone; the plan is what a
program keeps between calls.
"""
import math

import numpy as np
import torch

from paper_1106_5273_gb300 import (FMM_OUT_STRETCHING, FMM_OUT_STRETCHING_TRANSPOSE, FMM_OUT_VELOCITY,
                                   FMM_SIGMA_MIXED, Params, Plan, direct)

TWO_PI = 2.0 * math.pi
PLUMMER_A = 0.1
EXACT_PAIRS = 1.6e10  # pairs that the FP64 reference sums in a few seconds


def listed():
    return [
        # the smallest problem of a batch, sent alone: launches and host round trips are all of it
        dict(name="ball_1000", kind="free", cloud="ball", n=1000, p=4, theta=0.5, ncrit=64, out="both", sigma="one"),
        # the accuracy workload: 16^3 jittered lattice, small leaves
        dict(name="lattice_4096", kind="free", cloud="lattice", n=4096, p=6, theta=0.5, ncrit=32, out="both",
             sigma="one"),
        # an ordinary clustered request at the middle order, a ragged size
        dict(name="plummer_30011", kind="free", cloud="plummer", n=30011, p=8, theta=0.5, ncrit=64, out="both",
             sigma="one"),
        # a uniform cloud with the conserving (transpose) stretching scheme
        dict(name="ball_100003_transpose", kind="free", cloud="ball", n=100003, p=8, theta=0.5, ncrit=64,
             out="transpose", sigma="one"),
        # core spreading leaves every blob its own core width
        dict(name="ball_60000_widths", kind="free", cloud="ball", n=60000, p=4, theta=0.5, ncrit=64, out="both",
             sigma="each"),
        # the largest problem of a batch, at its highest order: a deep adaptive tree
        dict(name="plummer_1m_p12", kind="free", cloud="plummer", n=1000000, p=12, theta=0.5, ncrit=64, out="both",
             sigma="one"),
        # the headline workload: 2,097,152 blobs, periodic
        dict(name="taylor_green_128", kind="periodic", field="taylor_green", side=128, p=10, theta=0.4, ncrit=64,
             images=3, out="both"),
        # a periodic turbulence request of odd side
        dict(name="spectrum_61", kind="periodic", field="spectrum", side=61, p=8, theta=0.5, ncrit=64, images=5,
             out="both"),
        # re-initialisation puts the blobs back on their lattice: only the strengths are new
        dict(name="strengths_64", kind="strengths", field="spectrum", side=64, p=10, theta=0.4, ncrit=64, images=3,
             out="both"),
        # a velocity field sampled on points of its own
        dict(name="targets_60k_50k", kind="targets", cloud="plummer", n=60001, nt=50021, p=8, theta=0.5, ncrit=64),
        # independent problems of mixed size in one call (leaf size as the tuner picks it for batches)
        dict(name="batch_32", kind="batch", nprob=32, nmin=1000, nmax=60000, mix=7, p=8, theta=0.5, ncrit=192),
        # the all-pairs sum that accuracy is checked against
        dict(name="direct_20000", kind="direct", cloud="ball", n=20000, sigma="one"),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("free", "free", "free", "periodic", "strengths", "targets", "batch", "direct"))
    p = rng.choice((4, 8, 12))
    if kind == "free":
        cloud = rng.choice(("ball", "plummer"))
        return dict(kind=kind, cloud=cloud, n=_log_uniform(rng, 1000, 400000), p=p, theta=0.5,
                    ncrit=rng.choice((32, 64, 64, 128)), out=rng.choice(("both", "both", "velocity", "transpose")),
                    sigma=rng.choice(("one", "one", "each", "mixed")))
    if kind in ("periodic", "strengths"):
        p = rng.choice((4, 8, 10, 10, 12))
        return dict(kind=kind, field=rng.choice(("taylor_green", "spectrum")), side=_log_uniform(rng, 16, 100), p=p,
                    theta=rng.choice((0.4, 0.5)), ncrit=64, images=rng.choice((3, 5)),
                    out=rng.choice(("both", "both", "velocity")))
    if kind == "targets":
        return dict(kind=kind, cloud=rng.choice(("ball", "plummer")), n=_log_uniform(rng, 2000, 200000),
                    nt=_log_uniform(rng, 1000, 200000), p=p, theta=0.5, ncrit=64)
    if kind == "batch":
        return dict(kind=kind, nprob=_log_uniform(rng, 2, 64), nmin=1000, nmax=_log_uniform(rng, 4000, 60000),
                    mix=rng.randrange(1 << 20), p=p, theta=0.5, ncrit=rng.choice((64, 128, 192)))
    return dict(kind=kind, cloud="ball", n=_log_uniform(rng, 500, 20000), sigma=rng.choice(("one", "each")))


# ---------------------------------------------------------------- inputs

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _normal(n, g):
    return torch.randn((n, 3), generator=g, device="cuda", dtype=torch.float64)


def _uniform(shape, g):
    return torch.rand(shape, generator=g, device="cuda", dtype=torch.float64)


def _width(cloud, n):
    """Core width: 1.5 mean spacings (of the unit ball, or inside a Plummer cloud's half-mass radius)."""
    if cloud == "plummer":
        rh = PLUMMER_A / math.sqrt(2.0 ** (2.0 / 3.0) - 1.0)
        return 1.5 * (4.0 / 3.0 * math.pi * rh ** 3 / max(n / 2.0, 1.0)) ** (1.0 / 3.0)
    if cloud == "lattice":
        return 1.5 / round(n ** (1.0 / 3.0))
    return 1.5 * (4.0 / 3.0 * math.pi / max(n, 1)) ** (1.0 / 3.0)


def _cloud(cloud, n, g):
    """Positions and Gaussian strengths (float32, CUDA) of a free-space cloud."""
    if cloud == "lattice":
        m = round(n ** (1.0 / 3.0))
        pos = _lattice(m, 1.0) + (_uniform((m ** 3, 3), g) - 0.5) * (0.5 / m)
        n = m ** 3
    else:
        v = _normal(n, g)
        v = v / v.norm(dim=1, keepdim=True)
        x = _uniform((n, 1), g)
        if cloud == "plummer":
            r = PLUMMER_A / torch.sqrt((0.999 * x).clamp_min(1e-12) ** (-2.0 / 3.0) - 1.0)
        else:
            r = x ** (1.0 / 3.0)
        pos = v * r
    return pos.float().contiguous(), _normal(n, g).float().contiguous()


def _widths(cloud, n, g):
    """One core width per blob, within a factor of two of each other."""
    return (_width(cloud, n) * (0.7 + 0.6 * _uniform((n,), g))).float().contiguous()


def _lattice(m, length):
    i = (torch.arange(m, device="cuda", dtype=torch.float64) + 0.5) * (length / m)
    return torch.stack(torch.meshgrid(i, i, i, indexing="ij"), -1).reshape(-1, 3)


def _taylor_green(m, seed):
    """(u, grad u) of a Taylor-Green field of random phase and amplitude at the lattice points, and its
    vorticity: u = a (sin X cos Y cos Z, -cos X sin Y cos Z, 0), X = x + phase."""
    rng = np.random.default_rng(seed)
    ph = torch.tensor(rng.uniform(0, TWO_PI, 3), device="cuda")
    amp = float(rng.uniform(0.5, 2.0))
    x = _lattice(m, TWO_PI).float().double() + ph
    s, c = torch.sin(x), torch.cos(x)
    sx, sy, sz, cx, cy, cz = s[:, 0], s[:, 1], s[:, 2], c[:, 0], c[:, 1], c[:, 2]
    zero = torch.zeros_like(sx)
    u = amp * torch.stack([sx * cy * cz, -cx * sy * cz, zero], 1)
    w = amp * torch.stack([-cx * sy * sz, -sx * cy * sz, 2.0 * sx * sy * cz], 1)
    grad = amp * torch.stack([torch.stack([cx * cy * cz, -sx * sy * cz, -sx * cy * sz], 1),
                              torch.stack([sx * sy * cz, -cx * cy * cz, cx * sy * sz], 1),
                              torch.stack([zero, zero, zero], 1)], 1)  # grad[i, a, b] = d u_a / d x_b
    return w, u, grad, 3.0


def _spectrum(m, seed, smooth=0.0, want_field=False):
    """Random-phase solenoidal field on the lattice, E(k) ~ k^4 exp(-2 (k/4)^2), |k| <= min(m/2 - 1, 20),
    u_rms = 1: its vorticity, and (want_field) u and grad u smoothed by exp(-smooth^2 k^2 / 2)."""
    g = _gen(seed)
    kmax = min(m // 2 - 1, 20)
    k1 = torch.fft.fftfreq(m, 1.0 / m, device="cuda", dtype=torch.float64)
    k = torch.stack(torch.meshgrid(k1, k1, k1, indexing="ij"), -1)
    k2 = (k * k).sum(-1)
    keep = (k2 > 0) & (k2 <= kmax * kmax)
    k2s = torch.where(keep, k2, torch.ones_like(k2))
    # the spectrum of a real white field is that of a real field whatever the phases are
    white = torch.fft.fftn(torch.randn((m, m, m, 3), generator=g, device="cuda", dtype=torch.float64), dim=(0, 1, 2))
    white = white - (white * k).sum(-1, keepdim=True) * k / k2s[..., None]
    uh = white * (torch.where(keep, k2s, torch.zeros_like(k2s)).sqrt() * torch.exp(-k2s / 16.0))[..., None]
    u = torch.fft.ifftn(uh, dim=(0, 1, 2)).real
    uh = uh / u.pow(2).sum(-1).mean().sqrt()

    def back(f):
        return torch.fft.ifftn(f, dim=(0, 1, 2)).real.reshape(-1, f.shape[-1])

    w = back(1j * torch.cross(k.to(uh.dtype), uh, dim=-1))
    if not want_field:
        return w, None, None
    us = uh * torch.exp(-0.5 * smooth * smooth * k2)[..., None]
    grad = torch.stack([back(1j * k[..., b:b + 1] * us) for b in range(3)], -1)
    return w, back(us), grad


def _periodic_input(case, seed, want_field=False):
    m = case["side"]
    h = TWO_PI / m
    sigma = float(np.float32(1.2 * h))
    pos = _lattice(m, TWO_PI).float().contiguous()
    if case["field"] == "taylor_green":
        w, u, grad, k2 = _taylor_green(m, seed)
        damp = math.exp(-0.5 * sigma * sigma * k2)
        u, grad = u * damp, grad * damp
    else:
        w, u, grad = _spectrum(m, seed, sigma, want_field)
    return pos, (w * h ** 3).float().contiguous(), sigma, u, grad


def _sizes(case):
    rng = np.random.default_rng(case["mix"])
    return [int(v) for v in np.exp(rng.uniform(math.log(case["nmin"]), math.log(case["nmax"]), case["nprob"]))]


def _batch_clouds(case, seed):
    g = _gen(seed)
    rng = np.random.default_rng(case["mix"] + 1)
    kinds = [("ball", "plummer")[int(v)] for v in rng.integers(0, 2, case["nprob"])]
    sizes = _sizes(case)
    return [_cloud(c, n, g) for c, n in zip(kinds, sizes)], [float(np.float32(_width(c, n)))
                                                            for c, n in zip(kinds, sizes)], sizes


def _free_input(case, seed):
    """(pos, gamma, per-blob widths or None, width) of a free or direct case."""
    g = _gen(seed)
    pos, gam = _cloud(case["cloud"], case["n"], g)
    if case["sigma"] == "one":
        return pos, gam, None, float(np.float32(_width(case["cloud"], case["n"])))
    return pos, gam, _widths(case["cloud"], case["n"], g), 0.0


# ---------------------------------------------------------------- the framework's calls

def _params(case, **kw):
    if case.get("out") == "transpose":
        kw["outputs"] = FMM_OUT_VELOCITY | FMM_OUT_STRETCHING_TRANSPOSE
    elif case.get("out") == "both":
        kw["outputs"] = FMM_OUT_VELOCITY | FMM_OUT_STRETCHING
    if case.get("sigma") == "mixed":
        kw["sigma_rule"] = FMM_SIGMA_MIXED
    if "images" in case:
        kw.update(periodic=1, box_min=(0.0, 0.0, 0.0), box_len=TWO_PI, images=case["images"])
    return Params.default(p=case["p"], theta=case["theta"], ncrit=case["ncrit"], **kw)


def prepare(case, seed):
    kind = case["kind"]
    st = dict(kind=kind, stretching=case.get("out") != "velocity")
    if kind in ("free", "direct"):
        st["pos"], st["gamma"], st["sigma"], st["width"] = _free_input(case, seed)
        if kind == "free":
            st["plan"] = Plan(st["pos"].shape[0], _params(case))
    elif kind in ("periodic", "strengths"):
        st["pos"], st["gamma"], st["width"], _, _ = _periodic_input(case, seed)
        st["plan"] = Plan(st["pos"].shape[0], _params(case))
        if kind == "strengths":  # the tree comes from an evaluation with other strengths
            st["plan"].eval(st["pos"], st["gamma"].roll(1, 0).contiguous(), sigma_uniform=st["width"],
                            stretching=st["stretching"])
    elif kind == "targets":
        g = _gen(seed)
        st["pos"], st["gamma"] = _cloud(case["cloud"], case["n"], g)
        st["tgt"] = _cloud(case["cloud"], case["nt"], g)[0]
        st["width"] = float(np.float32(_width(case["cloud"], case["n"])))
        st["plan"] = Plan(case["n"] + case["nt"], _params(case))
    else:
        clouds, widths, sizes = _batch_clouds(case, seed)
        st["pos"] = torch.cat([c[0] for c in clouds]).contiguous()
        st["gamma"] = torch.cat([c[1] for c in clouds]).contiguous()
        st["offsets"] = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
        st["widths"] = np.asarray(widths, np.float32)
        st["plan"] = Plan(int(st["offsets"][-1]), _params(case))
    return st


def run(st):
    kind = st["kind"]
    if kind in ("free", "periodic"):
        u, s = st["plan"].eval(st["pos"], st["gamma"], sigma=st.get("sigma"), sigma_uniform=st["width"],
                               stretching=st["stretching"])
    elif kind == "strengths":
        u, s = st["plan"].eval_strengths(st["gamma"], stretching=st["stretching"])
    elif kind == "targets":
        u, s = st["plan"].eval_targets(st["pos"], st["gamma"], st["tgt"], sigma_uniform=st["width"]), None
    elif kind == "batch":
        u, s = st["plan"].eval_batch(st["offsets"], st["pos"], st["gamma"], sigma_prob=st["widths"])
    else:
        u, s = direct(st["pos"], st["gamma"], sigma=st["sigma"], sigma_uniform=st["width"])
    return dict(u=u) if s is None else dict(u=u, s=s)


def work(case):
    """Bytes: inputs once, outputs once.  Flops: the pairs that only a pairwise sum can give (those
    within 5 core widths, where the kernel is regularised; all of them for the direct sum) at the
    singular kernel's flops per pair, and the terms of one multipole and one local expansion per blob."""
    kind = case["kind"]
    both = case.get("out") != "velocity" and kind != "targets"
    if kind == "batch":
        sizes, ratio = _sizes(case), 1.5
    elif kind in ("periodic", "strengths"):
        sizes, ratio = [case["side"] ** 3], 1.2
    else:
        sizes, ratio = [case["n"]], 1.5
    per_pair = 41.0 if both else 23.0
    near = 4.0 / 3.0 * math.pi * (5.0 * ratio) ** 3
    nbytes = flops = 0.0
    for n in sizes:
        nt = case["nt"] if kind == "targets" else n
        pairs = float(n) * (n - 1) if kind == "direct" else float(nt) * min(near, n)
        flops += per_pair * pairs + (n + nt) * 8.0 * case.get("p", 0) ** 2
        nbytes += 24.0 * n + (12.0 * nt if kind == "targets" else 0.0) + (24.0 if both else 12.0) * nt
        if case.get("sigma") in ("each", "mixed"):
            nbytes += 4.0 * n
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------- the same in FP64, without the package

def _pair_sum(tgt, src, gam, sig, tgam=None, tsig=None, transpose=False, same=True):
    """The FP64 sum over all pairs: u_i = (1/4 pi) sum_j S (gamma_j x d), and with the targets' strengths
    tgam the stretching of either scheme; S = g/r^3, T = S'(r)/r, g = erf(rho/sqrt 2) - sqrt(2/pi) rho
    exp(-rho^2/2); sig per source, or mixed with tsig.  The sums over j are matrix products."""
    x, y, g = tgt.double(), src.double(), gam.double()
    k = torch.linalg.cross(g, y)
    rhs = torch.cat([g, k], 1)  # sum S gamma_j, sum S gamma_j x x_j
    c = math.sqrt(2.0 / math.pi)
    nt, ns = x.shape[0], y.shape[0]
    u = torch.empty((nt, 3), device=x.device, dtype=torch.float64)
    s = None if tgam is None else torch.empty_like(u)
    block = max(1, int(3e7 // max(ns, 1)))
    for a in range(0, nt, block):
        b = min(nt, a + block)
        xi = x[a:b]
        r2 = torch.zeros((b - a, ns), device=x.device, dtype=torch.float64)
        for q in range(3):
            r2 += (xi[:, q:q + 1] - y[None, :, q]) ** 2
        if tsig is None:
            inv = (1.0 / sig.double())[None, :] if torch.is_tensor(sig) else 1.0 / float(sig)
        else:
            inv = torch.rsqrt(0.5 * (tsig[a:b].double()[:, None] ** 2 + sig.double()[None, :] ** 2))
        t2 = r2 * inv * inv
        rho = t2.sqrt()
        ex = torch.exp(-0.5 * t2)
        G = torch.special.erf(rho * math.sqrt(0.5)) - c * rho * ex
        small = t2 < 1e-3
        S = torch.where(small, c * inv ** 3 * (1.0 / 3.0 - t2 / 10.0 + t2 * t2 / 56.0 - t2 ** 3 / 432.0),
                        G / (r2 * r2.sqrt()))
        if same:
            S[torch.arange(b - a, device=x.device), torch.arange(a, b, device=x.device)] = 0.0
        AB = S @ rhs
        A = AB[:, :3]
        u[a:b] = torch.linalg.cross(A, xi) - AB[:, 3:]
        if s is None:
            continue
        T = torch.where(small, c * inv ** 5 * (-1.0 / 5.0 + t2 / 14.0 - t2 * t2 / 72.0 + t2 ** 3 / 528.0),
                        (c * ex * inv ** 3 - 3.0 * S) / r2)
        if same:
            T[torch.arange(b - a, device=x.device), torch.arange(a, b, device=x.device)] = 0.0
        gi = tgam[a:b].double()
        if transpose:  # S (gamma_i x gamma_j) + T (gamma_i . (gamma_j x d)) d, gamma_j x d = gamma_j x x_i - k_j
            T *= torch.linalg.cross(xi, gi) @ g.T - gi @ k.T
            s[a:b] = torch.linalg.cross(gi, A) + T.sum(1, keepdim=True) * xi - T @ y
        else:  # S (gamma_j x gamma_i) + T (gamma_i . d)(gamma_j x d)
            T *= (gi * xi).sum(1, keepdim=True) - gi @ y.T
            CD = T @ rhs
            s[a:b] = torch.linalg.cross(A, gi) + torch.linalg.cross(CD[:, :3], xi) - CD[:, 3:]
    f = 1.0 / (4.0 * math.pi)
    return u * f, None if s is None else s * f


def exact(case, seed):
    kind = case["kind"]
    both = case.get("out") != "velocity"
    if kind in ("periodic", "strengths"):
        pos, gam, _, u, grad = _periodic_input(case, seed, want_field=True)
        s = torch.einsum("iab,ib->ia", grad, gam.double())
        return dict(u=u, s=s) if both else dict(u=u)
    if kind == "targets":
        if float(case["n"]) * case["nt"] > EXACT_PAIRS:
            return None
        g = _gen(seed)
        pos, gam = _cloud(case["cloud"], case["n"], g)
        tgt = _cloud(case["cloud"], case["nt"], g)[0]
        return dict(u=_pair_sum(tgt, pos, gam, float(np.float32(_width(case["cloud"], case["n"]))), same=False)[0])
    if kind == "batch":
        if sum(float(n) * n for n in _sizes(case)) > EXACT_PAIRS:
            return None
        clouds, widths, _ = _batch_clouds(case, seed)
        got = [_pair_sum(p, p, g, w, tgam=g) for (p, g), w in zip(clouds, widths)]
        return dict(u=torch.cat([v[0] for v in got]), s=torch.cat([v[1] for v in got]))
    if float(case["n"]) ** 2 > EXACT_PAIRS:
        return None
    pos, gam, sig, width = _free_input(case, seed)
    u, s = _pair_sum(pos, pos, gam, width if sig is None else sig, tgam=gam if both else None,
                     tsig=sig if case["sigma"] == "mixed" else None, transpose=case.get("out") == "transpose")
    return dict(u=u, s=s) if both else dict(u=u)
