"""The work that users of the framework have it do, as cases to be timed.

Each case is one call, or the few calls of one step, through the public entry
points of ``paper_1312_1128_gb300``.  Inputs are drawn on the GPU from a seed.
The sizes are those of the repository's benchmark and tests, with small and
odd ones beside them; ``draw`` spreads over the same ranges.  ``exact`` gives
the untruncated sums in 64 bits by plain torch where that is quick enough.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1312_1128_gb300 as L

DEV = "cuda"
F64 = torch.float64
F32 = torch.float32


def listed():
    return [
        # a source-plane look-up: a few scattered rays through a small lens that
        # is already built (the smoke test's size); launches and latency
        dict(name="rays_4k_1000", kind="rays", n=4001, rays=1000, theta=0.3, group=0, alpha_only=False, dtype="f32"),
        # a map of a small simulated halo, lens built and shot once, at the
        # paper's recommended opening angle; odd sizes
        dict(name="map_20k_97sq", kind="map", n=20011, grid=97, theta=0.1, group=0, alpha_only=False, q=3.0),
        # the headline: a 1e6-particle halo built and mapped on 2048^2 rays, the
        # group size as the autotuner leaves it on this lens
        dict(name="map_1e6_2048sq", kind="map", n=1_000_000, grid=2048, theta=0.3, group=64, alpha_only=False, q=3.0),
        # one round of an adaptive refinement: 256 uneven batches through a
        # prebuilt lens of 1,000 NFW halos and 1e6 stars
        dict(name="batches_256", kind="batches", n=1_000_000, halos=1000, batches=256, nmin=1000, nmax=1_000_000,
             theta=0.3, group=64),
        # a microlensing magnification map: 1e7 stars and an SIS, 4096^2 rays
        # over a 1e-6-wide patch, group size as autotuned
        dict(name="stars_1e7_4096sq", kind="stars", n=10_000_000, grid=4096, theta=0.1, group=128, width=1e-6),
        # one step of a lens fit (build, forward, adjoint): the benchmark's size
        dict(name="fit_1e5_1000sq", kind="fit", n=100_000, grid=1000, theta=0.3),
        # one step of a small fit, as an optimiser repeats it thousands of times
        dict(name="fit_5k_101sq", kind="fit", n=5003, grid=101, theta=0.3),
        # time delays: the potential and deflection of a built lens on a map
        dict(name="potential_3e5_1000sq", kind="potential", n=300_000, grid=1000, theta=0.3, group=0),
        # the FP64 reference forms: direct sum and tree of 2,000 point masses
        dict(name="fp64_2000_64sq", kind="fp64", n=2000, grid=64, theta=0.1),
        # the smoothing lengths of a 1e6-particle snapshot (32nd neighbour)
        dict(name="smoothing_1e6_k32", kind="smoothing", n=1_000_000, k=32),
        # refinement of a map's cells by the linear lens equation, by thirds
        dict(name="refine_2048sq_k3", kind="refine", grid=2048, k=3, mode=0, alpha="f64"),
        # image finding: the SIS test's 62 sources in one call (FP64)
        dict(name="images_sis_62", kind="images", sources=21, grid=64),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["rays", "map", "map", "batches", "stars", "stars", "fit", "fit", "potential", "fp64", "smoothing",
                       "refine", "images"])
    if kind == "rays":
        return dict(kind=kind, n=_log_int(rng, 500, 300_000), rays=_log_int(rng, 1, 200_000),
                    theta=rng.choice([0.1, 0.3, 0.5]), group=rng.choice([0, 0, 64, 128]),
                    alpha_only=rng.random() < 0.4, dtype=rng.choice(["f32", "f64"]))
    if kind == "map":
        return dict(kind=kind, n=_log_int(rng, 1000, 1_000_000), grid=_log_int(rng, 16, 1500),
                    theta=rng.choice([0.2, 0.3, 0.5]), group=rng.choice([0, 0, 64, 128]),
                    alpha_only=rng.random() < 0.3, q=rng.choice([2.5, 3.0, 3.0, 3.5]))
    if kind == "batches":
        return dict(kind=kind, n=_log_int(rng, 10_000, 1_000_000), halos=_log_int(rng, 10, 1000),
                    batches=_log_int(rng, 2, 256), nmin=_log_int(rng, 5, 1000), nmax=_log_int(rng, 2000, 300_000),
                    theta=rng.choice([0.1, 0.3]), group=rng.choice([0, 64, 128]))
    if kind == "stars":
        return dict(kind=kind, n=_log_int(rng, 10_000, 5_000_000), grid=_log_int(rng, 30, 2000),
                    theta=rng.choice([0.1, 0.2, 0.3]), group=rng.choice([0, 0, 64, 128]),
                    width=10.0 ** rng.uniform(-6.0, -1.0))
    if kind == "fit":
        return dict(kind=kind, n=_log_int(rng, 500, 100_000), grid=_log_int(rng, 20, 900),
                    theta=rng.choice([0.1, 0.3, 0.5]))
    if kind == "potential":
        return dict(kind=kind, n=_log_int(rng, 1000, 500_000), grid=_log_int(rng, 16, 1000),
                    theta=rng.choice([0.2, 0.3]), group=rng.choice([0, 64]))
    if kind == "fp64":
        return dict(kind=kind, n=_log_int(rng, 100, 20_000), grid=_log_int(rng, 8, 128), theta=rng.choice([0.1, 0.3]))
    if kind == "smoothing":
        return dict(kind=kind, n=_log_int(rng, 200, 1_000_000), k=rng.choice([1, 8, 16, 32, 32, 48, 64]))
    if kind == "refine":
        return dict(kind=kind, grid=_log_int(rng, 16, 1500), k=rng.choice([1, 3, 3, 5]), mode=rng.choice([0, 1]),
                    alpha=rng.choice(["f32", "f64"]))
    return dict(kind=kind, sources=rng.randrange(2, 22), grid=rng.choice([32, 64, 65, 100]))


# ------------------------------------------------------------------ inputs

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device=DEV, dtype=F64)


def _halo_positions(n, g, rs=0.1, rmax=1.0):
    """3D positions (n, 3) of an NFW density out to rmax, and the radii."""
    cdf = lambda x: torch.log1p(x) - x / (1 + x)  # noqa: E731
    top = rmax / rs
    target = _rand(g, n) * (math.log1p(top) - top / (1 + top))
    lo, hi = torch.zeros(n, device=DEV, dtype=F64), torch.full((n,), top, device=DEV, dtype=F64)
    for _ in range(50):
        mid = 0.5 * (lo + hi)
        below = cdf(mid) < target
        lo, hi = torch.where(below, mid, lo), torch.where(below, hi, mid)
    r = 0.5 * (lo + hi) * rs
    mu, phi = 2 * _rand(g, n) - 1, 2 * math.pi * _rand(g, n)
    s = torch.sqrt(1 - mu * mu)
    return torch.stack([r * s * torch.cos(phi), r * s * torch.sin(phi), r * mu], 1), r


def _halo_particles(n, g, k=32, sigma=None):
    """Projected equal-mass particles {x, y, m, r_sm}: r_sm as the distance to
    the k-th neighbour is distributed in the local density."""
    rs, rmax = 0.1, 1.0
    p, r = _halo_positions(n, g, rs, rmax)
    if sigma is None:
        top = rmax / rs
        x = torch.clamp(r / rs, min=1e-6)
        dens = n / (4 * math.pi * rs ** 3 * (math.log1p(top) - top / (1 + top))) / (x * (1 + x) ** 2)
        hits = torch.zeros(n, device=DEV, dtype=F64)
        for _ in range(k):
            hits -= torch.log(1 - _rand(g, n))
        sig = (3 * hits / (4 * math.pi * dens)) ** (1 / 3)
    else:
        sig = torch.full((n,), sigma, device=DEV, dtype=F64)
    return torch.stack([p[:, 0], p[:, 1], torch.full((n,), 1.0 / n, device=DEV, dtype=F64), sig], 1).to(F32)


def _grid(n, lo, hi, dtype=F32):
    c = lo + (torch.arange(n, device=DEV, dtype=F64) + 0.5) * ((hi - lo) / n)
    return (c.repeat(n).to(dtype), c.repeat_interleave(n).to(dtype))


def _star_masses(n, g, total):
    a = 1.0 - 2.35
    m = (0.1 ** a + _rand(g, n) * (1.0 - 0.1 ** a)) ** (1 / a)
    return m * (total / m.sum())


def _inputs(case, seed):
    """The arrays of a case, from the seed alone."""
    g, kind = _gen(seed), case["kind"]
    d = {}
    if kind in ("rays", "map", "potential"):
        d["parts"] = _halo_particles(case["n"], g)
        if kind == "rays":
            dt = F64 if case["dtype"] == "f64" else F32
            d["rx"], d["ry"] = ((1.6 * _rand(g, case["rays"]) - 0.8).to(dt) for _ in range(2))
        else:
            d["rx"], d["ry"] = _grid(case["grid"], -1.0, 1.0)
    elif kind == "batches":
        n, h, nb = case["n"], case["halos"], case["batches"]
        m = 10.0 ** (-4 + torch.randn(h, generator=g, device=DEV, dtype=F64))
        d["nfw"] = torch.stack([2 * _rand(g, h) - 1, 2 * _rand(g, h) - 1, m, 0.02 * (m / 1e-4) ** (1 / 3)], 1).to(F32)
        d["stars"] = torch.stack([0.295 + 0.01 * _rand(g, n), 0.195 + 0.01 * _rand(g, n),
                                  _star_masses(n, g, 0.5e-4 / math.pi), torch.zeros(n, device=DEV, dtype=F64)], 1).to(F32)
        # sizes spread over the logarithm of their range, levels over nine
        # refinements; which batch has which is the seed's
        h_rng = np.random.Generator(np.random.PCG64(seed))
        ratio = case["nmax"] / case["nmin"]
        sizes = np.array([int(case["nmin"] * ratio ** ((b + 0.5) / nb)) for b in range(nb)], np.int64)
        h_rng.shuffle(sizes)
        level = h_rng.permutation(np.arange(nb) % 9)
        d["offsets"] = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
        d["origins"] = np.stack([0.295 + 0.01 * h_rng.random(nb), 0.195 + 0.01 * h_rng.random(nb)], 1)
        t = torch.from_numpy(sizes).to(DEV)
        b = torch.repeat_interleave(torch.arange(nb, device=DEV), t)
        i = torch.arange(int(sizes.sum()), device=DEV) - torch.from_numpy(d["offsets"][:-1]).to(DEV)[b]
        side = torch.from_numpy(0.01 * 3.0 ** (-level.astype(np.float64))).to(DEV)[b]
        k = torch.from_numpy(np.ceil(np.sqrt(sizes)).astype(np.int64)).to(DEV)[b]
        cell = side / k
        d["rx"] = (((i % k) + _rand(g, i.numel())) * cell - 0.5 * side).to(F32)
        d["ry"] = (((i // k) + _rand(g, i.numel())) * cell - 0.5 * side).to(F32)
    elif kind == "stars":
        n, w = case["n"], case["width"]
        r, phi = torch.sqrt(_rand(g, n)), 2 * math.pi * _rand(g, n)
        d["stars"] = torch.stack([r * torch.cos(phi), r * torch.sin(phi), _star_masses(n, g, 0.5),
                                  torch.zeros(n, device=DEV, dtype=F64)], 1).to(F32)
        d["rx"], d["ry"] = _grid(case["grid"], -0.5 * w, 0.5 * w)
        d["origin"], d["r_e"] = (0.5, 0.0), 0.5
    elif kind == "fit":
        d["parts"] = _halo_particles(case["n"], g, sigma=0.01)
        d["rx"], d["ry"] = _grid(case["grid"], -1.0, 1.0)
        # the observed deflections: a cored isothermal sphere, which the
        # particles do not fit yet
        x, y = d["rx"].to(F64), d["ry"].to(F64)
        f = (0.6 + 0.2 * float(_rand(g, 1))) / torch.sqrt(x * x + y * y + 0.0025)
        d["target"] = torch.stack([f * x, f * y], 1).to(F32)
    elif kind == "fp64":
        n = case["n"]
        r, phi = torch.sqrt(_rand(g, n)), 2 * math.pi * _rand(g, n)
        d["points"] = torch.stack([r * torch.cos(phi), r * torch.sin(phi), torch.full((n,), 1.0 / n, device=DEV, dtype=F64),
                                   torch.zeros(n, device=DEV, dtype=F64)], 1).to(F32).to(F64)
        d["rx"], d["ry"] = _grid(case["grid"], -1.2, 1.2, F64)
    elif kind == "smoothing":
        d["xyz"] = _halo_positions(case["n"], g)[0].to(F32)
    elif kind == "refine":
        # a map of a field of cored halos, from their closed forms
        n, width = case["grid"], 0.03
        d["h"], d["x0"], d["y0"] = width / n, 0.3 - 0.5 * width + 0.5 * width / n, 0.2 - 0.5 * width + 0.5 * width / n
        x, y = _grid(n, -0.5 * width, 0.5 * width, F64)
        a1, a2, ka, g1, g2 = (torch.zeros(n * n, device=DEV, dtype=F64) for _ in range(5))
        for _ in range(24):
            u = _rand(g, 4).tolist()
            m, s2 = 10.0 ** (-7.0 + 1.5 * u[0]), (0.001 + 0.004 * u[1]) ** 2
            wx, wy = x - width * (u[2] - 0.5), y - width * (u[3] - 0.5)
            b = 1 / (wx * wx + wy * wy + s2)
            a1 += m * wx * b
            a2 += m * wy * b
            ka += m * s2 * b * b
            g1 -= m * (wx * wx - wy * wy) * b * b
            g2 -= 2 * m * wx * wy * b * b
        dt = F64 if case["alpha"] == "f64" else F32
        d["a1"], d["a2"], d["ka"], d["g1"], d["g2"] = a1.to(dt), a2.to(dt), ka.to(F32), g1.to(F32), g2.to(F32)
    elif kind == "images":
        # source centres 0.03, 0.13, ... Einstein radii from the lens, moved a
        # little by the seed (the number of images stays the same)
        rng = np.random.Generator(np.random.PCG64(seed))
        src = []
        for r in (0.1, 0.01, 1e-4):
            for b in range(case["sources"]):
                dist, phi = 0.1 * b + 0.03 + 0.002 * rng.random(), 0.05 * rng.random()
                if r > 1e-3 or b > 0:
                    src.append((dist * math.cos(phi), dist * math.sin(phi), r))
        d["sources"] = np.array(src)
    return d


class _State:
    def __init__(self, case, d):
        self.case = case
        self.__dict__.update(d)


def prepare(case, seed):
    s = _State(case, _inputs(case, seed))
    kind = case["kind"]
    # lenses that a user builds once and shoots many times
    if kind in ("rays", "potential"):
        s.lens = L.Lens([L.Species.gauss(s.parts, 3.0)], theta=case["theta"], group_rays=case["group"])
    elif kind == "batches":
        s.lens = L.Lens([L.Species.points(s.stars), L.Species.nfw(s.nfw, 3.0)], theta=case["theta"],
                        group_rays=case["group"])
        s.lens.reserve(int(s.offsets[-1]), case["batches"])
    elif kind == "fp64":
        s.lens = L.Lens([L.Species.points(s.points)], theta=case["theta"], precision="fp64")
    elif kind == "images":
        s.lens = L.Lens([], [L.Halo.sis(0.0, 0.0, 1.0)], theta=0.3, precision="fp64")
    elif kind == "fit":
        s.parts.requires_grad_(True)
    return s


def run(s):
    c = s.case
    kind = c["kind"]
    if kind == "rays":
        out = s.lens.shoot(s.rx, s.ry, flags=L.ALPHA_ONLY if c["alpha_only"] else 0)
        return [o for o in out if o is not None]
    if kind == "map":
        lens = L.Lens([L.Species.gauss(s.parts, c["q"])], theta=c["theta"], group_rays=c["group"])
        out = lens.shoot(s.rx, s.ry, flags=L.ALPHA_ONLY if c["alpha_only"] else 0)
        return [o for o in out if o is not None]
    if kind == "batches":
        return s.lens.shoot_batches(s.offsets, s.origins, s.rx, s.ry)
    if kind == "stars":
        lens = L.Lens([L.Species.points(s.stars)], [L.Halo.sis(0.0, 0.0, s.r_e)], theta=c["theta"],
                      group_rays=c["group"])
        return lens.shoot(s.rx, s.ry, origin=s.origin)
    if kind == "fit":
        lens = L.Lens([L.Species.gauss(s.parts.detach(), 3.0)], theta=c["theta"])
        alpha = L.shoot(lens, s.rx, s.ry, species_data=[s.parts])
        loss = ((alpha - s.target) ** 2).sum()
        (grad,) = torch.autograd.grad(loss, [s.parts])
        return [alpha.detach(), loss.detach(), grad[:, 0], grad[:, 1], grad[:, 2], grad[:, 3]]
    if kind == "potential":
        return s.lens.potential(s.rx, s.ry)
    if kind == "fp64":
        return [s.lens.shoot(s.rx, s.ry, flags=L.DIRECT), s.lens.shoot(s.rx, s.ry)]
    if kind == "smoothing":
        return L.smoothing_lengths(s.xyz, c["k"])
    if kind == "refine":
        return L.refine_cells(s.x0, s.y0, s.h, c["grid"], c["grid"], s.a1, s.a2, s.ka, s.g1, s.g2, k=c["k"],
                              mode=c["mode"])
    images, _ = s.lens.find_images(s.sources, -10.0, -10.0, 20.0, n=c["grid"], max_cells=1 << 26, max_images=1024)
    return {key: np.array([im[key] for im in images]) for key in ("source", "n_cells", "area", "mu", "first")}


# -------------------------------------------------------------------- work

def work(case):
    """Each input read and each output written once.  Operations: what any
    method has to spend, some tens on each particle (its moments) and a
    hundred or so on each ray (its field); the direct sum's and the neighbour
    search's pairs in full."""
    kind = case["kind"]
    if kind in ("rays", "map", "potential", "stars", "batches", "fit"):
        n = case["n"]
        if kind == "rays":
            nr, rb = case["rays"], 16 if case["dtype"] == "f64" else 8
        elif kind == "batches":
            ratio, nb = case["nmax"] / case["nmin"], case["batches"]
            nr, rb = sum(int(case["nmin"] * ratio ** ((b + 0.5) / nb)) for b in range(nb)), 8
            n += case["halos"]
        else:
            nr, rb = case["grid"] ** 2, 8
        outs = 3 if kind == "potential" else 2 if kind == "fit" or case.get("alpha_only") else 5
        by = 16 * n + nr * (rb + 4 * outs)
        if kind == "fit":  # target and upstream gradient read, gradients written
            by += nr * 16 + 16 * n
        return {"bytes": by, "flops": 60 * n + 150 * nr * (2 if kind == "fit" else 1)}
    if kind == "fp64":
        n, nr = case["n"], case["grid"] ** 2
        return {"bytes": 32 * n + nr * (16 + 80), "flops": 22.0 * n * nr}
    if kind == "smoothing":
        return {"bytes": 16 * case["n"], "flops": 8.0 * case["n"] * 4 * case["k"]}
    if kind == "refine":
        n, k = case["grid"], case["k"]
        a = 8 if case["alpha"] == "f64" else 4
        return {"bytes": n * n * (2 * a + (12 if case["mode"] == 0 else 0)) + (n - 2) ** 2 * (1 + 16 + 16 * k * k),
                "flops": (n - 2) ** 2 * (20.0 + 8 * k * k)}
    # the new cells of the refinement, their key and field written and read
    cells = 230_000 * (3 * case["sources"] - 1)
    return {"bytes": cells * 32, "flops": cells * 40.0}


# ------------------------------------------------------------------- exact

def _circular(wx, wy, kb, ka, D):
    c2, s2 = wx * wx - wy * wy, 2 * wx * wy
    return kb * wx, kb * wy, ka, -D * c2, -D * s2


def _profile(kind, wx, wy, p, shape):
    """kb, kappa, D = (kb - kappa)/r^2 of particles p (n, 4) at separations w."""
    r2 = wx * wx + wy * wy
    m = p[:, 2][None]
    if kind == "point":
        inv = torch.where(r2 > 0, 1 / r2, 0.0)
        return m * inv, torch.zeros_like(r2), m * inv * inv
    if kind == "gauss":
        c = (0.5 / p[:, 3] ** 2)[None]
        u, top = r2 * c, 0.5 * shape * shape
        N = -math.expm1(-top)
        e, inv = torch.exp(-u), 1 / torch.clamp(r2, min=1e-300)
        inside, small = u < top, u < 1e-2
        h = torch.where(small, 1 - u / 2 * (1 - u / 3 * (1 - u / 4 * (1 - u / 5 * (1 - u / 6)))), -torch.expm1(-u) * inv / c)
        dh = torch.where(small, c * (1 / 2 - u / 3 + u * u / 8 - u ** 3 / 30 + u ** 4 / 144 - u ** 5 / 840), (h - e) * inv)
        mc = m * c / N
        return (torch.where(inside, mc * h, m * inv), torch.where(inside, mc * e, 0.0),
                torch.where(inside, mc * dh, m * inv * inv))
    rs = p[:, 3][None]
    x, X = torch.clamp(torch.sqrt(r2) / rs, min=1e-9), torch.tensor(shape, device=DEV, dtype=F64)

    def F(x):
        u = 1 - x * x
        t = torch.sqrt(u.abs())
        near = 1 + u / 3 + u * u / 5 + u ** 3 / 7 + u ** 4 / 9
        far = torch.where(u > 0, torch.log((1 + t) / x) / t, torch.atan(t) / t)
        return torch.where(u.abs() < 1e-3, near, far)

    f = F(x)
    u = 1 - x * x
    shape_f = torch.where(u.abs() < 1e-3, 1 / 3 + u / 5 + u * u / 7 + u ** 3 / 9, (f - 1) / torch.where(u == 0, 1.0, u))
    A = m / (torch.log(X / 2) + F(X))
    inside, inv = x < shape, torch.where(r2 > 0, 1 / r2, 0.0)
    kb = torch.where(inside, A * (torch.log(x / 2) + f) * inv, m * inv)
    ka = torch.where(inside, 0.5 * A * shape_f / (rs * rs), 0.0)
    return kb, ka, (kb - ka) * inv


_MAX_PAIRS = 4e9  # about ten seconds of 64-bit torch
_CHUNK = 1 << 24


def _direct(species, x, y):
    """Five sums over all particles of species [(kind, data, shape)]."""
    out = torch.zeros(5, x.numel(), device=DEV, dtype=F64)
    for kind, data, shape in species:
        p = data.detach().to(F64)
        step = max(1, _CHUNK // p.shape[0])
        for i in range(0, x.numel(), step):
            wx, wy = x[i:i + step, None] - p[None, :, 0], y[i:i + step, None] - p[None, :, 1]
            for q, v in enumerate(_circular(wx, wy, *_profile(kind, wx, wy, p, shape))):
                out[q, i:i + step] += v.sum(1)
    return list(out)


def _direct_potential(p, q, x, y):
    p, top = p.to(F64), 0.5 * q * q
    N = -math.expm1(-top)

    def ein(u):
        s, t = torch.zeros_like(u), torch.ones_like(u)
        for k in range(1, 45):
            t = t * (-u) / k
            s -= t / k
        return s

    a = _direct([("gauss", p, q)], x, y)
    psi = torch.zeros_like(x)
    m, sig = p[:, 2][None], p[:, 3][None]
    e_top = float(ein(torch.tensor(top, device=DEV, dtype=F64)))
    step = max(1, _CHUNK // p.shape[0])
    for i in range(0, x.numel(), step):
        wx, wy = x[i:i + step, None] - p[None, :, 0], y[i:i + step, None] - p[None, :, 1]
        r2 = wx * wx + wy * wy
        u = r2 / (2 * sig * sig)
        inner = m * torch.log(q * sig) - m / (2 * N) * (e_top - ein(torch.clamp(u, max=top)))
        psi[i:i + step] = torch.where(u < top, inner, 0.5 * m * torch.log(torch.clamp(r2, min=1e-300))).sum(1)
    return [psi, a[0], a[1]]


def exact(case, seed):
    kind = case["kind"]
    if kind == "images":
        return None
    if kind == "smoothing" and case["n"] > 40_000:
        return None
    if kind in ("rays", "map", "potential", "stars", "fit", "fp64"):
        nr = case["rays"] if kind == "rays" else case["grid"] ** 2
        if case["n"] * nr > _MAX_PAIRS / (4 if kind in ("potential", "fit") else 1):
            return None
    if kind == "batches":
        ratio, nb = case["nmax"] / case["nmin"], case["batches"]
        if (case["n"] + case["halos"]) * sum(int(case["nmin"] * ratio ** ((b + 0.5) / nb)) for b in range(nb)) > _MAX_PAIRS:
            return None
    d = _inputs(case, seed)
    if kind in ("rays", "map"):
        out = _direct([("gauss", d["parts"], case.get("q", 3.0))], d["rx"].to(F64), d["ry"].to(F64))
        return out[:2] if case["alpha_only"] else out
    if kind == "batches":
        b = np.repeat(np.arange(case["batches"]), np.diff(d["offsets"]))
        o = torch.from_numpy(d["origins"][b]).to(DEV)
        return _direct([("point", d["stars"], 0.0), ("nfw", d["nfw"], 3.0)], o[:, 0] + d["rx"].to(F64),
                       o[:, 1] + d["ry"].to(F64))
    if kind == "stars":
        x, y = d["origin"][0] + d["rx"].to(F64), d["origin"][1] + d["ry"].to(F64)
        r = torch.sqrt(x * x + y * y)
        sis = _circular(x, y, d["r_e"] / r, 0.5 * d["r_e"] / r, 0.5 * d["r_e"] / r ** 3)
        return [a + b for a, b in zip(_direct([("point", d["stars"], 0.0)], x, y), sis)]
    if kind == "fit":
        x, y, p = d["rx"].to(F64), d["ry"].to(F64), d["parts"].to(F64)
        a1, a2, *_ = _direct([("gauss", p, 3.0)], x, y)
        alpha = torch.stack([a1, a2], 1)
        res = alpha - d["target"].to(F64)
        G = 2 * res
        grad = torch.zeros(p.shape[0], 4, device=DEV, dtype=F64)
        step = max(1, _CHUNK // p.shape[0])
        for i in range(0, x.numel(), step):
            wx, wy = x[i:i + step, None] - p[None, :, 0], y[i:i + step, None] - p[None, :, 1]
            kb, ka, D = _profile("gauss", wx, wy, p, 3.0)
            g1, g2 = G[i:i + step, 0, None], G[i:i + step, 1, None]
            gw = g1 * wx + g2 * wy
            s1, s2 = -D * (wx * wx - wy * wy), -D * 2 * wx * wy
            grad[:, 0] -= (g1 * (ka + s1) + g2 * s2).sum(0)
            grad[:, 1] -= (g1 * s2 + g2 * (ka - s1)).sum(0)
            grad[:, 2] += (kb * gw).sum(0) / p[:, 2]
            grad[:, 3] -= (ka * gw).sum(0) * 2 / p[:, 3]
        return [alpha, (res * res).sum(), grad[:, 0], grad[:, 1], grad[:, 2], grad[:, 3]]
    if kind == "potential":
        return _direct_potential(d["parts"], 3.0, d["rx"].to(F64), d["ry"].to(F64))
    if kind == "fp64":
        out = _direct([("point", d["points"], 0.0)], d["rx"], d["ry"])
        return [out, out]
    if kind == "smoothing":
        p = d["xyz"].to(F64)
        step = max(1, _CHUNK // p.shape[0])
        r = [torch.topk(((p[i:i + step, None] - p[None]) ** 2).sum(2), case["k"] + 1, largest=False)[0][:, -1]
             for i in range(0, p.shape[0], step)]
        return torch.sqrt(torch.cat(r))
    # refine: the flags compare 32- or 64-bit inputs as they are; kappa and gamma mode only
    if case["mode"] == 1:
        return None
    n, k, h = case["grid"], case["k"], d["h"]
    mid = lambda t: t.view(n, n)[1:-1, 1:-1]  # noqa: E731
    diff = torch.zeros(n - 2, n - 2, device=DEV)
    for t in (d["ka"], d["g1"], d["g2"]):
        v = t.view(n, n)
        for w in (v[1:-1, 2:], v[2:, 1:-1], v[1:-1, :-2], v[:-2, 1:-1]):
            diff = torch.maximum(diff, (w - mid(t)).abs())
    flat = (diff <= torch.tensor(1e-4, device=DEV, dtype=F32)).reshape(-1)
    ka, g1, g2 = (mid(t).to(F64).reshape(-1) for t in (d["ka"], d["g1"], d["g2"]))
    a = torch.stack([1 - ka - g1, -g2, -g2, 1 - ka + g1], 1)
    i = torch.arange(1, n - 1, device=DEV, dtype=F64)
    yx = d["x0"] + i.repeat(n - 2) * h - mid(d["a1"]).to(F64).reshape(-1)
    yy = d["y0"] + i.repeat_interleave(n - 2) * h - mid(d["a2"]).to(F64).reshape(-1)
    o = (torch.arange(k, device=DEV, dtype=F64) - 0.5 * (k - 1)) * h / k
    da, db = o[None, None, :], o[None, :, None]
    y = torch.stack([yx[:, None, None] + a[:, 0, None, None] * da + a[:, 1, None, None] * db,
                     yy[:, None, None] + a[:, 2, None, None] * da + a[:, 3, None, None] * db], 3)
    return [None, a, torch.where(flat[:, None, None, None], y, float("nan"))]
