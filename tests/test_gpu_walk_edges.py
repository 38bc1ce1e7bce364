"""Edge cases of the walk's forms: rays at infinity, faint lenses."""
import numpy as np
import pytest

import lensgen
import oracle
from lens_testutil import comps_nfw, comps_points

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1312_1128_gb300 as L  # noqa: E402


def cu(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def shoot(species, dx, dy, walk="warp", theta=0.3):
    lens = L.Lens(species, theta=theta, group_rays=32, walk=walk)
    o = lens.shoot(cu(dx), cu(dy))
    lens.sync()
    got = np.stack([x.double().cpu().numpy() for x in o], axis=1)
    lens.close()
    return got


@pytest.mark.parametrize("kind", ["nfw", "points"])
def test_infinite_ray(kind):
    """A ray at infinity leaves the other rays of its group as they are: the
    form without expansions as the reference, 1e-6 of the sum of |terms| (the
    same terms in another order)."""
    g = lensgen.rng(7)
    if kind == "nfw":
        p, n = lensgen.nfw_test_halos(3000, 22, 0.3), 1000
        species, comps = [L.Species.nfw(cu(p), 3.0)], comps_nfw(p, 3.0)
    else:
        p, n = lensgen.point_disk(20000, 33), 16384 * 32 + 5  # (from 16,384 groups on: supergroups)
        species, comps = [L.Species.points(cu(p))], comps_points(p)
    dx, dy = (g.uniform(-0.9, 0.9, n).astype(np.float32) for _ in range(2))
    dx[[3, n // 2]], dy[n - 1] = (np.inf, -np.inf), np.inf
    got, ref = shoot(species, dx, dy), shoot(species, dx, dy, walk="pairs")
    fin = np.isfinite(dx) & np.isfinite(dy)
    assert np.isfinite(ref[fin]).all()
    assert np.isfinite(got[fin]).all()
    # (the rays that share a group with one at infinity are not known from
    # outside: all of a small call, a sample of a large one)
    idx = np.flatnonzero(fin)
    if n > 2000:
        idx = idx[lensgen.rng(3).integers(0, idx.size, 400)]
    _, absum = oracle.direct_sum(comps, dx[idx].astype(np.float64), dy[idx].astype(np.float64), with_absum=True)
    assert (np.abs(got[idx] - ref[idx]) / (absum + 1e-300)).max() <= 1e-6


@pytest.mark.parametrize("power", [-20, -40, -60])
@pytest.mark.parametrize("n", [1, 2, 33])
def test_unit_of_mass(power, n):
    """The fields scale with the unit of mass, also for a group of one ray (a
    call of one ray, the 33rd of a call, coincident rays): FP32 rounding does
    not depend on a power of two, so the bar is a few roundings of each field
    (1e-6 of the largest of its kind)."""
    p = lensgen.nfw_test_halos(300, 22, 0.3)
    q = p.copy()
    q[:, 2] *= 2.0 ** power
    if n == 2:
        dx, dy = np.full(2, 0.37, np.float32), np.full(2, -0.11, np.float32)
    else:
        dx, dy = (lensgen.rng(5).uniform(-2.0, 2.0, n).astype(np.float32) for _ in range(2))
    ref, got = shoot([L.Species.nfw(cu(p), 3.0)], dx, dy), shoot([L.Species.nfw(cu(q), 3.0)], dx, dy) * 2.0 ** -power
    scale = np.abs(ref).max(axis=1, keepdims=True)
    assert (np.abs(got - ref) / scale).max() <= 1e-6


@pytest.mark.parametrize("call", ["shoot", "potential"])
@pytest.mark.parametrize("kind,theta", [("points", 0.01), ("gauss", 0.01), ("nfw", 0.01)])
def test_repeated_call_is_bitwise_equal_when_most_groups_are_cut(kind, theta, call):
    """8,450 groups, most of them above the limit of a cut (16,384 entries):
    more cuts than could all have several parts of their own."""
    p = lensgen.nfw_particles(60_000, 9, nsph=32)
    if kind == "nfw":
        p[:, 3] = 0.01
    species = L.Species.points(cu(p)) if kind == "points" else getattr(L.Species, kind)(cu(p), 3.0)
    lens = L.Lens([species], theta=theta, group_rays=32)
    rx, ry = lensgen.grid_rays(520, -1.0, 1.0, dtype=np.float32)
    dx, dy = cu(rx), cu(ry)
    run = lens.shoot if call == "shoot" else lens.potential
    lens.shoot(dx, dy, flags=L.COUNT)
    c = lens.counters()
    assert c["cells"] // 2 + c["leaf_particles"] + c["big_kept"] > 16384 * c["groups"]
    first = [o.clone() for o in run(dx, dy)]
    for _ in range(5):
        assert all(torch.equal(a, b) for a, b in zip(first, run(dx, dy)))
    lens.close()


def test_scratch_of_a_small_lens():
    """The scratch of small calls: stacks (159 MB on 152 SMs), the direct sum's
    partial sums (12 MB) and little else; the cuts lie in the stacks' region.
    Eight lenses at once, at most 200 MB each."""
    p = lensgen.nfw_particles(4000, 11, nsph=16)
    dx, dy = (cu(lensgen.rng(12).uniform(-0.8, 0.8, 512).astype(np.float32)) for _ in range(2))
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    lenses = [L.Lens([L.Species.gauss(cu(p), 3.0)], theta=0.3) for _ in range(8)]
    for lens in lenses:
        lens.shoot(dx, dy)
        lens.sync()
    used = before - torch.cuda.mem_get_info()[0]
    for lens in lenses:
        lens.close()
    assert used <= 8 * 200e6, used / 8


def ray_groups(dx, dy, group):
    """The rays of each group (Morton order of 16-bit positions in their box)
    and the groups whose box is stretched: a side over 16 times that of an
    even share of the rays' box."""
    x0, y0 = dx.min(), dy.min()
    wx, wy = dx.max() - x0, dy.max() - y0
    inv = 65535.99 / max(wx, wy)

    def spread(v):
        v = v.astype(np.uint64)
        for s, m in ((8, 0x00ff00ff), (4, 0x0f0f0f0f), (2, 0x33333333), (1, 0x55555555)):
            v = (v | (v << np.uint64(s))) & np.uint64(m)
        return v

    keys = spread(np.floor((dx - x0) * inv)) | (spread(np.floor((dy - y0) * inv)) << np.uint64(1))
    order = np.argsort(keys, kind="stable")
    groups = [order[i:i + group] for i in range(0, order.size, group)]
    share = np.sqrt(group / dx.size)
    stretched = [g for g in groups if np.ptp(dx[g]) > 16 * share * wx or np.ptp(dy[g]) > 16 * share * wy]
    return groups, stretched


def outside_a_disk(n):
    """A grid of rays without a disk in its middle: Morton-consecutive rays
    across the hole make groups that span it."""
    rx, ry = lensgen.grid_rays(n, -1.0, 1.0, dtype=np.float32)
    m = rx ** 2 + ry ** 2 > 0.3
    return rx[m], ry[m]


@pytest.mark.parametrize("form", ["gauss", "gauss_alpha", "gauss_64", "gauss_fp64", "few_particles", "cut_form", "potential"])
def test_stretched_groups_are_cut(form):
    """Stretched groups in the launches that cut them: from 24,576 groups on (or
    with fewer than 24,576 particles) by themselves while the plain kernel takes
    the others, below with all groups; more than four particles a group.
    Reference: the producer/consumer form, 1e-6 of the sum of |terms| (1e-14 in
    FP64; the potential's: its direct evaluation of those rays alone, which cuts
    its one group per call into parts)."""
    from lens_testutil import comps_gauss
    group = 64 if form == "gauss_64" else 32
    n = 23_000 if form == "few_particles" else 172_000
    dx, dy = outside_a_disk(1800 if form == "gauss_64" else 480 if form == "few_particles" else
                            900 if form in ("cut_form", "potential") else 1300)
    groups, stretched = ray_groups(dx, dy, group)
    if form not in ("cut_form", "potential"):
        assert len(groups) >= 24576 or (4096 < len(groups) and n < 24576)
    else:
        assert 4096 < len(groups) < 24576
    assert n > 4 * len(groups) and len(stretched) > 0
    p = lensgen.nfw_particles(n, 9, nsph=32)
    prec = "fp64" if form == "gauss_fp64" else "fp32"
    dt = np.float64 if prec == "fp64" else np.float32
    dx, dy = dx.astype(dt), dy.astype(dt)
    lens = L.Lens([L.Species.gauss(cu(p), 3.0)], theta=0.3, group_rays=group, precision=prec)
    ref = L.Lens([L.Species.gauss(cu(p), 3.0)], theta=0.3, group_rays=group, precision=prec, walk="pairs")
    widest = max(stretched, key=lambda g: np.ptp(dx[g]) + np.ptp(dy[g]))
    lens.shoot(cu(dx[widest]), cu(dy[widest]), flags=L.COUNT)
    c = lens.counters()
    assert c["cells"] // 2 + c["leaf_particles"] + c["big_kept"] > 8192  # (the least a cut takes)
    idx = np.unique(np.concatenate(stretched[:8] + [widest] + [groups[0], groups[-1]]))
    flags = L.ALPHA_ONLY if form == "gauss_alpha" else 0
    if form == "potential":
        got = np.stack([o.double().cpu().numpy()[idx] for o in lens.potential(cu(dx), cu(dy))], 1)
        want = np.stack([o.double().cpu().numpy() for o in ref.potential(cu(dx[idx]), cu(dy[idx]))], 1)
        # (other groups take other decisions near a cell's radius: the tree's
        # own accuracy at theta 0.3)
        assert (np.abs(got - want).max(0) / np.abs(want).max(0)).max() <= 1e-3
    else:
        got, want = (np.stack([o.double().cpu().numpy()[idx] for o in q.shoot(cu(dx), cu(dy), flags=flags) if o is not None], 1)
                     for q in (lens, ref))
        _, absum = oracle.direct_sum(comps_gauss(p, 3.0), dx[idx].astype(np.float64), dy[idx].astype(np.float64), with_absum=True)
        d = np.abs(got - want) / (absum[:, :got.shape[1]] + 1e-300)
        assert d.max() <= (1e-14 if prec == "fp64" else 1e-6)
    lens.close()
    ref.close()


def test_adjoint_after_cut_groups():
    """The lists kept by parts of stretched groups give the walk's gradients."""
    g = lensgen.rng(3)
    dx, dy = outside_a_disk(1300)
    p = lensgen.nfw_particles(172_000, 9, nsph=32)
    a, b = (cu((0.01 * g.standard_normal(dx.size)).astype(np.float32)) for _ in range(2))
    lens = L.Lens([L.Species.gauss(cu(p), 3.0)], theta=0.3, group_rays=32)
    x, y = cu(dx), cu(dy)
    (walked,) = lens.backward(x, y, a, b)
    lens.shoot(x, y, flags=L.ALPHA_ONLY | L.KEEP_LISTS)
    (replayed,) = lens.backward(x, y, a, b, flags=L.KEEP_LISTS)
    for k in range(4):
        assert (replayed[:, k] - walked[:, k]).abs().max() <= 1e-6 * walked[:, k].abs().max()
    lens.close()


@pytest.mark.parametrize("kind", ["gauss", "nfw", "points", "points_fp64"])
@pytest.mark.parametrize("groups", [1, 2, 512, 513, 4096, 4097])
def test_group_counts_at_the_rules(kind, groups):
    """Group counts next to the rules, full groups and one ray more than the
    count before; trees of 1,000 and 20,000 particles (fewer than 512 are not
    cut).  1e-6 of the sum of |terms| (FP64: 1e-14)."""
    from lens_testutil import comps_gauss
    g = lensgen.rng(groups)
    prec = "fp64" if kind == "points_fp64" else "fp32"
    dt = np.float64 if prec == "fp64" else np.float32
    for n, rays in ((1000, 32 * groups), (20000 if kind != "nfw" else 3000, 32 * (groups - 1) + 1)):
        if kind == "gauss":
            p = lensgen.nfw_particles(n, 7, nsph=32)
            species, comps = L.Species.gauss(cu(p), 3.0), comps_gauss(p, 3.0)
        elif kind == "nfw":
            p = lensgen.nfw_test_halos(n, 22, 0.3)
            species, comps = L.Species.nfw(cu(p), 3.0), comps_nfw(p, 3.0)
        else:
            p = lensgen.point_disk(n, 33)
            species, comps = L.Species.points(cu(p)), comps_points(p)
        dx, dy = (g.uniform(-0.9, 0.9, rays).astype(dt) for _ in range(2))
        out = []
        for walk in ("warp", "pairs"):
            lens = L.Lens([species], theta=0.3, precision=prec, group_rays=32, walk=walk)
            out.append(np.stack([o.double().cpu().numpy() for o in lens.shoot(cu(dx), cu(dy))], 1))
            lens.close()
        idx = np.unique(np.r_[0, rays - 1, g.integers(0, rays, 60)])
        _, absum = oracle.direct_sum(comps, dx[idx].astype(np.float64), dy[idx].astype(np.float64), with_absum=True)
        assert (np.abs(out[0][idx] - out[1][idx]) / (absum + 1e-300)).max() <= (1e-14 if prec == "fp64" else 1e-6)


@pytest.mark.parametrize("width,group", [(1.3e-6, 128), (1.5e-6, 128), (0.0138, 64), (0.0144, 64), (0.9, 32), (1.6, 32), (1.6, 64)])
@pytest.mark.parametrize("batches", [1, 2])
def test_supergroup_rules(width, group, batches):
    """Point masses over patches on both sides of the rules for supergroups: a
    group's side an eighth of FP32's rounding, a patch 0.01 of the lens's
    r_cm (1.41), fields with few and with many stars near a supergroup; as one
    batch and as two, whose groups share a supergroup.  Reference: the
    producer/consumer form, 1e-6 of the sum of |terms|."""
    p = lensgen.point_disk(60_000, 55)
    n = 1460 if group == 128 else 1030 if group == 64 else 760
    dx, dy = lensgen.patch_offsets(n, width)
    origin = (0.5, 0.01) if width < 1 else (0.0, 0.0)
    assert dx.size >= 16384 * group
    x, y, rays = cu(dx), cu(dy), dx.size
    idx = np.unique(np.r_[0, rays - 1, lensgen.rng(3).integers(0, rays, 200)])
    pick = torch.from_numpy(idx).cuda()
    out = []
    for walk in ("warp", "pairs"):
        lens = L.Lens([L.Species.points(cu(p))], theta=0.3, group_rays=group, walk=walk)
        if batches == 1:
            o = lens.shoot(x, y, origin=origin)
        else:
            o = lens.shoot_batches(np.array([0, rays // 2 + 17, rays]), np.array([origin, origin]), x, y)
        out.append(np.stack([v[pick].double().cpu().numpy() for v in o], 1))
        lens.close()
    rx, ry = origin[0] + dx[idx].astype(np.float64), origin[1] + dy[idx].astype(np.float64)
    _, absum = oracle.direct_sum(comps_points(p), rx, ry, with_absum=True)
    # (the reference groups at most 64 rays; over 1.5e-6 the decisions are the same)
    assert (np.abs(out[0] - out[1]) / (absum + 1e-300)).max() <= 1e-6


@pytest.mark.parametrize("groups", [512, 513, 2500])
def test_few_groups_of_a_large_tree(groups):
    """Trees of 200,000 particles: all groups are cut up to 512 of them, heavy ones
    above.  1e-6 of the sum of |terms|."""
    from lens_testutil import comps_gauss
    g = lensgen.rng(groups)
    p = lensgen.nfw_particles(200_000, 7, nsph=32)
    n = 32 * groups
    dx, dy = (g.uniform(-0.9, 0.9, n).astype(np.float32) for _ in range(2))
    got, ref = shoot([L.Species.gauss(cu(p), 3.0)], dx, dy), shoot([L.Species.gauss(cu(p), 3.0)], dx, dy, walk="pairs")
    idx = np.unique(np.r_[0, n - 1, g.integers(0, n, 60)])
    _, absum = oracle.direct_sum(comps_gauss(p, 3.0), dx[idx].astype(np.float64), dy[idx].astype(np.float64), with_absum=True)
    assert (np.abs(got[idx] - ref[idx]) / (absum + 1e-300)).max() <= 1e-6
