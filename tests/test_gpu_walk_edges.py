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
