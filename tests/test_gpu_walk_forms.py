"""The forms of the tree walk that the launch picks by the number of ray groups,
by the shape of their boxes and by the kind of tree give one result: groups
cut into parts (few groups, heavy ones, stretched ones), the plain kernel,
supergroups with local expansions (point masses), and the producer/consumer
form, which none of these rules touch, as the reference.

Tolerance: the same terms in another order, 1e-6 of the sum of |terms| for FP32
(the bar the walk forms already meet) and 1e-14 for FP64; an expansion's first
omitted term is 1.2e-9 of its source, far below.
"""
import numpy as np
import pytest

import lensgen
import oracle
from lens_testutil import comps_gauss, comps_nfw, comps_points

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_1312_1128_gb300 as L  # noqa: E402


def cu(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def both(species, dx, dy, origin=(0.0, 0.0), flags=0, prec="fp32", group=64, theta=0.3):
    out = []
    for walk in ("warp", "pairs"):
        lens = L.Lens(species, theta=theta, precision=prec, group_rays=group, walk=walk)
        o = lens.shoot(dx, dy, origin=origin, flags=flags)
        lens.sync()
        out.append(np.stack([x.double().cpu().numpy() for x in o if x is not None], axis=1))
        lens.close()
    return out


def check(comps, dx, dy, origin, got, ref, prec="fp32", sample=400):
    n = got.shape[0]
    idx = np.unique(np.r_[0, n - 1, lensgen.rng(3).integers(0, n, sample)])
    rx, ry = origin[0] + dx[idx].astype(np.float64), origin[1] + dy[idx].astype(np.float64)
    _, absum = oracle.direct_sum(comps, rx, ry, with_absum=True)
    d = np.abs(got[idx] - ref[idx]) / (absum[:, :got.shape[1]] + 1e-300)
    assert d.max() <= (1e-14 if prec == "fp64" else 1e-6), d.max(axis=0)


@pytest.mark.parametrize("n_rays", [1, 33, 2047, 2048 * 32 + 5, 4096 * 32 + 33])
@pytest.mark.parametrize("kind", ["gauss", "nfw", "points", "points_fp64"])
def test_cut_groups(kind, n_rays):
    """Group counts on both sides of the rules (1, 2, 512, 4096 groups of 32)."""
    g = lensgen.rng(101)
    prec = "fp64" if kind == "points_fp64" else "fp32"
    if kind == "gauss":
        p = lensgen.nfw_particles(20000, 7, nsph=32)
        species, comps = [L.Species.gauss(cu(p), 3.0)], comps_gauss(p, 3.0)
    elif kind == "nfw":
        p = lensgen.nfw_test_halos(3000, 22, 0.3)
        species, comps = [L.Species.nfw(cu(p), 3.0)], comps_nfw(p, 3.0)
    else:
        p = lensgen.point_disk(20000, 33)
        species, comps = [L.Species.points(cu(p))], comps_points(p)
    dt = np.float64 if prec == "fp64" else np.float32
    dx, dy = (g.uniform(-0.9, 0.9, n_rays).astype(dt) for _ in range(2))
    got, ref = both(species, cu(dx), cu(dy), prec=prec, group=32)
    check(comps, dx, dy, (0.0, 0.0), got, ref, prec, 60)


@pytest.mark.parametrize("alpha_only", [False, True])
def test_stretched_groups(alpha_only):
    """Rays outside a radius: Morton-consecutive rays across the hole make
    groups that span it (the plain kernel leaves them to the cut form)."""
    p = lensgen.nfw_particles(150_000, 9, nsph=32)
    rx, ry = lensgen.grid_rays(1300, -1.0, 1.0, dtype=np.float32)
    m = rx ** 2 + ry ** 2 > 0.3
    dx, dy = rx[m], ry[m]
    flags = L.ALPHA_ONLY if alpha_only else 0
    got, ref = both([L.Species.gauss(cu(p), 3.0)], cu(dx), cu(dy), flags=flags, group=32)
    check(comps_gauss(p, 3.0), dx, dy, (0.0, 0.0), got, ref, sample=60)


@pytest.mark.parametrize("width,group", [(1e-6, 128), (1e-4, 32), (0.05, 64), (0.6, 32)])
def test_supergroups(width, group):
    """Point masses, 16,384 and more groups: a tiny patch (one expansion for
    nearly everything), a narrow one (no expansions), wide ones."""
    p = lensgen.point_disk(60_000, 55)
    n = 1460 if group == 128 else 1030 if group == 64 else 760
    dx, dy = lensgen.patch_offsets(n, width)
    origin = (0.5, 0.01)
    got, ref = both([L.Species.points(cu(p))], cu(dx), cu(dy), origin=origin, group=group, theta=0.2)
    if group == 128:
        # (the reference form groups at most 64 rays; over this patch the
        # decisions are the same)
        assert dx.size >= 16384 * 128
    check(comps_points(p), dx, dy, origin, got, ref, sample=60)
