"""Spheres at the walls: the rows of a sphere's cube beyond a wall are solid
and belong to nobody.  Just off, touching and set into the lower and the upper
wall, fixed and free, as sphere 0 and beside another, in boxes of few and many
planes: owners, links, populations and forces against the FP64 oracle, and the
batched form bit for bit."""
import math

import numpy as np
import pytest

import oracle
from paper_1703_05158_gb300 import lbm

pytestmark = pytest.mark.gpu

# a soft contact, so that a sphere set into a wall stays within the motion one step allows
KW = dict(tau0=0.7, cs=0.15, g=(2e-6, 0.0, 0.0), u_hi=(0.02, 0.0, 0.0), rho_s=2.5, kn=1.0, restitution=0.8,
          dem_substeps=8)
RADII = [2.2, 2.5, 3.3, 4.0, 4.4]
GAPS = [0.45, 0.1, 0.0, -0.15, -0.6, -1.4]  # from the wall's surface, negative: set into it


def case(radius, wall, gap, fixed, first, planes, wide=0):
    n = 2 * (math.ceil(radius) + 3) + 1 + wide
    nz = 2 * math.ceil(radius) + 3 + planes
    z = radius + gap - 0.5
    z = z if wall == "lower" else nz - 1 - z
    X, R, V, fx = [(n / 2 + 0.3, 0.6, z)], [radius], [(0.02, -0.013, -0.007 if wall == "lower" else 0.007)], [fixed]
    if not first:  # the sphere at the wall is sphere 1, the other one is in the opposite half
        X.insert(0, (0.4, n / 2 + 0.2, nz - 1 - z + (-0.3 if wall == "lower" else 0.3)))
        R.insert(0, 2.0), V.insert(0, (0.01, 0.0, 0.0)), fx.insert(0, False)
    return (n, n, nz), np.array(X), np.array(R), np.array(V), np.array(fx, dtype=np.uint8)


def place(side, X, R, V, fx):
    side.set_particles(X, V=V, Om=0.15 * V, R=R, fixed=fx)


def brute_links(owner):
    fluid = owner < 0
    solid = np.argwhere(~fluid)
    count, c = 0, oracle.tables()[0]
    for j in range(1, 19):
        x = solid - c[j][::-1]
        x[:, 1] %= owner.shape[1]
        x[:, 2] %= owner.shape[2]
        x = x[(x[:, 0] >= 0) & (x[:, 0] < owner.shape[0])]
        count += int(fluid[tuple(x.T)].sum())
    return count


def compare(box, X, R, V, fx):
    lat = lbm.Lattice(*box, max_particles=len(R), max_radius=max(R), **KW)
    ref = oracle.Oracle(*box, **KW)
    for side in (lat, ref):
        place(side, X, R, V, fx)
    for steps in (1, 1, 2):  # both parities, from a graph of one step and of two
        for side in (lat, ref):
            side.step(steps)
        owner = ref.owner()
        assert np.array_equal(lat.owner(), owner)
        assert lat.info()["links"] == brute_links(owner)
        want = ref.populations()[:, owner < 0]
        assert (np.abs(lat.populations()[:, owner < 0] - want) / np.abs(want)).max() <= 1e-5
        for a, b, floor in zip(lat.forces(), ref.forces(), (1e-7, 1e-6 * R.max())):
            for p in range(len(R)):
                assert np.linalg.norm(a[p] - b[p]) <= 1e-4 * np.linalg.norm(b[p]) + floor
        # a load off by 1e-4 of itself moves a sphere by 1e-4 |F| / m t^2 / 2: with |F| / m <= 0.05 and t = 4, 4e-5
        for a, b in zip(lat.particles(), ref.particles()):
            assert np.abs(a - b).max() <= 4e-5


@pytest.mark.parametrize("fixed", [True, False])
@pytest.mark.parametrize("gap", GAPS)
@pytest.mark.parametrize("wall", ["lower", "upper"])
@pytest.mark.parametrize("radius", RADII)
def test_a_sphere_at_a_wall(radius, wall, gap, fixed):
    for first, planes, wide in ((True, 2, 0), (False, 14, 3)):
        compare(*case(radius, wall, gap, fixed, first, planes, wide))


@pytest.mark.parametrize("radius", [2.2, 4.4])
def test_a_wide_flat_box(radius):
    """One sphere where a plane holds more nodes than the sphere arrays hold words."""
    compare(*case(radius, "lower", -0.1, False, True, 0, 101))
    compare(*case(radius, "upper", -0.1, False, True, 0, 101))


@pytest.mark.parametrize("nz", [1, 2, 3])
def test_a_sphere_through_both_walls(nz):
    X, V = np.array([(8.3, 7.6, (nz - 1) / 2 + 0.2)]), np.array([(0.02, -0.01, 0.003)])
    compare((17, 19, nz), X, np.array([2.2]), V, np.array([1], dtype=np.uint8))


@pytest.mark.parametrize("precision", ["fp32", "bf16"])
def test_members_of_a_batch(precision):
    cases = [case(R, wall, gap, False, first, planes) for R, wall, gap, first, planes in
             ((2.2, "lower", 0.1, True, 2), (3.3, "upper", 0.1, False, 9), (2.5, "upper", -0.15, True, 0),
              (4.4, "lower", -0.6, False, 6), (4.0, "lower", -0.6, True, 2))]
    kw = dict(KW, precision=precision, max_particles=2, max_radius=4.4)
    kw.pop("g")
    batch = lbm.Batch([dict(nx=b[0] + 4, ny=b[1] + 4, nz=b[2], g=(1e-6, 0.0, 0.0), **kw) for b, *_ in cases])
    alone = [lbm.Lattice(b[0] + 4, b[1] + 4, b[2], g=(1e-6, 0.0, 0.0), **kw) for b, *_ in cases]
    for m, a, (_, *parts) in zip(batch.members, alone, cases):
        place(m, *parts)
        place(a, *parts)
        a.step(5)
    batch.step(5)
    batch.sync()
    for m, a in zip(batch.members, alone):
        assert np.array_equal(m.owner(), a.owner())
        assert np.array_equal(m.populations(), a.populations())
        for x, y in zip(m.forces() + m.particles(), a.forces() + a.particles()):
            assert np.array_equal(x, y)
