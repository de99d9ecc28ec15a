"""The link kernel's cube of rows at its edges: the smallest and largest
radii, cubes that cross the periodic faces and the walls, rows of every
alignment and rows just wide enough for the cube.  Links, populations and
forces against the FP64 oracle."""
import math

import numpy as np
import pytest

import oracle
from paper_1703_05158_gb300 import lbm

pytestmark = pytest.mark.gpu

KW = dict(tau0=0.7, cs=0.15, g=(2e-6, 0.0, 0.0), u_hi=(0.02, 0.0, 0.0), rho_s=2.5, kn=1e3, restitution=0.8,
          dem_substeps=8)


@pytest.mark.parametrize("radius", [0.7, 1.0, 2.5, 4.0, 7.3, 12.9, 16.0])
@pytest.mark.parametrize("pad", [0, 1, 2, 7])
@pytest.mark.parametrize("place", ["centre", "corner", "low_face", "walls"])
def test_one_sphere(radius, pad, place):
    n = 2 * (math.ceil(radius) + 3) + 1 + pad
    nz = 2 * math.ceil(radius) + 5
    X = {"centre": (n / 2 + 0.3, n / 2 - 0.2, nz / 2 - 0.4), "corner": (n - 0.4, n - 0.7, nz / 2 - 0.1),
         "low_face": (0.2, n / 2, nz / 2 - 0.45), "walls": (n / 2, 0.6, radius + 0.2)}[place]
    out = []
    for side in (lbm.Lattice(n, n, nz, max_particles=1, max_radius=radius, **KW), oracle.Oracle(n, n, nz, **KW)):
        side.set_particles([X], V=[(0.02, -0.013, 0.007)], Om=[(0.003, -0.002, 0.001)], R=[radius])
        side.step(4)
        out.append((side.owner(), side.populations(), *side.forces()))
        if isinstance(side, lbm.Lattice):
            links = side.info()["links"]
    (owner, f, F, T), (ref_owner, ref, Fr, Tr) = out
    assert np.array_equal(owner, ref_owner)
    fluid = ref_owner < 0
    solid = np.argwhere(~fluid)
    want = 0
    c = oracle.tables()[0]
    for j in range(1, 19):
        x = solid - c[j][::-1]
        x[:, 1:] %= n
        ok = (x[:, 0] >= 0) & (x[:, 0] < nz)
        want += int(fluid[tuple(x[ok].T)].sum())
    assert links == want
    assert (np.abs(f - ref)[:, fluid] / np.abs(ref[:, fluid])).max() <= 1e-5
    assert np.linalg.norm(F - Fr) <= 1e-4 * np.linalg.norm(Fr) + 1e-7
    assert np.linalg.norm(T - Tr) <= 1e-4 * np.linalg.norm(Tr) + 1e-6 * radius
