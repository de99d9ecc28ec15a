"""Cut links of the channel where their records meet: one or two fluid nodes
between two spheres, a sphere and a wall, a sphere and the plate, spheres
next to the inlet and outlet planes, and rows that end inside a block or
cross one.  Populations and gradient against the FP64 channel oracle, with
the tolerances of the other channel tests."""
import numpy as np
import pytest

import oracle
from paper_1703_05158_gb300 import lbm

pytestmark = pytest.mark.gpu

BASE = dict(ny=12, nz=14, tau0=0.6, cs=0.15, gx=2e-6, u_peak=0.04, steps=40, avg_from=21)

# name: (nx, plate box, spheres (x, y, z, r))
CASES = {
    "one_node_between_spheres": (40, ((26, 3, 3), (27, 8, 10)), [(9.0, 6.0, 7.0, 3.0), (16.1, 6.2, 7.1, 3.05)]),
    "two_nodes_between_spheres": (40, ((26, 3, 3), (27, 8, 10)), [(9.0, 6.0, 7.0, 2.8), (16.2, 6.1, 6.8, 2.9)]),
    "sphere_on_the_wall_and_the_plate": (40, ((18, 3, 3), (19, 8, 10)), [(10.0, 6.0, 3.3, 3.0), (14.2, 6.0, 9.8, 2.9)]),
    "spheres_at_inlet_and_outlet": (36, ((16, 3, 3), (17, 8, 10)), [(4.05, 6.0, 6.5, 3.0), (30.9, 5.5, 7.5, 3.0)]),
    "overlapping_across_the_period": (33, ((20, 0, 5), (20, 11, 8)), [(8.0, 0.4, 6.0, 3.0), (9.5, 10.7, 8.5, 2.5)]),
    "row_longer_than_a_block": (141, ((130, 3, 3), (131, 8, 10)), [(126.4, 6.0, 7.0, 2.6), (20.0, 6.0, 7.0, 3.0)]),
    "no_obstacle": (29, ((5, 3, 3), (4, 8, 10)), []),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_populations_and_gradient(name):
    nx, (lo, hi), sph = CASES[name]
    X = np.array([s[:3] for s in sph]).reshape(-1, 3)
    R = np.array([s[3] for s in sph])
    cfg = dict(BASE, nx=nx, plate_lo=lo, plate_hi=hi)
    ch = lbm.Channel(**cfg, checkpoint_every=7, X=X, R=R)
    J = ch.forward()
    g = ch.backward()
    ref = oracle.channel(**cfg, X=X, R=R, populations=True)
    open_ = (ref["type"] != 1) & (ref["type"] != 4)
    assert np.array_equal(ch.geometry(), ref["type"])
    f = ch.populations()
    assert (np.abs(f - ref["f"])[:, open_] / np.abs(ref["f"][:, open_])).max() <= 1e-5
    assert abs(J - ref["J"]) <= 1e-4 * abs(ref["J"])
    for k in range(3):
        d = np.zeros(3)
        d[k] = 1.0
        want = oracle.channel(**cfg, X=X, R=R, dtheta=d)["dJ"]
        assert abs(g[k] - want) <= 1e-3 * abs(want), (k, g[k], want)
    assert np.array_equal(ch.backward(), g)  # a second sweep starts from the same state
