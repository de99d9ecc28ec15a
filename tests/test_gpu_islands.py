"""The DEM by components of the contact graph: chains of spheres of every
size class (alone, a group of 8 lanes, a warp, more than a warp) step bitwise
as in the batched form, which runs all spheres of a member in one cluster, in
the cluster and the grid form of the large components."""
import numpy as np
import pytest

from paper_1703_05158_gb300 import lbm

pytestmark = pytest.mark.gpu

SIZES = (1, 2, 8, 9, 31, 32, 33, 70)
BOX = (180, 40, 24)


def chains():
    g = np.random.default_rng(7)
    X = [(2.0 + 2.5 * k, 2.5 + 5.0 * row, 11.3) for row, n in enumerate(SIZES) for k in range(n)]
    X = np.array(X) + g.uniform(-0.02, 0.02, (len(X), 3))
    perm = g.permutation(len(X))  # members of a chain at any index
    return X[perm], g.uniform(-0.05, 0.05, (len(X), 3)), g.uniform(-0.01, 0.01, (len(X), 3)), np.full(len(X), 1.2)


@pytest.mark.parametrize("friction", [False, True])
@pytest.mark.parametrize("mode", ["auto", "cluster", "grid"])
def test_chains_step_as_in_one_cluster(mode, friction):
    X, V, Om, R = chains()
    kw = dict(nx=BOX[0], ny=BOX[1], nz=BOX[2], tau0=0.7, cs=0.15, kn=50.0, restitution=0.8, dem_substeps=15,
              max_particles=len(R), max_radius=1.2)
    if friction:
        kw.update(kt=20.0, mu=0.3, restitution_t=0.7)
    alone = lbm.Lattice(dem_mode=mode, **kw)
    batch = lbm.Batch([kw])
    state = []
    for lat, run in ((alone, alone), (batch[0], batch)):
        lat.set_particles(X, V=V, Om=Om, R=R)
        run.step(25)
        state.append(lat.particles() + lat.forces())
    assert np.abs(state[0][1] - V).max() > 1e-2  # the chains did collide
    for a, b in zip(*state):
        assert np.array_equal(a, b)
