"""Node classes kept between steps: spheres that are alone, come within reach
of each other, overlap (soft contacts), part again and cross the periodic
faces own the oracle's nodes after every step, with and without the momentum
correction, whose marks visit every node instead."""
import numpy as np
import pytest

import oracle
from paper_1703_05158_gb300 import lbm

pytestmark = pytest.mark.gpu

KW = dict(tau0=0.8, cs=0.1, rho_s=2.5, kn=5.0, restitution=0.9, dem_substeps=8)


@pytest.mark.parametrize("correction", [False, True])
@pytest.mark.parametrize("schedule", ["serial", "overlap"])
def test_owners_over_an_encounter(schedule, correction):
    X = np.array([(4.0, 10.2, 9.7), (13.9, 10.9, 10.2), (26.1, 20.0, 5.2), (1.2, 26.6, 5.6)])
    V = np.array([(0.12, 0.01, 0.0), (-0.11, 0.0, 0.01), (0.10, 0.12, 0.02), (-0.1, -0.05, 0.0)])
    R = np.array([3.3, 4.0, 2.7, 3.6])
    lat = lbm.Lattice(30, 28, 20, max_particles=4, max_radius=4.0, schedule=schedule,
                      momentum_correction=correction, **KW)
    orc = oracle.Oracle(30, 28, 20, momentum_correction=correction, **KW)
    for o in (lat, orc):
        o.set_particles(X, V=V, R=R)
    touched = 0
    for _ in range(70):
        lat.step(1)
        orc.step(1)
        want = orc.owner()
        assert np.array_equal(lat.owner(), want)
        d = lat.particles()[0]
        gap = d[0] - d[1]
        touched += np.linalg.norm(gap - np.round(gap / [30, 28, 1e9]) * [30, 28, 0]) < R[0] + R[1] - 0.5
    assert touched > 5
    fluid = want < 0
    f, ref = lat.populations(), orc.populations()
    assert (np.abs(f - ref)[:, fluid] / np.abs(ref[:, fluid])).max() <= 1e-5
