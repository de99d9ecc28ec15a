"""The collide that stages whole rows in shared memory gives the bits of the
node-wise kernels (which the overlapped schedule runs): rows of one and more
buffers' worth, several rows per unit with a part of one left over, the
periodic ends, both walls, spheres across them, every storage."""
import numpy as np
import pytest

from paper_1703_05158_gb300 import inputs, lbm

pytestmark = pytest.mark.gpu

# at least 2^21 nodes each: smaller lattices take the node kernels anyway
SHAPES = {"fp32": [(256, 64, 129), (252, 67, 125), (128, 129, 128), (116, 139, 131)],
          "fp16": [(512, 64, 65), (520, 64, 64)],
          "bf16": [(1024, 45, 46), (1000, 47, 46)]}


@pytest.mark.parametrize("precision,shape", [(p, s) for p in SHAPES for s in SHAPES[p]])
def test_rows_are_bitwise_the_node_kernels(precision, shape):
    nx, ny, nz = shape
    R = 2.6
    X = np.array([(0.3, 5.2, 4.1), (nx - 1.2, ny - 0.4, nz - 4.4), (nx / 2, ny / 2, nz / 2), (5.9, 12.1, 20.7)])
    V = np.array([(0.06, 0.03, -0.02), (-0.05, 0.04, 0.02), (0.03, -0.06, 0.05), (0.02, 0.01, 0.06)])
    f = np.repeat(np.array([12] + [2] * 3 + [1] * 6 + [2] * 3 + [1] * 6)[:, None] / 36.0, nx * ny * nz, 1)
    f *= 1 + inputs.perturbation(f.shape, 0.02, 11)
    out = []
    for schedule in ("serial", "overlap"):
        lat = lbm.Lattice(nx, ny, nz, tau0=0.6, cs=0.17, g=(1e-5, 2e-6, 0.0), u_lo=(0.0, -0.02, 0.0),
                          u_hi=(0.05, 0.0, 0.0), max_particles=4, max_radius=2.6, precision=precision,
                          schedule=schedule)
        lat.set_particles(X, V=V, R=np.full(4, R))
        lat.set_populations(f)
        lat.step(3)
        odd = lat.populations()
        lat.step(4)
        out.append((odd, lat.populations(), lat.owner()) + lat.forces() + lat.particles())
        lat.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)

