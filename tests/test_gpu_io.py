"""Populations in and out are the FP64 operations bit for bit (the kernels use
integer arithmetic where it gives the same), for values in and out of the
binade of their weight, zeros, subnormals, infinities and NaN, at both step
parities and in every storage; loads and sphere state reach host and device
arrays, also ones that do not start at a whole double."""
import ctypes

import numpy as np
import pytest

import oracle
from paper_1703_05158_gb300 import lbm

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def stored(d, precision):
    t = torch.from_numpy(d)
    kind = {"fp32": torch.float32, "bf16": torch.bfloat16, "fp16": torch.float16}[precision]
    return t.to(kind).to(torch.float32).numpy()


@pytest.mark.parametrize("precision", ["fp32", "bf16", "fp16"])
@pytest.mark.parametrize("steps", [0, 1])
@pytest.mark.parametrize("shape", [(17, 9, 7), (64, 4, 3)])
def test_populations_are_the_fp64_operations(shape, steps, precision):
    nx, ny, nz = shape
    _, w, _ = oracle.tables()
    g = np.random.default_rng(3)
    N = nx * ny * nz
    f = w[:, None] + g.normal(size=(19, N)) * 10.0 ** g.uniform(-45, 2, (19, N))
    near = g.random((19, N)) < 0.5
    f[near] = (w[:, None] * (1 + 0.3 * g.uniform(-1, 1, (19, N))))[near]
    f[:, :12] = np.stack([w, 0 * w, -0.0 * w, w + 5e-324, np.nextafter(w, 1), np.nextafter(w, 0), 2.0 * w, 0.5 * w, -w,
                          0 * w + np.inf, 0 * w - np.inf, 0 * w + np.nan], 1)
    f[:, 12:60] = w[:, None] + 2.0 ** -np.arange(20.0, 68.0) * 1.3
    lat = lbm.Lattice(nx, ny, nz, tau0=0.7, precision=precision)
    lat.step(steps)
    lat.set_populations(f)
    with np.errstate(all="ignore"):
        want = w[:, None] + stored((f - w[:, None]).astype(np.float32), precision).astype(np.float64)
    assert np.array_equal(lat.populations().reshape(19, N), want, equal_nan=True)


def test_sphere_state_to_every_kind_of_array():
    n = 300
    g = np.random.default_rng(5)
    X = np.array([(6.0 + 9 * i, 6.0 + 9 * j, 6.0 + 9 * k) for i in range(10) for j in range(6) for k in range(5)])
    lat = lbm.Lattice(96, 60, 50, tau0=0.7, max_particles=n, max_radius=3.0)
    lat.set_particles(X, V=g.uniform(-0.01, 0.01, (n, 3)), R=g.uniform(2, 3, n))
    lat.set_load(F=g.uniform(-1e-3, 1e-3, (n, 3)), T=g.uniform(-1e-3, 1e-3, (n, 3)))
    lat.step(3)
    host = lat.forces() + lat.particles()
    together = [np.empty((n, 3)) for _ in range(5)]
    lbm.lbm_particle_state(lat.h, *together)
    dev = torch.empty((5, n, 3), dtype=torch.float64, device="cuda")
    lbm.lbm_particle_state(lat.h, *dev)
    odd = torch.zeros(5 * n * 24 + 8, dtype=torch.uint8, device="cuda")
    at = [ctypes.c_void_p(odd.data_ptr() + 4 + k * n * 24) for k in range(5)]
    assert lbm.load().lbm_particle_state(lat.h, *at, lbm.LBM_DEVICE) == 0
    bytes_ = odd.cpu().numpy()[4:4 + 5 * n * 24].tobytes()
    shifted = np.frombuffer(bytes_, dtype=np.float64).reshape(5, n, 3)
    for k, want in enumerate(host):
        assert np.abs(want).max() > 0
        assert np.array_equal(together[k], want)
        assert np.array_equal(dev[k].cpu().numpy(), want)
        assert np.array_equal(shifted[k], want)
    only = np.empty((n, 3))
    lbm.lbm_particle_state(lat.h, pos=only)
    assert np.array_equal(only, host[2])


@pytest.mark.parametrize("where", ["host", "device", "device_shifted"])
@pytest.mark.parametrize("given", ["both", "force", "torque", "none"])
def test_loads_from_every_kind_of_array(where, given):
    def run(call):
        lat = lbm.Lattice(40, 30, 24, tau0=0.7, max_particles=2, max_radius=3.0)
        lat.set_particles([(10.0, 10.0, 10.0), (25.0, 20.0, 12.0)], R=[3.0, 2.5])
        lat.set_load(np.ones((2, 3)), np.ones((2, 3)))  # replaced below
        call(lat)
        lat.step(2)
        return lat.particles()

    F, T = np.array([(1e-3, 2e-3, -1e-3), (0.0, -2e-3, 1e-3)]), np.array([(3e-3, 0.0, 1e-3), (-1e-3, 1e-3, 2e-3)])
    F, T = (F if given in ("both", "force") else None), (T if given in ("both", "torque") else None)
    want = run(lambda lat: lat.set_load(F, T))
    if where == "host":
        got = run(lambda lat: lat.set_load(F, T))
    else:
        shift = 4 if where == "device_shifted" else 0
        buf = torch.zeros(128, dtype=torch.uint8, device="cuda")
        for k, a in enumerate((F, T)):
            if a is not None:
                buf[shift + 48 * k:shift + 48 * (k + 1)] = torch.from_numpy(np.frombuffer(a.tobytes(), np.uint8).copy())
        torch.cuda.synchronize()
        at = [None if a is None else ctypes.c_void_p(buf.data_ptr() + shift + 48 * k) for k, a in enumerate((F, T))]
        got = run(lambda lat: lbm.load().lbm_set_particle_load(lat.h, *at, lbm.LBM_DEVICE))
    zero = run(lambda lat: lat.set_load(None, None))
    for a, b, c in zip(got, want, zero):
        assert np.array_equal(a, b)
    assert given == "none" or not np.array_equal(got[1], zero[1]) or not np.array_equal(got[2], zero[2])
