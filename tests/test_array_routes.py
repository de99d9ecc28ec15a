"""Which arrays of a call a kernel may touch: memory of the handle's own device
that starts at a whole double, pinned arrays of a call that says host memory,
and nothing else (no other device's memory, no host memory in a call that says
device memory); nor does the host write to device memory in a call that says
host memory.  The rule is compiled by itself, so that it is tried for every
kind of memory without a GPU.  Many spheres are read by copies, a few through
pinned memory: the values are the same."""
import ctypes
import itertools
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1703_05158_gb300", "csrc")
PAGEABLE, PINNED, DEVICE, MANAGED = range(4)
KERNEL, STAGED, COPY = range(3)


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    d = tmp_path_factory.mktemp("route")
    (d / "r.cpp").write_text('#include "lbm_route.cuh"\nusing namespace lbm;\nextern "C" {\n'
                             "int dev(int m, int here, unsigned long at) { return (int)route_device({(Mem)m, here != 0, at}); }\n"
                             "int host(int m, int here, unsigned long at, int st) "
                             "{ return (int)route_host({(Mem)m, here != 0, at}, st != 0); }\n}\n")
    out = str(d / "r.so")
    subprocess.run(["g++", "-shared", "-fPIC", "-I", CSRC, str(d / "r.cpp"), "-o", out], check=True)
    return ctypes.CDLL(out)


def test_device_calls(rule):
    for mem, here, off in itertools.product(range(4), (0, 1), range(9)):
        want = KERNEL if mem == DEVICE and here and off % 8 == 0 else COPY
        assert rule.dev(mem, here, ctypes.c_ulong(4096 + off)) == want, (mem, here, off)


def test_host_calls(rule):
    for mem, here, stage, at in itertools.product(range(4), (0, 1), (0, 1), (0, 4096, 4100, 4104)):
        want = COPY if mem == DEVICE or not stage else STAGED
        if mem == PINNED and here and at in (4096, 4104):
            want = KERNEL
        assert rule.host(mem, here, ctypes.c_ulong(at), stage) == want, (mem, here, stage, at)


@pytest.mark.gpu
def test_a_device_load_in_a_capture():
    """The load of device arrays is stream work alone: recorded once, replayed with other values."""
    torch = pytest.importorskip("torch")
    from paper_1703_05158_gb300 import lbm

    s = torch.cuda.Stream()
    F = torch.full((1, 3), 1e-3, dtype=torch.float64, device="cuda")
    T = torch.full((1, 3), 2e-3, dtype=torch.float64, device="cuda")
    runs = []
    for captured in (True, False):
        lat = lbm.Lattice(24, 24, 24, tau0=0.7, max_particles=1, max_radius=3.0, stream=s.cuda_stream)
        lat.set_particles([(12.0, 12.0, 12.0)], R=[3.0])
        torch.cuda.synchronize()
        if captured:
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=s):
                lbm.lbm_set_particle_load(lat.h, F, T)
        for k in (1.0, -3.0):
            with torch.cuda.stream(s):
                F.fill_(k * 1e-3)
                T.fill_(k * 2e-3)
                if captured:
                    g.replay()
                else:
                    lbm.lbm_set_particle_load(lat.h, F, T)
            lat.step(1)
        runs.append(lat.particles())
        assert np.abs(runs[-1][1]).max() > 0
        lat.close()
    for a, b in zip(*runs):
        assert np.array_equal(a, b)


@pytest.mark.gpu
@pytest.mark.parametrize("n", [1, 4096, 4097, 9000])
def test_host_arrays_of_every_kind(n):
    torch = pytest.importorskip("torch")
    from paper_1703_05158_gb300 import lbm

    X = np.array([(3.0 + 5 * (a % 32), 3.0 + 5 * (a // 32 % 32), 3.0 + 5 * (a // 1024)) for a in range(n)])
    lat = lbm.Lattice(160, 160, 48, tau0=0.7, max_particles=n + 3, max_radius=2.0)
    lat.set_particles(X, V=np.full((n, 3), 0.01), R=np.full(n, 1.8))
    lat.set_load(F=1e-3 * X, T=2e-3 * X)
    lat.step(3)
    dev = [torch.empty((n, 3), dtype=torch.float64, device="cuda") for _ in range(5)]
    lbm.lbm_particle_state(lat.h, *dev)
    want = [d.cpu().numpy() for d in dev]
    assert all(np.abs(w).max() > 0 for w in want)
    pageable = [np.empty((n, 3)) for _ in range(5)]
    pinned = [torch.empty((n, 3), dtype=torch.float64, pin_memory=True).numpy() for _ in range(5)]
    odd = torch.empty(5 * n * 24 + 8, dtype=torch.uint8, pin_memory=True).numpy()
    shifted = [np.frombuffer(odd[4 + k * n * 24:4 + (k + 1) * n * 24].data, dtype=np.float64).reshape(n, 3)
               for k in range(5)]
    for arrays in (pageable, pinned, shifted, [pageable[0] * 0, pinned[1] * 0] + shifted[2:]):
        at = [ctypes.c_void_p(a.ctypes.data) for a in arrays]
        assert lbm.load().lbm_particle_state(lat.h, *at, lbm.LBM_HOST) == 0
        for a, w in zip(arrays, want):
            assert np.array_equal(a, w)
    lat.close()
