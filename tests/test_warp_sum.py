"""The warp sums of the adjoint's parameter gradients: 32 floats added as
integers aligned to the largest of them.  The pieces run on the host; the sum
has to be within one FP64 rounding and 32 x 2^-57 of the largest value of the
exact one, which is no further off than FP64 additions may be."""
import ctypes
import math
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1703_05158_gb300", "csrc")

SOURCE = """
#include "lbm_sum.cuh"
#include <cstring>
using namespace lbm;
extern "C" double total(const uint32_t *u) {
    int E = 1;
    for (int l = 0; l < 32; ++l) E = sum_exp(u[l]) > E ? sum_exp(u[l]) : E;
    uint32_t lo = 0, mid = 0;
    int32_t hi = 0;
    for (int l = 0; l < 32; ++l) {
        const long long a = sum_fixed(u[l], E);
        lo += sum_lo(a), mid += sum_mid(a), hi += sum_hi(a);
    }
    const long long b = sum_unit_bits(E);
    double unit;
    std::memcpy(&unit, &b, 8);
    return (double)sum_total(lo, mid, hi) * unit;
}
"""


@pytest.fixture(scope="module")
def total(tmp_path_factory):
    d = tmp_path_factory.mktemp("sum")
    (d / "s.cpp").write_text(SOURCE)
    out = str(d / "s.so")
    subprocess.run(["g++", "-O1", "-shared", "-fPIC", "-I", CSRC, str(d / "s.cpp"), "-o", out], check=True)
    f = ctypes.CDLL(out).total
    f.restype, f.argtypes = ctypes.c_double, [ctypes.c_void_p]
    return lambda v: f(np.ascontiguousarray(v, dtype=np.float32).ctypes.data)


def test_sums(total):
    g = np.random.default_rng(5)
    big = np.float32(3.4028235e38)
    cases = [np.zeros(32), np.full(32, big), np.full(32, -big), np.full(32, 1.4e-45), -np.arange(32) * 1.4e-45,
             np.r_[big, -big, np.full(30, 1e-45)], np.r_[1.0, -1.0, 2.0 ** -40, np.zeros(29)],
             np.r_[1.0, np.full(31, 2.0 ** -24)], np.r_[-1.0, np.full(31, 2.0 ** -33)]]
    for spread in (0, 2, 8, 20, 36):
        for _ in range(200):
            v = (g.normal(size=32) * 10.0 ** g.uniform(-spread, spread / 4, 32)).astype(np.float32)
            cases += [v, v * (g.random(32) < 0.2), np.r_[v[:16], -v[:16] * np.float32(1 + 2.0 ** -20)]]
    for v in cases:
        v = np.asarray(v, dtype=np.float32)
        exact = math.fsum(v.astype(np.float64))
        assert abs(total(v) - exact) <= 2.0 ** -53 * abs(exact) + 32 * 2.0 ** -57 * np.abs(v).max(), v
        if np.ptp(np.frexp(v[v != 0])[1]) <= 34 if (v != 0).any() else True:  # nothing is cut off: one rounding
            assert total(v) == exact, v


@pytest.mark.gpu
def test_two_gradients_of_one_channel_are_the_same():
    """Sums in a fixed order of slots: the same bits again, and finite."""
    from paper_1703_05158_gb300 import lbm

    grads = []
    for _ in range(2):
        ch = lbm.Channel(33, 9, 12, 0.6, 0.15, 1e-5, 0.04, (14, 2, 3), (15, 6, 8), 40, 21, 10,
                         X=np.array([(8.3, 4.2, 5.6)]), R=np.array([2.3]))
        ch.forward()
        grads.append(ch.backward())
        ch.close()
    assert np.all(np.isfinite(grads[0])) and np.all(grads[0] != 0)
    assert np.array_equal(*grads)
