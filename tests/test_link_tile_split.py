"""The link kernel splits a node index t < B^3 of a sphere's cube into (x, y, z)
and a row index r < B^2 into (y, z) by multiplying with 2^32 / B^2 + 1 and
2^32 / B + 1 and taking the high word.  The quotients are checked for every
index of every cube a radius the ABI takes can have (B = 2 e + 4, e = ceil(R) =
1 .. 16), against the constants and bounds of the source."""
import os
import re

import numpy as np

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1703_05158_gb300", "csrc")


def test_splits_are_exact_for_every_cube():
    src = open(os.path.join(CSRC, "lbm_links.cuh")).read()
    assert src.count("lo(-e - 1), B(2 * e + 4)") == 1 and src.count("B = 2u * (unsigned)e + 4u;") == 1
    assert re.search(r"e = min\(ext, \(int\)ceilf\(Fr\.R\)\)", src)
    assert "0xFFFFFFFFu / B + 1u, 0xFFFFFFFFu / (B * B) + 1u" in src
    assert "z = (int)__umulhi((unsigned)r, mB);" in src and "z = (int)__umulhi((unsigned)t, mB2);" in src
    high = np.uint64(32)
    for e in range(1, 17):
        B = 2 * e + 4
        assert B <= 36 and B ** 3 <= 1 << 16  # row masks of 64 bits, node indexes of 16, coordinates of 6
        mB, mB2 = (np.uint64(0xFFFFFFFF // d + 1) for d in (B, B * B))
        t = np.arange(B ** 3, dtype=np.uint64)
        z = (t * mB2) >> high
        assert np.array_equal(z, t // np.uint64(B * B))
        r = t - z * np.uint64(B * B)
        assert np.array_equal((r * mB) >> high, r // np.uint64(B))
        # the row loop also splits the rows past the last one of its block (at most 255 of them)
        r = np.arange(B * B + 256, dtype=np.uint64)
        assert np.array_equal((r * mB) >> high, r // np.uint64(B))
