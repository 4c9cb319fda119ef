"""The FP64 normals at the edges of their tables: the first and last values of the radius' segments (every
power of two of u and of 1 - u, the segments of one value below 2^9), the middle where the two sides meet,
and the ends of the angle's quadrants and sub-ranges; against the oracle's Box-Muller."""
import numpy as np
import pytest

import oracle
from paper_1808_05168_gb300 import capi

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("side", ["u", "1-u"])
def test_table_edges(side):
    # q = 2 k + 1 counts u (or 1 - u) in units of 2^-24
    edges = {1, 3, 255, 257, 509, 511, 513, 515}
    for e in range(9, 24):
        for s in (0, 1, 2, 127, 128, 255, 256):  # segment starts of the octave [2^e, 2^(e+1))
            for d in (-3, -1, 1, 3):
                edges.add((1 << e) + (s << max(e - 8, 0)) + d)
    q = np.array(sorted(v for v in edges if 0 < v < 1 << 23 and v % 2), dtype=np.int64)
    m = q if side == "u" else (1 << 24) - q
    angle = {1, 3, (1 << 24) - 1}
    for a in range(1, 16):
        angle |= {(a << 20) + d for d in (-1, 1)}
    for a in range(0, 4096, 97):
        angle |= {(a << 12) + d for d in (1, 4095)}
    n = np.array(sorted(angle), dtype=np.int64)
    words = np.empty((m.size, n.size, 2), np.uint32)
    words[..., 0] = ((m - 1) // 2)[:, None]
    words[..., 1] = ((n - 1) // 2)[None, :]
    words = words.reshape(-1)
    got = capi.lb_debug_box_muller(capi.LB_PREC_FP64, words)
    want = oracle.box_muller(words)
    # both round their radius (at most 5.8: half a unit is 4.4e-16) and their sine and cosine (half a unit
    # 5.6e-17, times the radius 3.2e-16) a few times: 4e-15 covers five roundings of each on both sides
    assert np.max(np.abs(got - want)) < 4e-15
