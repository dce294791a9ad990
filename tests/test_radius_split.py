"""The split u_a = 2^e f, f in [3/4, 3/2), of the Box-Muller radius over all 2^23 radius words.

The kernels take e and the scale of f from the exponent of (8/3)(u_a / 2), rounded to fp32
(jb_rng.cuh, polar2). Here the same steps in numpy's fp32 against frexp in 64 bits. Every
step but that product is exact, so equality is the bound.
"""
import numpy as np


def test_exponent_of_four_thirds_u():
    i = np.arange(1 << 23, dtype=np.uint32)
    u = (np.uint32(0x3F000000) | i).view(np.float32) - np.float32(float.fromhex("0x1.fffffep-2"))
    ua = (i.astype(np.float64) + 0.5) * 2.0**-23
    assert np.array_equal(u.astype(np.float64), ua / 2)

    m, x = np.frexp(ua)                      # ua = m 2^x, m in [1/2, 1)
    e = np.where(m >= 0.75, x, x - 1)        # f = m 2^(x - e) in [3/4, 3/2)
    h = (u * np.float32(float.fromhex("0x1.555556p+1"))).view(np.uint32)
    got = (np.uint32(0x4B000000) | (h >> np.uint32(23))).view(np.float32) - np.float32(8388735.0)
    assert np.array_equal(got.astype(np.int64), e)

    scale = (~h & np.uint32(0x7F800000)).view(np.float32)
    t = u.astype(np.float64) * scale.astype(np.float64) - 1.0
    assert np.array_equal(t, np.ldexp(ua, -e) - 1.0)
    assert np.array_equal(t.astype(np.float32).astype(np.float64), t)  # exact in fp32
