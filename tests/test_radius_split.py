"""The split u_a = 2^e f, f in [3/4, 3/2), of the Box-Muller radius over all 2^23 radius words.

The kernels take e and the scale of f from the exponent of (8/3)(u_a / 2), rounded to fp32
(jb_rng.cuh, polar2). Here the same steps in numpy's fp32, with the constants read from the
kernel's source, against frexp in 64 bits. Every step but that product is exact, so equality
is the bound.
"""
import os
import re

import numpy as np

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def steps():
    """The radius's steps in polar2, in order, with their constants."""
    with open(os.path.join(ROOT, "paper_2306_10015_gb300", "csrc", "jb_rng.cuh")) as f:
        text = re.sub(r"//[^\n]*", "", f.read())
    body = "".join(text[text.index("Polar2 polar2(uint4 w)"):].split())
    number = r"([-+0-9a-fx.p]+)f"
    found = re.search(
        r"float2u=add2\(make_float2\(shift_under\((0x[0-9A-F]+)u,w\.x,(\d+)\),shift_under\(\1u,w\.z,\2\)\),splat\(" + number +
        r"\)\);constfloat2v=mul2\(u,splat\(" + number + r"\)\);"
        r"constuint32_thA=__float_as_uint\(v\.x\),hB=__float_as_uint\(v\.y\);"
        r"constfloat2e=add2\(make_float2\(shift_under\((0x[0-9A-F]+)u>>(\d+),hA,(\d+)\),"
        r"shift_under\(\5u>>\6,hB,\7\)\),splat\(" + number + r"\)\);"
        r"constfloat2t=fma2\(u,make_float2\(__uint_as_float\(~hA&(0x[0-9A-F]+)u\),"
        r"__uint_as_float\(~hB&\9u\)\),splat\(" + number + r"\)\);", body)
    assert found, "polar2 forms the radius by other steps than these"
    real = lambda s: np.float32(float.fromhex(s) if "x" in s else float(s))
    g = found.groups()
    return {"under_u": int(g[0], 16), "shift_u": int(g[1]), "less_u": real(g[2]), "scale": real(g[3]),
            "under_e": int(g[4], 16) >> int(g[5]), "shift_e": int(g[6]), "less_e": real(g[7]),
            "mask": int(g[8], 16), "less_t": real(g[9])}


def shift_under(hi, lo, n):
    """The low word of hi : lo shifted right by n."""
    return ((np.uint64(hi) << np.uint64(32) | lo.astype(np.uint64)) >> np.uint64(n)).astype(np.uint32).view(np.float32)


def test_exponent_of_four_thirds_u():
    k = steps()
    i = np.arange(1 << 23, dtype=np.uint32)
    u = shift_under(k["under_u"], i << np.uint32(9) | i & np.uint32(511), k["shift_u"]) + k["less_u"]
    ua = (i.astype(np.float64) + 0.5) * 2.0**-23
    assert np.array_equal(u.astype(np.float64), ua / 2)

    m, x = np.frexp(ua)                      # ua = m 2^x, m in [1/2, 1)
    e = np.where(m >= 0.75, x, x - 1)        # f = m 2^(x - e) in [3/4, 3/2)
    h = (u * k["scale"]).view(np.uint32)
    got = shift_under(k["under_e"], h, k["shift_e"]) + k["less_e"]
    assert np.array_equal(got.astype(np.int64), e)

    scale = (~h & np.uint32(k["mask"])).view(np.float32)
    t = u.astype(np.float64) * scale.astype(np.float64) + np.float64(k["less_t"])
    assert np.array_equal(t, np.ldexp(ua, -e) - 1.0)
    assert np.array_equal(t.astype(np.float32).astype(np.float64), t)  # exact in fp32
