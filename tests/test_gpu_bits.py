"""The bits of z: a replay rounds to bf16 after each of its steps, so a late joiner ends with
the weights of those that trained on only if every z keeps its bits from build to build (the
parity tests allow 1e-6). Fingerprints of the transform's outputs over every radius word and
every angle word, the other word of the pair mixed; the same from the present form of the
transform (bits placed under exponents) and the one before it (integer conversions and an
octant reflection). A change of one bit of one output changes them."""
import ctypes

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FINGERPRINTS = {"radius": 0x76DB13A66ED10ED8, "angle": 0x7C499EBDB9F880C0}


@pytest.fixture(scope="module")
def jb():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2306_10015_gb300 import build
    build.build()
    import paper_2306_10015_gb300 as pkg
    pkg.lib()
    return pkg


def fingerprint(jb, which):
    i = torch.arange(1 << (23 if which == "radius" else 24), device="cuda", dtype=torch.int64)
    mixed = (i * 0x9E3779B1 + (i >> 7) * 0x85EBCA77) & 0xFFFFFFFF
    radius, angle = (i << 9 | mixed & 511, mixed) if which == "radius" else (mixed, i << 8 | mixed & 255)
    words = torch.stack([radius, angle], dim=1).contiguous()
    words = torch.where(words >= 1 << 31, words - (1 << 32), words).to(torch.int32)
    z = torch.empty(2 * i.numel(), device="cuda", dtype=torch.float32)
    stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    assert jb.lib().jb_debug_box_muller(words.data_ptr(), i.numel(), z.data_ptr(), stream) == 0
    place = torch.arange(z.numel(), device="cuda", dtype=torch.int64)
    return int((z.view(torch.int32).to(torch.int64) * (2 * place + 1)).sum().item()) & (2**64 - 1)


@pytest.mark.parametrize("which", ["radius", "angle"])
def test_bits_of_the_transform(jb, which):
    assert fingerprint(jb, which) == FINGERPRINTS[which], hex(fingerprint(jb, which))
