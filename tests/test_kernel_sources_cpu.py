"""Rules of the kernel sources that no run shows to be broken reliably.

Kernels that may start while the one before them is still writing (chained launches) must not
read its results through the non-coherent path: that path is for data which nobody writes while
the kernel lives.  Words made of a float's bits are multiplied without a sign, as they exceed 32 bits."""
import os
import re

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1912_11040_b200", "csrc")

# parameters that a kernel running beside the start of this one may write
WRITTEN_BEFORE = [("conv.cu", "rir_length_kernel", ["rir"]),
                  ("conv.cu", "rir_spectra2_kernel", ["rir", "leff"]),
                  ("conv.cu", "plan_kernel", ["leff", "leff_all"]),
                  ("conv.cu", "convolve_kernel", ["plans", "units", "n_units", "drawn", "hspec"]),
                  ("conv.cu", "snr_gain_kernel", ["energy"]),
                  ("conv.cu", "mix_kernel", ["ys", "vv", "gain"]),
                  ("feat.cu", "frames_kernel", ["in_a", "in_b", "gain"]),
                  ("feat.cu", "logmel_kernel", ["melw", "melstart"])]


def source(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", text, flags=re.S)


@pytest.mark.parametrize("name,kernel,params", WRITTEN_BEFORE)
def test_results_of_the_kernel_before_are_read_coherently(name, kernel, params):
    m = re.search(r"__global__[^;{]*?\b" + kernel + r"\s*\(([^{]*)\)\s*\{", source(name))
    assert m, kernel
    decl = [d.strip() for d in re.sub(r"\s+", " ", m.group(1)).split(",")]
    for p in params:
        d = [x for x in decl if re.search(r"\b" + p + r"$", x)]
        assert len(d) == 1, (kernel, p)
        assert "__restrict__" not in d[0], d[0]


def test_explicit_non_coherent_loads_are_of_constant_data():
    """Inline non-coherent loads only where the audio is read, __ldg only of audio and twiddles."""
    s = source("conv.cu")
    body = s[s.index("void load_segment("):s.index("struct Bins")]
    assert s.count("ld.global.nc") == body.count("ld.global.nc")
    for m in re.finditer(r"__ldg\(([^)]*)\)", s.replace(body, "")):
        assert "tw[" in m.group(1), m.group(0)


def test_bits_of_floats_are_multiplied_without_a_sign():
    """Rounding of loud taps: 16 times the bits of about 1.5 2^23 wraps, which only unsigned words may."""
    assert not re.search(r"\*\s*__float_as_int|__float_as_int\([^)]*\)\s*\*", source("rir.cu"))
    rng = np.random.default_rng(0)
    v = np.concatenate([rng.uniform(-1, 1, 100000) * 2.0 ** 25, [2.0 ** 25, -2.0 ** 25, 2.0 ** 22, -2.0 ** 22, 0.5, 0.0]])
    v = v.astype(np.float32)
    magic = np.float32(1.5 * 2.0 ** 23)
    f32 = lambda x: x.astype(np.float32)                       # the kernel's fused operations: one rounding each
    hi = f32(v.astype(np.float64) / 16 + magic)
    lo = f32(f32(f32(magic - hi).astype(np.float64) * 16 + v) + magic)
    bits = lambda x: x.view(np.uint32)
    with np.errstate(over="ignore"):
        got = (np.uint32(16) * bits(hi) + bits(lo) - np.uint32(17 * 0x4B400000 % 2 ** 32)).view(np.int32)
    assert np.array_equal(got, np.rint(v.astype(np.float64)).astype(np.int32))
