"""Kernels that may start while the one before them is still writing (chained launches) must not
read its results through the non-coherent path: that path is for data which nobody writes while
the kernel lives.  Checked on the sources, as no run shows the difference reliably."""
import os
import re

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
