"""Rules of the kernel sources that no run shows to be broken reliably.

Kernels that may start while the one before them is still writing (chained launches) must not
read its results through the non-coherent path: that path is for data which nobody writes while
the kernel lives.  Words made of a float's bits are multiplied without a sign, as they exceed 32 bits."""
import ctypes
import os
import re
import subprocess

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


def test_work_is_planned_before_the_next_kernel_is_let_in():
    """plan_kernel is short and follows the transforms of the responses: it lets the convolution's CTAs in when these
    have ended, not while the waiting ones would take their places."""
    s = source("conv.cu")
    body = s[s.index("plan_kernel(const __grid_constant__"):]
    body = body[: body.index("\n}")]
    assert body.index("chain_wait();") < body.index("chain_next();")


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


def test_distance_of_an_image_is_right_to_its_last_bits(tmp_path):
    """The header's arithmetic, compiled for the host, from seeds two units off either way (what the fp32 reciprocal
    square root may be): two roundings and that of the reference."""
    src = tmp_path / "distance.cpp"
    src.write_text('#include "image_delay.cuh"\n'
                   'extern "C" void distances(const double *d2, const float *r0, double *d, double *e, int n) {\n'
                   '    for (int i = 0; i < n; ++i) d[i] = image_distance(d2[i], r0[i], e[i]);\n}\n')
    so = str(tmp_path / "distance.so")
    subprocess.run(["g++", "-O2", "-ffp-contract=off", "-shared", "-fPIC", "-I", CSRC, "-o", so, str(src)], check=True)
    rng = np.random.default_rng(0)
    d2 = np.repeat(np.exp(rng.uniform(np.log(1e-4), np.log(1e6), 20000)), 5)
    r0 = (1 / np.sqrt(d2)).astype(np.float32)
    r0 = (r0.view(np.int32) + np.tile(np.arange(-2, 3, dtype=np.int32), 20000)).view(np.float32)
    d, e = np.empty_like(d2), np.empty_like(d2)
    p = lambda a, t: a.ctypes.data_as(ctypes.POINTER(t))
    ctypes.CDLL(so).distances(p(d2, ctypes.c_double), p(r0, ctypes.c_float), p(d, ctypes.c_double),
                              p(e, ctypes.c_double), len(d2))
    assert np.max(np.abs(d / np.sqrt(d2) - 1)) <= 3 * np.finfo(np.float64).eps
    assert np.max(np.abs(r0 * (1 + e / 2) * np.sqrt(d2) - 1)) <= np.max(np.abs(e)) ** 2
