"""hi + lo of two floats as binary64 bits in integer arithmetic (csrc/convert.cuh, the
finishing pass of the tensor-core forms) against the host's double addition."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1906_08148_gb300", "csrc")


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = str(tmp_path_factory.mktemp("pair"))
    src, so = os.path.join(d, "shim.cpp"), os.path.join(d, "libshim.so")
    with open(src, "w") as f:
        f.write('#include "convert.cuh"\n'
                'extern "C" void pair(const uint32_t* h, const uint32_t* l, int64_t n, uint64_t* out, uint8_t* ok) {\n'
                "  for (int64_t i = 0; i < n; ++i) {\n"
                "    ok[i] = f32_pair_sum_covers(h[i], l[i]);\n"
                "    out[i] = ok[i] ? f32_pair_sum_bits(h[i], l[i]) : 0;\n"
                "  }\n"
                "}\n")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-I", CSRC, "-o", so, src])
    L = ctypes.CDLL(so)
    L.pair.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int64, ctypes.c_void_p, ctypes.c_void_p]
    return L


def test_pair_sum_equals_double_addition(lib):
    rng = np.random.default_rng(9)
    n = 1000000
    u32 = lambda x: x.astype(np.uint32)
    h = u32(rng.integers(0, 1 << 32, n, dtype=np.uint64))
    e = (h >> 23) & 0xFF
    # the other float: near in exponent, the same or opposite, zero of either sign, or anything
    near = u32(np.clip(e.astype(np.int64) - rng.integers(-32, 33, n), 0, 255))
    l = (u32(rng.integers(0, 2, n)) << 31) | (near << 23) | u32(rng.integers(0, 1 << 23, n))
    k = rng.random(n)
    l = np.select([k < 0.05, k < 0.1, k < 0.2, k < 0.25, k < 0.27],
                  [h, h ^ np.uint32(1 << 31), np.uint32(0), u32(rng.integers(0, 1 << 32, n, dtype=np.uint64)),
                   np.uint32(1 << 31)], l)
    swap = rng.random(n) < 0.3  # lo the larger of the two
    h, l = u32(np.where(swap, l, h)), u32(np.where(swap, h, l))
    out, ok = np.zeros(n, np.uint64), np.zeros(n, np.uint8)
    lib.pair(h.ctypes.data, l.ctypes.data, n, out.ctypes.data, ok.ctypes.data)
    with np.errstate(invalid="ignore", over="ignore"):
        want = (h.view(np.float32).astype(np.float64) + l.view(np.float32).astype(np.float64)).view(np.uint64)
    at = ok.astype(bool)
    assert np.array_equal(out[at], want[at])
    # what is left to the FP64 addition: a subnormal, Inf or NaN, or exponents more than 28 apart
    eh, el = ((h >> 23) & 255).astype(int), ((l >> 23) & 255).astype(int)
    mh, ml = h & np.uint32(0x7FFFFFFF), l & np.uint32(0x7FFFFFFF)
    big, small = np.maximum(mh, ml) >> 23, np.minimum(mh, ml)
    covered = (big > 0) & (big < 255) & ((small == 0) | ((small >> 23 > 0) & (np.abs(eh - el) <= 28)))
    assert np.array_equal(at, covered) and at.mean() > 0.5
