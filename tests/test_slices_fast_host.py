"""The 32-bit digit form of the BF16 split (csrc/slices.cuh, S = 3 and 4) equals the
general 64-bit form on every kind of input, and the two-at-a-time conversion equals the
single one; compiled for the host."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1906_08148_gb300", "csrc")


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = str(tmp_path_factory.mktemp("slices"))
    src, so = os.path.join(d, "shim.cpp"), os.path.join(d, "libshim.so")
    with open(src, "w") as f:
        f.write('#include "slices.cuh"\n'
                'extern "C" {\n'
                "int64_t differ(int S, const uint64_t* b, const int* emax, int64_t n) {\n"
                "  int64_t bad = 0;\n"
                "  for (int64_t i = 0; i < n; ++i) {\n"
                "    int32_t x[4] = {0, 0, 0, 0}, y[4] = {0, 0, 0, 0};\n"
                "    if (S == 3) { slice_digits<3>(b[i], emax[i], x); slice_digits_wide<3>(b[i], emax[i], y); }\n"
                "    else { slice_digits<4>(b[i], emax[i], x); slice_digits_wide<4>(b[i], emax[i], y); }\n"
                "    for (int s = 0; s < S; ++s) bad += x[s] != y[s];\n"
                "  }\n"
                "  return bad;\n"
                "}\n"
                "int64_t differ_x2() {\n"
                "  int64_t bad = 0;\n"
                "  for (int p = -140; p <= 20; ++p)\n"
                "    for (int d = -256; d <= 256; ++d) {\n"
                "      const uint32_t two = slice_bf16_x2(d, -d, slice_unit(p));\n"
                "      const uint32_t a = slice_bf16_bits(d, p), b = slice_bf16_bits(-d, p);\n"
                "      const uint32_t m = p < -126 ? 0x7FFFu : 0xFFFFu;  // a dropped digit: a zero of either sign\n"
                "      bad += ((two & 0xFFFFu) & m) != a || ((two >> 16) & m) != b;\n"
                "    }\n"
                "  return bad;\n"
                "}\n"
                "}\n")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-I", CSRC, "-o", so, src])
    L = ctypes.CDLL(so)
    L.differ.argtypes = [ctypes.c_int, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int64]
    L.differ.restype = ctypes.c_int64
    L.differ_x2.restype = ctypes.c_int64
    return L


@pytest.mark.parametrize("S", [3, 4])
def test_narrow_digits_equal_wide_digits(lib, S):
    rng = np.random.default_rng(S)
    n = 400000
    E = rng.integers(0, 2047, n)
    frac = rng.integers(0, 1 << 52, n, dtype=np.uint64)
    # mantissas whose digits sit on the ties of balancing and rounding, and at the ends
    at = rng.random(n) < 0.5
    ones = (np.uint64(1) << rng.integers(0, 52, n).astype(np.uint64)) - np.uint64(1)
    frac[at] = np.where(rng.random(at.sum()) < 0.5, ones[at], np.uint64(0xFFFFFFFFFFFFF) ^ ones[at])
    tie = rng.random(n) < 0.2
    frac[tie] = (rng.integers(0, 1 << 6, tie.sum()).astype(np.uint64) << np.uint64(46)) | (
        np.uint64(1) << rng.integers(0, 52, tie.sum()).astype(np.uint64))
    b = (rng.integers(0, 2, n).astype(np.uint64) << np.uint64(63)) | (E.astype(np.uint64) << np.uint64(52)) | frac
    # the line's largest exponent: from the element's own to far above it
    emax = np.minimum(E + np.where(rng.random(n) < 0.8, rng.integers(0, 60, n), rng.integers(0, 2046, n)), 2046)
    b, emax = np.ascontiguousarray(b), np.ascontiguousarray(emax.astype(np.int32))
    assert lib.differ(S, b.ctypes.data, emax.ctypes.data, n) == 0


def test_two_at_a_time_conversion(lib):
    assert lib.differ_x2() == 0
