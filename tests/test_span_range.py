"""The range within which the direct-load kernel takes some of its exponentials on the FMA pipe, from the
functions it calls, over every bf16 reference it may have."""
import ctypes as C
import math
import os
import subprocess

import numpy as np

from conftest import ROOT

SOURCE = """
#include "ssd_ranges.cuh"
extern "C" unsigned lo(float m) { return ssd::ranges::bf16_floor(m); }
extern "C" unsigned hi(float m) { return ssd::ranges::bf16_ceiling(m); }
extern "C" float limit() { return ssd::ranges::kSpanSumLimit; }
"""


def test_floor_and_ceiling_of_every_reference(tmp_path):
    (tmp_path / "b.cpp").write_text(SOURCE)
    so = str(tmp_path / "b.so")
    subprocess.run([os.environ.get("CXX", "g++"), "-std=c++17", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_2603_11243_b200", "csrc"), str(tmp_path / "b.cpp"), "-o", so], check=True)
    lib = C.CDLL(so)
    lib.lo.argtypes = lib.hi.argtypes = [C.c_float]
    lib.lo.restype = lib.hi.restype = C.c_uint
    lib.limit.restype = C.c_float
    values = (np.arange(1 << 16, dtype=np.uint32) << 16).view(np.float32)
    as_float = lambda bits: float(np.array([bits << 16], np.uint32).view(np.float32)[0])
    least = math.inf
    for m in values[np.isfinite(values) & (np.abs(values) < 4096)]:
        m = float(m)
        below, above = m - as_float(lib.lo(m)), as_float(lib.hi(m)) - m
        # m - 85 and m + 85 are fp32: half an ulp at 4,181
        assert 64.0 <= below <= 85.0 + 2.0 ** -12 and 64.0 <= above <= 85.0 + 2.0 ** -12, m
        least = min(least, below, above)
    assert least == 64.0
    # a clamped exponential alone takes the sum over the limit, with room for the polynomial's error
    assert math.exp(least) * (1 - 1e-6) > 2 * lib.limit()
    # a million terms at their floor do not show beside the reference's own 1
    assert 1e6 * math.exp(-least) < 2.0 ** -25
