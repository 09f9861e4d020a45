"""The integer orientation code of csrc/cch_internal.cuh (63-bit and 128-bit
coordinate differences), compiled for the CPU from the source itself, against
exact rational arithmetic: collinear and nearly collinear triples whose
coordinates differ by up to 2^80 in magnitude, grids, zeros and ties."""
import ctypes
import os
import re
import shutil
import subprocess
from fractions import Fraction as F

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SHIM = r"""
#include <cstdint>
#include <cstring>
#include <algorithm>
using std::max; using std::min;
#define __device__
#define __forceinline__ inline
#define __noinline__
static long long __double_as_longlong(double d) { long long v; memcpy(&v, &d, 8); return v; }
static int __clzll(long long v) { return v ? __builtin_clzll((unsigned long long)v) : 64; }
static int __ffsll(long long v) { return __builtin_ffsll(v); }
"""
CALLS = r"""
extern "C" int narrow(const double* p, int* s) { return orient_f64_int(p[0], p[1], p[2], p[3], p[4], p[5], *s); }
extern "C" int wide(const double* p, int* s) { return orient_f64_wide(p[0], p[1], p[2], p[3], p[4], p[5], *s); }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("needs g++")
    src = open(os.path.join(ROOT, "paper_1508_05488_gb300", "csrc", "cch_internal.cuh")).read()
    a = src.index("// Exact difference of two float64 values")
    b = src.index("// FP64 filter with Shewchuk")
    d = tmp_path_factory.mktemp("orient")
    (d / "o.cpp").write_text(SHIM + re.sub(r"#pragma unroll.*", "", src[a:b]) + CALLS)
    so = str(d / "o.so")
    subprocess.run(["g++", "-O1", "-shared", "-fPIC", "-o", so, str(d / "o.cpp")], check=True)
    return ctypes.CDLL(so)


def exact(p):
    ax, ay, bx, by, cx, cy = (F(float(v)) for v in p)
    d = (ax - cx) * (by - cy) - (ay - cy) * (bx - cx)
    return (d > 0) - (d < 0)


def triples():
    rng = np.random.default_rng(12)
    for k in range(3000):
        e = rng.integers(-80, 80, 3) if k % 3 else rng.integers(-12, 12, 3)
        t = rng.random(3) * 2.0 ** e * rng.choice([-1.0, 1.0], 3)
        m, c = rng.integers(-7, 8), (0.0 if k % 2 else float(rng.integers(-4, 5)))
        p = np.stack([t, m * t + c], 1).ravel()              # collinear where the sums are exact
        yield p
        q = p.copy()
        j = int(rng.integers(0, 6))
        q[j] = np.nextafter(q[j], q[j] + rng.choice([-1.0, 1.0]))
        if q[j] == 0 or abs(q[j]) >= 2.0 ** -400:
            yield q                                          # one ulp off
        z = p.copy()
        z[rng.integers(0, 6, 2)] = 0.0
        yield z
        yield p[[0, 1, 2, 3, 0, 1]]                          # coincident points
        yield rng.integers(-5, 6, 6) * 2.0 ** float(rng.integers(-60, 60))
        yield rng.integers(0, 2 ** 53, 6) * 2.0 ** -53       # a common grid, every magnitude


def test_signs(lib):
    decided = [0, 0]
    total = 0
    for p in triples():
        p = np.ascontiguousarray(p, dtype=np.float64)
        want = exact(p)
        total += 1
        for k, f in enumerate((lib.narrow, lib.wide)):
            s = ctypes.c_int(7)
            if f(p.ctypes.data_as(ctypes.c_void_p), ctypes.byref(s)):
                decided[k] += 1
                assert s.value == want, (k, p)
    assert decided[0] > total // 5 and decided[1] > total // 2


def test_gaps_up_to_63_bits_are_decided(lib):
    s = ctypes.c_int(7)
    for g in range(0, 70):
        x = (1.0 + 2.0 ** -52) * 2.0 ** -g                   # no trailing zero
        p = np.array([x, 3.0 * 2.0 ** -g, 1.25, 1.75, -1.5, 1.125])
        ok = lib.wide(p.ctypes.data_as(ctypes.c_void_p), ctypes.byref(s))
        assert bool(ok) == (g <= 62) or g == 63, g
        if ok:
            assert s.value == exact(p)
