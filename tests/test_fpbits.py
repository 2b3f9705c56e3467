"""The double-single conversion of an int64 (csrc/fpbits.h ds_of_i64, the epilogue of the (T) products) compiled
for the host, against exact integers: rounding carries and ties, signs, small and missing rests, the ends of the
FP32 range."""
import ctypes
import os
import random
import shutil
import subprocess
from fractions import Fraction

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2004_03682_gb300", "csrc")

SHIM = r"""
#include <cmath>
#include <cstdint>
#include <cstring>
#include <algorithm>
using std::max;
#define __device__
#define __forceinline__ inline
#define __noinline__
struct float2 { float x, y; };
static inline float2 make_float2(float x, float y) { return {x, y}; }
template <typename T, typename F> static T bits(F f) { T t; memcpy(&t, &f, sizeof t); return t; }
static inline int __clzll(long long x) { return x ? __builtin_clzll((unsigned long long)x) : 64; }
static inline float __uint_as_float(unsigned u) { return bits<float>(u); }
static inline unsigned __float_as_uint(float f) { return bits<unsigned>(f); }
static inline double __longlong_as_double(long long v) { return bits<double>(v); }
static inline long long __double_as_longlong(double d) { return bits<long long>(d); }
static inline float __int2float_rn(int i) { return float(i); }
static inline float __double2float_rn(double d) { return float(d); }
static inline float __fmul_rn(float a, float b) { return a * b; }
static inline float __fadd_rn(float a, float b) { return a + b; }
static inline float __fsub_rn(float a, float b) { return a - b; }
static inline float __fmaf_rn(float a, float b, float c) { return fmaf(a, b, c); }
#include "fpbits.h"
extern "C" void of_i64(long long R, int e, float* o) { const float2 x = ds_of_i64(R, e); o[0] = x.x; o[1] = x.y; }
extern "C" void of_f64(double d, float* o) { const float2 x = ds_split(d); o[0] = x.x; o[1] = x.y; }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("fpbits")
    (d / "shim.cpp").write_text(SHIM)
    subprocess.run([gxx, "-O1", "-std=c++17", "-fPIC", "-shared", "-ffp-contract=off", "-I", CSRC, "-o", str(d / "shim.so"),
                    str(d / "shim.cpp")], check=True)
    return ctypes.CDLL(str(d / "shim.so"))


def _call(f, *args):
    out = (ctypes.c_float * 2)()
    f(*args, out)
    return out[0], out[1]


def _nearest24(R):
    """|R| rounded to 24 bits, ties to even, with its sign."""
    m = abs(R)
    s = max(m.bit_length() - 24, 0)
    q, rest = m >> s, m & ((1 << s) - 1)
    if s and (2 * rest > 1 << s or (2 * rest == 1 << s and q & 1)):
        q += 1
    return (q << s) * (1 if R >= 0 else -1)


def _values():
    rng = random.Random(5)
    for w in range(1, 64):
        for _ in range(20):
            yield rng.getrandbits(w) | 1 << (w - 1)
        yield (1 << w) - 1  # rounds up to a power of two from 25 bits on
    for s in range(1, 40):
        for q in (0x800000, 0x800001, 0xFFFFFE, 0xFFFFFF):
            for d in (-1, 0, 1, 300, 511, 512, 513):  # around ties, and rests near nothing
                for base in ((q << s) + (1 << (s - 1)), q << s):
                    if 0 < base + d < 1 << 63:
                        yield base + d
    yield (1 << 63) - 1


def test_int64_to_double_single(lib):
    for m in _values():
        for R in (m, -m):
            for e in (0, -100, 37):
                h, lo = _call(lib.of_i64, ctypes.c_longlong(R), e)
                x, two = Fraction(R) * Fraction(2) ** e, Fraction(2) ** e
                assert Fraction(h) == _nearest24(R) * two, (R, e)
                # the rest to 24 bits, or to 2^-54 of R where that is more
                assert abs(x - Fraction(h) - Fraction(lo)) <= abs(x) / 2 ** 48, (R, e)
                if abs(R) < 1 << 53:
                    assert (h, lo) == _call(lib.of_f64, ctypes.c_double(R * 2.0 ** e)), (R, e)
    assert _call(lib.of_i64, ctypes.c_longlong(-1 << 63), 0) == (-2.0 ** 63, 0.0)
    assert _call(lib.of_i64, ctypes.c_longlong(0), 5) == (0.0, 0.0)


def test_ends_of_the_fp32_range(lib):
    inf = float("inf")
    for s in (1, -1):
        at = lambda R, e: _call(lib.of_i64, ctypes.c_longlong(s * R), e)  # noqa: E731
        assert at(1, -126) == (s * 2.0 ** -126, 0.0)
        for R, e in ((1, -127), (3, -128), ((1 << 62) + 1, -189), (5, -1000)):  # below the normal range
            assert at(R, e) == (0.0, 0.0)
        h, lo = at((1 << 30) + 1, -150)  # a rest below the normal range is dropped
        assert (h, lo) == (s * 2.0 ** -120, 0.0)
        assert at(0xFFFFFF, 104) == (s * float(0xFFFFFF) * 2.0 ** 104, 0.0)  # the largest
        for R, e in ((1, 128), (1 << 62, 66), (3, 4000), ((1 << 25) - 1, 103), ((1 << 62) - 1, 66)):
            assert at(R, e) == (s * inf, 0.0)  # beyond it, or rounded up beyond it
