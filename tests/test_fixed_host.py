"""Integer arithmetic of csrc/dg_fixed.cuh and csrc/dg_f32.cuh on the host: the
rounding of sums to FP64, the logarithm of a ratio, and the small-difference
series of the FP32 log means, against exact or 40-digit values."""
import ctypes
import os
import random
import subprocess

import mpmath as mp
import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2108_06476_gb300", "csrc")


def _between(text, first, last):
    i = text.index(first)
    return text[i:text.index(last, i)]


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("fxh")
    src, so = d / "fxh.cpp", d / "fxh.so"
    f32 = open(os.path.join(CSRC, "dg_f32.cuh")).read()
    series = _between(f32, "__device__ __forceinline__ unsigned long long series_term",
                      "// Q(t^2) = t/atanh(t)")
    src.write_text(r"""
#define DG_FX_HOST
#include "dg_fixed.cuh"
#define __device__
#define __forceinline__ inline
static unsigned __float_as_uint(float x) { unsigned b; __builtin_memcpy(&b, &x, 4); return b; }
static float __uint_as_float(unsigned b) { float x; __builtin_memcpy(&x, &b, 4); return x; }
""" + series + r"""
extern "C" double to_double(long long a, int e) { return dg::fx::to_double_int(a, e); }
extern "C" double ratio(double x, double y) { return dg::fx::ln_ratio(x, y); }
extern "C" int in_range(double x, double y) { return dg::fx::ln_ratio_in_range(x, y); }
extern "C" void series(float a, float b, float* r) { series_r(a, b, r[0], r[1]); }
""")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-fPIC", "-shared", "-I", CSRC,
                    str(src), "-o", str(so)], check=True)
    L = ctypes.CDLL(str(so))
    L.to_double.argtypes, L.to_double.restype = [ctypes.c_longlong, ctypes.c_int], ctypes.c_double
    L.ratio.argtypes, L.ratio.restype = [ctypes.c_double] * 2, ctypes.c_double
    L.in_range.argtypes = [ctypes.c_double] * 2
    L.series.argtypes = [ctypes.c_float] * 2 + [ctypes.POINTER(ctypes.c_float)]
    return L


def test_sums_round_to_the_nearest_double(lib):
    rng = random.Random(1)
    values = [0, 1, -1, 2 ** 53, 2 ** 53 + 1, 2 ** 54 - 1, 2 ** 62, 2 ** 63 - 1, -(2 ** 63 - 1),
              2 ** 54 + 2, 2 ** 54 + 6, 2 ** 60 - 64, 2 ** 60 - 65, 2 ** 60 - 63]
    values += [rng.getrandbits(k) * rng.choice((1, -1)) for k in range(1, 63) for _ in range(40)]
    # ties and the carry into the next power of two at every length
    values += [s * (((rng.getrandbits(52) | 1 << 52) << k) + (1 << k >> 1) + d)
               for k in range(2, 10) for s in (1, -1) for d in (-1, 0, 1)]
    values += [s * ((1 << 63) - (1 << k)) for k in range(0, 12) for s in (1, -1)]
    for a in values:
        for e in (0, -60, 37, -300, 300):
            got = lib.to_double(a, e)
            m = abs(a)
            shift = max(0, m.bit_length() - 53)
            q = (m >> shift) + (m >> (shift - 1) & 1 if shift else 0)  # ties away from zero
            ref = float(q << shift) if q else 0.0
            assert got == (-ref if a < 0 else ref) * 2.0 ** e, (a, e)


def test_logarithm_of_a_ratio(lib):
    # two significands' logarithms within 2^-53 each, and the result's rounding
    mp.mp.dps = 40
    rng = np.random.default_rng(2)
    for j in (0, 1, -1, 2, 5, 9, -9, 10, -10, 11, 40, -300, 900, -1900):
        for _ in range(60):
            x = float(rng.uniform(1, 2)) * 2.0 ** (-j // 2)
            y = float(rng.uniform(1, 2)) * 2.0 ** (-j // 2 + j)
            assert lib.in_range(x, y)
            ref = mp.log(mp.mpf(y) / mp.mpf(x))
            err = abs(mp.mpf(lib.ratio(x, y)) - ref)
            assert err <= 2.0 ** -52 + 2.0 ** -53 * abs(ref), (x, y)
    for bad in (0.0, -1.0, np.nan, np.inf, -np.inf, 5e-324, 1e305, 1e-305):
        assert not lib.in_range(bad, 1.0) and not lib.in_range(1.0, bad)


def test_small_difference_series_on_integers(lib):
    # R(a) = 1/3 + (4/45) a + O(a^2) and R(a) + (4/45) b as the branch takes
    # them, correctly rounded to FP32 but for ties (half a unit and 2^-20 of it)
    mp.mp.dps = 40
    rng = np.random.default_rng(3)
    a = np.concatenate([[0.0, 1e-45, 1e-38, 9.9999e-5], 10.0 ** rng.uniform(-30, -4, 400)])
    for x in a:
        for y in (0.0, float(rng.choice(a))):
            x32, y32 = np.float32(x), np.float32(y)
            r = (ctypes.c_float * 2)()
            lib.series(x32, y32, r)
            for got, ref in ((r[0], mp.mpf(1) / 3 + mp.mpf(4) / 45 * mp.mpf(float(x32))),
                             (r[1], mp.mpf(1) / 3
                              + mp.mpf(4) / 45 * (mp.mpf(float(x32)) + mp.mpf(float(y32))))):
                assert abs(mp.mpf(got) - ref) <= 2.0 ** -26 * (1 + 2.0 ** -20), (x, y)
