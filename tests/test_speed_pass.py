"""The wave-speed passes' decision to pass over an element (csrc/dg_device.cuh
`speed_skip`): the kernels go on with full-warp shuffles, so all lanes of a warp
have to decide alike, although each reads the running maximum for itself while
other warps raise it. Shown on the host: the function with the lanes of a warp
one after another, the votes collected first.
"""
import ctypes
import itertools
import os
import re
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2108_06476_gb300", "csrc")


def _text(name):
    return open(os.path.join(CSRC, name)).read()


def _function(text, head):
    i = text.index(head)
    depth = 0
    for j in range(text.index("{", i), len(text)):
        depth += {"{": 1, "}": -1}.get(text[j], 0)
        if not depth:
            return text[i:j + 1]


@pytest.mark.parametrize("name,kernel", [("dg_api.cu", "__global__ void speed_kernel("),
                                         ("dg_mhd.cu", "__global__ void mhd_speed_kernel("),
                                         ("dg_ensemble.cu",
                                          "__global__ void ensemble_speed_kernel(")])
def test_the_passes_leave_an_element_by_the_vote_only(name, kernel):
    body = re.sub(r"//[^\n]*", "", _function(_text(name), kernel))
    skips = [s.strip() for s in re.split(r"[;{}]", body) if s.strip().endswith("continue")]
    assert len(skips) == body.count("continue;") > 0
    assert all(re.match(r"if \((dg::)?speed_skip\(", s) for s in skips), skips


def test_all_lanes_decide_alike(tmp_path):
    src, so = tmp_path / "skip.cpp", tmp_path / "skip.so"
    src.write_text(r"""
#define __device__
#define __forceinline__ inline
static bool collecting, agreed;
static bool vote(bool p) { if (collecting) agreed = agreed && p; return agreed; }
#define __all_sync(mask, p) vote(p)
static float d2f(double x) { return (float)x; }
""" + _function(_text("dg_device.cuh"), "__device__ __forceinline__ bool speed_skip(") + r"""
extern "C" int decide(const int* fine, float bound, const double* most) {
  int n = 0;
  agreed = true;
  for (int pass = 0; pass < 2; ++pass) {
    collecting = pass == 0;
    n = 0;
    for (int i = 0; i < 32; ++i) n += speed_skip(fine[i], bound, most[i]);
  }
  return n;  // the lanes that pass over the element
}
""")
    subprocess.run(["g++", "-O1", "-fPIC", "-shared", str(src), "-o", str(so)], check=True)
    lib = ctypes.CDLL(str(so))

    def decide(fine, bound, most):
        return lib.decide((ctypes.c_int * 32)(*fine), ctypes.c_float(bound),
                          (ctypes.c_double * 32)(*most))

    assert decide([1] * 32, 1.0, [2.0] * 32) == 32
    assert decide([1] * 32, 2.0, [1.0] * 32) == 0
    # lanes that read the maximum before and after another warp raised it
    for k in range(32):
        assert decide([1] * 32, 1.5, [2.0] * k + [1.0] * (32 - k)) in (0, 32)
        assert decide([1] * 32, 1.5, [1.0] * k + [2.0] * (32 - k)) in (0, 32)
    assert decide([1] * 31 + [0], 1.0, [2.0] * 32) == 0
    assert decide([1] * 32, float("nan"), [2.0] * 32) == 0


def test_the_bound_holds_wherever_it_is_used(tmp_path):
    # speed_bound on the host (FP32 with subnormals, as on the device) against
    # 40-digit wave speeds, over every size of state that it accepts
    mp = pytest.importorskip("mpmath")
    mp.mp.dps = 40
    src, so = tmp_path / "bound.cpp", tmp_path / "bound.so"
    body = _function(_text("dg_device.cuh"), "__device__ __forceinline__ bool speed_bound(")
    src.write_text(r"""
#include <cmath>
using std::fabs;
#define __device__
#define __forceinline__ inline
static float d2f(double x) { return (float)x; }
template <int D>
""" + body + r"""
extern "C" int bound(const double* c, double gamma, float* lam) {
  return speed_bound<3>(c, gamma, gamma - 1.0, lam);
}
""")
    subprocess.run(["g++", "-O1", "-ffp-contract=off", "-fPIC", "-shared", str(src), "-o",
                    str(so)], check=True)
    lib = ctypes.CDLL(str(so))
    used = 0
    for rho, prel, mach, gamma in itertools.product(
            (1e-29, 1e-10, 1.0, 1e10, 1e22, 9e29), (1e-50, 1e-44, 1e-38, 1e-29, 1e-12, 1.0, 1e12),
            (0.0, 1e-2, 0.7, 3.0), (1.4, 5.0 / 3.0)):
        p = prel * rho
        cs = (gamma * prel) ** 0.5
        v = [mach * cs * s for s in (1.0, -0.5, 0.25)]
        c = [rho, *(rho * x for x in v), p / (gamma - 1.0) + 0.5 * rho * sum(x * x for x in v)]
        lam = (ctypes.c_float * 3)(0.0, 0.0, 0.0)
        if not lib.bound((ctypes.c_double * 5)(*c), ctypes.c_double(gamma), lam):
            continue
        used += 1
        m = [mp.mpf(x) for x in c]
        pe = (mp.mpf(gamma) - 1) * (m[4] - sum(x * x for x in m[1:4]) / m[0] / 2)
        ce = mp.sqrt(mp.mpf(gamma) * pe / m[0])
        for k in range(3):
            assert lam[k] >= abs(m[1 + k] / m[0]) + ce, (rho, prel, mach, gamma, k)
    assert used > 60
