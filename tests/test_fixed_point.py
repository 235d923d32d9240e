"""The fixed-point two-point flux (csrc/dg_fixed.cuh).

The header's arithmetic is plain integer code, so it is compiled for the host
and compared with the flux's formula in 40-digit arithmetic over the whole
range of states that it accepts: density and energy ratios through every range
of the logarithmic means, velocities from far below to far above the sound
speed, zero velocities, units of any size, and isobaric pairs (where the
largest density times the largest internal energy exceeds the pressure by the
density ratio). The bar is FP64's own: an error of a few units of 2^-53 of each
flux's natural size. On the GPU, meshes whose elements lie inside and outside
the accepted range are compared with the oracle.
"""
import ctypes
import itertools
import subprocess

import mpmath as mp
import numpy as np
import pytest

import os

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2108_06476_gb300", "csrc")
GAMMA = 1.4

SHIM = r"""
#define DG_FX_HOST
#include "dg_fixed.cuh"
using namespace dg::fx;
static unsigned hi(double x) { return (unsigned)(dbits(x) >> 32); }
// a, b: rho, e, p, v1, v2, v3; f: the flux; returns whether the pair's scale
// (that of an element of these two nodes) is accepted
extern "C" int flux(const double* a, const double* b, double gm1, double* f) {
  const double* q[2] = {a, b};
  unsigned key[6] = {0, ~0u, 0, ~0u, 0, 0};
  for (int i = 0; i < 2; ++i) {
    const double* w = q[i];
    if (hi(w[0]) > key[0]) key[0] = hi(w[0]);
    if (hi(w[0]) < key[1]) key[1] = hi(w[0]);
    if (hi(w[1]) > key[2]) key[2] = hi(w[1]);
    if (hi(w[1]) < key[3]) key[3] = hi(w[1]);
    if (hi(w[2]) > key[5]) key[5] = hi(w[2]);
    for (int k = 0; k < 3; ++k) {
      const unsigned h = hi(w[3 + k]) & 0x7fffffffu;
      if (h > key[4]) key[4] = h;
    }
  }
  int c[2];
  scale_bits(gm1, c);
  const Scale s = element_scale(key, c);
  if (!s.ok) return 0;
  Node<3> n[2];
  for (int i = 0; i < 2; ++i) {
    const double* w = q[i];
    n[i].r = half_fixed(w[0], s.er);
    n[i].lr = ln_fixed(w[0], s.er);
    n[i].e = half_fixed(w[1], s.ee);
    n[i].le = ln_fixed(w[1], s.ee);
    n[i].p = half_fixed(w[2], s.em);
    for (int k = 0; k < 3; ++k) n[i].v[k] = half_fixed(w[3 + k], s.ev);
  }
  i64 g[5];
  pair_flux<3>(n[0], n[1], s, g);
  for (int k = 0; k < 5; ++k)
    if (g[k] >= (1LL << 62) || g[k] <= -(1LL << 62)) return -1;
  f[0] = to_double(g[0], s.er + s.ev - 62);
  for (int k = 0; k < 3; ++k) f[1 + k] = to_double(g[1 + k], s.em - 63);
  f[4] = to_double(g[4], s.em + s.ev - 61);
  return 1;
}
extern "C" double ln_error(double x, double ref_hi, double ref_lo, int E) {
  const double l = (double)(ln_fixed(x, E) >> 20) * 0x1p-40;  // 2^-40 units first
  const double r = (double)(ln_fixed(x, E) & 0xfffff) * 0x1p-60;
  return ((l - ref_hi) - ref_lo) + r;
}
"""


@pytest.fixture(scope="module")
def shim(tmp_path_factory):
    d = tmp_path_factory.mktemp("fx")
    src, so = d / "fx.cpp", d / "fx.so"
    src.write_text(SHIM)
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-fPIC", "-shared", "-I", CSRC,
                    str(src), "-o", str(so)], check=True)
    lib = ctypes.CDLL(str(so))
    dp = ctypes.POINTER(ctypes.c_double)
    lib.flux.argtypes = [dp, dp, ctypes.c_double, dp]
    lib.ln_error.argtypes = [ctypes.c_double, ctypes.c_double, ctypes.c_double, ctypes.c_int]
    lib.ln_error.restype = ctypes.c_double
    return lib


def ln_mean(x, y):
    return x if x == y else (y - x) / mp.log(y / x)


def exact_flux(a, b, gm1):
    a, b = [mp.mpf(float(x)) for x in a], [mp.mpf(float(x)) for x in b]
    rho = ln_mean(a[0], b[0])
    e = 1 / ln_mean(1 / a[1], 1 / b[1])
    f0 = rho * (a[3] + b[3]) / 2
    f = [f0] + [f0 * (a[3 + k] + b[3 + k]) / 2 for k in range(3)]
    f[1] += (a[2] + b[2]) / 2
    vv = sum(a[3 + k] * b[3 + k] for k in range(3))
    return f + [f0 * (vv / 2 + e) + (a[2] * b[3] + b[2] * a[3]) / 2]


def run(lib, a, b, gm1):
    v = [np.ascontiguousarray(x, dtype=np.float64) for x in (a, b, np.zeros(5))]
    p = [x.ctypes.data_as(ctypes.POINTER(ctypes.c_double)) for x in v]
    return lib.flux(p[0], p[1], gm1, p[2]), v[2]


@pytest.mark.parametrize("gamma", [1.4, 5.0 / 3.0, 1.05, 3.0])
def test_pair_flux_against_the_formula(shim, gamma):
    mp.mp.dps = 40
    gm1 = gamma - 1.0
    rng = np.random.default_rng(7)
    taken = 0
    # |ln ratio| through the short (< 0.25), mid (< 1) and far ranges of both
    # means, at their switches, and isobaric pairs
    logs = (0.0, 1e-9, 1e-3, 0.1, 0.2499999, 0.2500001, 0.7, 0.9999999, 1.0000001, 2.5, 4.0)
    for lr, iso, mach, units in itertools.product(logs, (True, False), (0.0, 1e-4, 0.3, 2.0),
                                                  (1.0, 1e-30, 1e25)):
        for le in ((-lr,) if iso else (0.0, 0.1, -0.8, 1.5)):
            rho = units * np.exp(rng.uniform(-2, 2)) * np.exp([0.0, lr])
            e = np.exp(rng.uniform(-2, 2)) * np.exp([0.0, le])
            p = gm1 * rho * e
            if iso:
                p[1] = p[0]
                e[1] = p[0] / (gm1 * rho[1])
            c = np.sqrt(gamma * gm1 * e.max())
            v = mach * c * rng.uniform(-1, 1, size=(2, 3))
            ok, f = run(shim, [rho[0], e[0], p[0], *v[0]], [rho[1], e[1], p[1], *v[1]], gm1)
            assert ok >= 0  # inside the formats' bounds
            if not ok:
                continue
            taken += 1
            x = exact_flux([rho[0], e[0], p[0], *v[0]], [rho[1], e[1], p[1], *v[1]], gm1)
            vm = np.abs(v).max()
            pm = p.max() + rho.max() * vm ** 2
            size = [rho.max() * vm, pm, pm, pm, pm * vm * (1 + 1 / gm1)]
            for k in range(5):
                # the final rounding to FP64 and the truncation of the node
                # values, of the flux's natural size
                assert abs(f[k] - x[k]) <= 4 * 2.0 ** -53 * size[k], (lr, le, mach, units, k)
    assert taken > 300


def test_logarithm(shim):
    # the documented error of the logarithm, 2^-52, over mantissas at and
    # between the table's nodes and over the exponents in use
    mp.mp.dps = 40
    rng = np.random.default_rng(3)
    m = np.concatenate([1 + np.arange(128) / 128, np.nextafter(1 + np.arange(1, 129) / 128, 0),
                        rng.uniform(1, 2, 2000)])
    for x, j in zip(m, itertools.cycle((-8, -3, -1))):
        x = float(x) * 2.0 ** j
        r = mp.log(mp.mpf(x))
        err = shim.ln_error(x, float(r), float(r - mp.mpf(float(r))), 0)
        assert abs(err) <= 2.0 ** -52, x


def test_refused_states_take_the_fp64_form(shim):
    base = [1.0, 2.0, 0.8, 0.1, 0.2, 0.3]
    for k, bad in ((0, 0.0), (0, -1.0), (0, np.nan), (0, np.inf), (1, -2.0), (1, np.nan),
                   (1, np.inf), (3, np.nan), (4, -np.inf), (0, 100.0), (1, 500.0), (0, 1e-300),
                   (5, 1e60), (2, np.nan)):
        other = list(base)
        other[k] = bad
        if k != 2:
            assert run(shim, base, other, 0.4)[0] == 0, (k, bad)


def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


@pytest.mark.gpu
@pytest.mark.parametrize("d,N,n", [(2, 1, (27, 25)), (2, 2, (3, 5)), (2, 3, (26, 25)),
                                   (2, 7, (25, 26)), (3, 1, (9, 9, 9)), (3, 2, (4, 3, 2)),
                                   (3, 2, (9, 9, 8)), (3, 3, (4, 3, 5)), (3, 3, (10, 9, 7)),
                                   (3, 4, (3, 2, 3)), (3, 4, (9, 10, 7)), (3, 5, (2, 3, 2)),
                                   (3, 5, (9, 9, 8)), (3, 6, (2, 2, 2)), (3, 7, (2, 2, 1)),
                                   (3, 7, (8, 9, 9))])
@pytest.mark.parametrize("kind", ["mild", "wide", "mixed", "fast", "still", "units"])
def test_rhs_inside_and_outside_the_accepted_range(d, N, n, kind):
    torch = _gpu()
    import oracle
    from paper_2108_06476_gb300 import Mesh, workloads as W
    oracle.build()
    rng = np.random.default_rng([d, N, 5])
    ne, P = int(np.prod(n)), (N + 1) ** d
    w = {"mild": 0.2, "wide": 1.5, "mixed": 0.5, "fast": 0.5, "still": 0.5, "units": 0.5}[kind]
    rho = np.exp(rng.uniform(-w, w, (ne, P)))
    p = 2.0 * np.exp(rng.uniform(-w, w, (ne, P)))
    v = [rng.uniform(-0.5, 0.5, (ne, P)) for _ in range(d)]
    if kind == "mixed":  # every third element beyond the accepted ratio
        rho[::3, 0] = 1e4
        p[1::3, P - 1] = 5e3
    if kind == "fast":
        v = [30.0 + 2.0 * x for x in v]
    if kind == "still":
        v = [0.0 * x for x in v]
    if kind == "units":
        rho, p, v = rho * 1e-20, p * 1e-8, [x * 1e6 for x in v]
    u = W.prim_to_cons(rho, v, p).reshape(-1)
    u = np.ascontiguousarray(u)
    dom = W.box(d)
    m = Mesh(d, N, n)
    got = m.rhs(torch.from_numpy(u).cuda()).cpu().numpy()
    assert m.check() == 0
    elems = np.unique(np.linspace(0, ne - 1, 40).astype(np.int64))
    ref = oracle.rhs(d, N, n, dom, u, elems=elems).reshape(ne, d + 2, P)[elems]
    g = got.reshape(ne, d + 2, P)[elems]
    for e in range(len(elems)):  # element by element: both forms meet the bar
        err = np.linalg.norm(g[e] - ref[e]) / np.linalg.norm(ref[e])
        assert err <= 1e-12, (kind, int(elems[e]), err)


@pytest.mark.gpu
@pytest.mark.parametrize("d,N,n", [(2, 3, (4, 4)), (3, 3, (9, 9, 9)), (3, 4, (3, 3, 3))])
def test_a_state_at_rest_keeps_its_density_and_energy(d, N, n):
    # every mass and energy flux is zero, whatever the form
    torch = _gpu()
    from paper_2108_06476_gb300 import Mesh, workloads as W
    rng = np.random.default_rng(2)
    ne, P = int(np.prod(n)), (N + 1) ** d
    rho = rng.uniform(0.5, 2.0, (ne, P))
    u = W.prim_to_cons(rho, [0.0 * rho] * d, 3.0 + 0.0 * rho).reshape(-1)
    du = Mesh(d, N, n, surface_flux="ranocha").rhs(torch.from_numpy(u).cuda())
    du = du.cpu().numpy().reshape(ne, d + 2, P)
    assert not du[:, 0].any() and not du[:, d + 1].any()


@pytest.mark.gpu
@pytest.mark.parametrize("d,N,n", [(2, 1, (27, 25)), (2, 3, (26, 25)), (2, 6, (25, 27)),
                                   (3, 1, (9, 9, 9)), (3, 2, (40, 13, 17)), (3, 3, (10, 9, 7)),
                                   (3, 4, (9, 10, 7)), (3, 5, (9, 9, 8)), (3, 6, (9, 9, 8)),
                                   (3, 7, (8, 9, 9))])
@pytest.mark.parametrize("kind", ["random", "fast", "still", "units", "huge"])
def test_weak_form_against_the_oracle(d, N, n, kind):
    # the nodal-flux form of the central volume flux, in fixed point and (an
    # element with a value beyond its exponents) in FP64
    torch = _gpu()
    import oracle
    from paper_2108_06476_gb300 import Mesh, workloads as W
    oracle.build()
    rng = np.random.default_rng([d, N, 6])
    ne, P = int(np.prod(n)), (N + 1) ** d
    rho = np.exp(rng.uniform(-1, 1, (ne, P)))
    p = 2.0 * np.exp(rng.uniform(-1, 1, (ne, P)))
    v = [rng.uniform(-0.5, 0.5, (ne, P)) for _ in range(d)]
    if kind == "fast":
        v = [30.0 + 2.0 * x for x in v]
    if kind == "still":
        v = [0.0 * x for x in v]
    if kind == "units":
        rho, p, v = rho * 1e-20, p * 1e-8, [x * 1e6 for x in v]
    if kind == "huge":  # every other element beyond the accepted exponents
        rho[::2] *= 1e50
        p[::2] *= 1e50
    u = np.ascontiguousarray(W.prim_to_cons(rho, v, p).reshape(-1))
    dom = W.box(d)
    m = Mesh(d, N, n, volume_flux="central", surface_flux="hll")
    got = m.rhs(torch.from_numpy(u).cuda()).cpu().numpy().reshape(ne, d + 2, P)
    assert m.check() == 0
    elems = np.unique(np.linspace(0, ne - 1, 40).astype(np.int64))
    ref = oracle.rhs(d, N, n, dom, u, vflux=2, sflux=2, elems=elems).reshape(ne, d + 2, P)
    for e in elems:
        err = np.linalg.norm(got[e] - ref[e]) / np.linalg.norm(ref[e])
        assert err <= 1e-12, (kind, int(e), err)


@pytest.mark.gpu
@pytest.mark.parametrize("N,n", [(1, (3, 4, 5)), (2, (3, 2, 4)), (3, (3, 2, 3)), (3, (10, 9, 8)),
                                 (4, (2, 3, 2)), (4, (9, 10, 8)), (5, (3, 2, 2)), (6, (2, 2, 2)),
                                 (7, (2, 1, 2))])
@pytest.mark.parametrize("vf,sf", [("central", "hll"), ("central", "llf"), ("ec", "ec")])
@pytest.mark.parametrize("kind", ["random", "nofield", "strong", "still", "fast", "mixed", "units"])
def test_mhd_rhs_inside_and_outside_the_accepted_range(N, n, vf, sf, kind):
    torch = _gpu()
    import oracle
    from paper_2108_06476_gb300 import Mesh, workloads as W
    oracle.build()
    rng = np.random.default_rng([N, 8])
    ne, P = int(np.prod(n)), (N + 1) ** 3
    rho = np.exp(rng.uniform(-0.6, 0.6, (ne, P)))
    p = 2.0 * np.exp(rng.uniform(-0.6, 0.6, (ne, P)))
    v = rng.uniform(-0.5, 0.5, (3, ne, P))
    B = rng.uniform(-1, 1, (3, ne, P))
    if kind == "nofield":
        B *= 0.0
    if kind == "strong":
        B *= 10.0
    if kind == "still":
        v *= 0.0
    if kind == "fast":
        v[0] += 8.0
    if kind == "mixed":  # every third element beyond the accepted ratio
        rho[::3, 0] = 1e4
        p[1::3, P - 1] = 5e3
    if kind == "units":
        rho, p, v, B = rho * 1e-20, p * 1e-8, v * 1e6, B * 1e-4
    E = p / (5.0 / 3.0 - 1.0) + 0.5 * rho * (v ** 2).sum(0) + 0.5 * (B ** 2).sum(0)
    u = np.ascontiguousarray(np.stack([rho, *(rho * v), E, *B], axis=1).reshape(-1))
    m = Mesh(3, N, n, equations="mhd", volume_flux=vf, surface_flux=sf)
    got = m.rhs(torch.from_numpy(u).cuda()).cpu().numpy().reshape(ne, 8, P)
    assert m.check() == 0
    elems = np.unique(np.linspace(0, ne - 1, 30).astype(np.int64))
    ref = oracle.mhd_rhs(N, n, W.box(3), u, sflux=sf, vflux=vf, elems=elems).reshape(ne, 8, P)
    # "strong" and "fast" lose digits of p in E - m.v/2 - |B|^2/2 on either side
    bar = 1e-12 * (20.0 if kind in ("strong", "fast") else 1.0)
    for e in elems:
        err = np.linalg.norm(got[e] - ref[e]) / np.linalg.norm(ref[e])
        assert err <= bar, (kind, int(e), err)


@pytest.mark.gpu
@pytest.mark.parametrize("d,N,n", [(2, 1, (3, 4)), (2, 2, (5, 3)), (2, 7, (3, 3)), (3, 1, (3, 2, 4)),
                                   (3, 2, (2, 3, 4)), (3, 3, (3, 4, 2)), (3, 4, (3, 2, 3)),
                                   (3, 5, (2, 3, 1)), (3, 6, (2, 1, 2)), (3, 7, (2, 2, 1))])
@pytest.mark.parametrize("kind", ["mild", "wide", "far", "mixed", "fast", "still", "units", "mass",
                                  "momentum", "energy"])
def test_vjp_inside_and_outside_the_accepted_range(d, N, n, kind):
    # <w, J v> from the oracle's exact JVP against <J^T w, v>, v supported on
    # one element at a time: every element's block of J^T w meets the bar,
    # relative to the sum of the products' magnitudes (2^-53 times some
    # hundreds of operations per entry stays below 1e-12)
    torch = _gpu()
    import oracle
    from paper_2108_06476_gb300 import Mesh, workloads as W
    oracle.build()
    rng = np.random.default_rng([d, N, 9])
    ne, P = int(np.prod(n)), (N + 1) ** d
    s = {"mild": 0.05, "wide": 0.45, "far": 2.0}.get(kind, 0.3)
    rho = np.exp(rng.uniform(-s, s, (ne, P)))
    p = 2.0 * np.exp(rng.uniform(-s, s, (ne, P)))
    v = [rng.uniform(-0.5, 0.5, (ne, P)) for _ in range(d)]
    w = rng.standard_normal((ne, d + 2, P))
    if kind == "mixed":
        rho[::3, 0] = 1e4
        p[1::3, P - 1] = 5e3
        w[2::3, :, 0] = 0.0
        w[2] = 0.0
    if kind == "fast":
        v = [30.0 + 2.0 * x for x in v]
    if kind == "still":
        v = [0.0 * x for x in v]
    if kind == "units":
        rho, p, v = rho * 1e-20, p * 1e-8, [x * 1e6 for x in v]
    if kind in ("mass", "momentum", "energy"):
        keep = {"mass": [0], "momentum": list(range(1, d + 1)), "energy": [d + 1]}[kind]
        w[:, [k for k in range(d + 2) if k not in keep]] = 0.0
    u = np.ascontiguousarray(W.prim_to_cons(rho, v, p).reshape(-1))
    w = np.ascontiguousarray(w.reshape(-1))
    m = Mesh(d, N, n)
    ub = m.rhs_vjp(torch.from_numpy(u).cuda(), torch.from_numpy(w).cuda()).cpu().numpy()
    ub = ub.reshape(ne, -1)
    scale = np.abs(u.reshape(ne, d + 2, P)).max(axis=(0, 2))
    for e in range(min(ne, 6)):
        t = np.zeros((ne, d + 2, P))
        t[e] = rng.standard_normal((d + 2, P)) * scale[:, None]
        jv = oracle.rhs_jvp(d, N, n, W.box(d), u, np.ascontiguousarray(t.reshape(-1)))
        gap = abs(float(w @ jv) - float(ub[e] @ t[e].reshape(-1)))
        size = float(np.abs(w * jv).sum())
        assert gap <= 1e-12 * size or size == 0.0, (kind, e, gap, size)
