"""The work a user has this framework do, as measurable cases.

Right-hand sides, Runge-Kutta steps, ensembles and gradients of the 2D/3D
compressible Euler equations (Cartesian and warped meshes) and of 3D ideal
MHD, through the package's public classes (Mesh, Ensemble) and its autograd
function. `exact` evaluates the same discretisation in plain torch: in
double-double arithmetic (two float64 per value), or in float64 where
torch.autograd supplies the derivative.
"""
import math

import numpy as np
import torch

from paper_2108_06476_gb300 import Ensemble, Mesh
from paper_2108_06476_gb300 import autograd as dg_autograd

CFL = 0.5
RK_A = (0.0, -567301805773.0 / 1357537059087.0, -2404267990393.0 / 2016746695238.0,
        -3550918686646.0 / 2091501179385.0, -1275806237668.0 / 842570457699.0)
RK_B = (1432997174477.0 / 9575080441755.0, 5161836677717.0 / 13612068292357.0,
        1720146321549.0 / 2090206949498.0, 3134564353537.0 / 4481467310338.0,
        2277821191437.0 / 14882151754819.0)
RK_C = (0.0, 1432997174477.0 / 9575080441755.0, 2526269341429.0 / 6820363962896.0,
        2006345519317.0 / 3224310063776.0, 2802321613138.0 / 2924317926251.0)


def _case(name, eq, do, d, N, n, vf, sf, state, prec="fp64", graph=False):
    return {"name": name, "eq": eq, "do": do, "d": d, "N": N, "nx": n[0], "ny": n[1],
            "nz": n[2] if d == 3 else 1, "vf": vf, "sf": sf, "state": state, "prec": prec,
            "graph": graph}


def listed():
    return [
        # the smallest configured run: one rhs call on 4,096 nodes, latency
        _case("rhs_2d_16sq_n3", "euler", "rhs", 2, 3, (16, 16), "ranocha", "llf", "wave"),
        # a small 3D simulation advanced by replayed steps (a user's time loop)
        _case("step_graph_8cubed_n3", "euler", "step", 3, 3, (8, 8, 8), "ranocha", "llf", "noisy",
              graph=True),
        # an odd, ragged mesh with the entropy-conservative faces on rough data
        _case("rhs_ec_19x14x11_n5", "euler", "rhs", 3, 5, (19, 14, 11), "ranocha", "ranocha",
              "random"),
        # the weak form (central volume flux, HLL faces), the paper's other solver
        _case("rhs_weak_32cubed_n4", "euler", "rhs", 3, 4, (32, 32, 32), "central", "hll", "noisy"),
        # the configured high-degree mesh
        _case("rhs_24cubed_n7", "euler", "rhs", 3, 7, (24, 24, 24), "ranocha", "llf", "noisy"),
        # the headline: time steps of the 64^3 mesh of degree 3
        _case("step_64cubed_n3", "euler", "step", 3, 3, (64, 64, 64), "ranocha", "llf", "noisy"),
        # the same simulation with the FP32 kernels
        _case("step_64cubed_n3_fp32", "euler", "step", 3, 3, (64, 64, 64), "ranocha", "llf",
              "noisy", prec="fp32"),
        # the configured ensemble: 48 simulations of mixed degrees, one step each
        {"name": "ensemble_48", "eq": "euler", "do": "ensemble", "sims": 48, "n_lo": 8,
         "n_hi": 24, "prec": "fp64"},
        # a gradient through the rhs (differentiating through a simulation)
        _case("grad_16cubed_n4", "euler", "grad", 3, 4, (16, 16, 16), "ranocha", "llf", "noisy"),
        # steps on the paper's warped box with the manufactured source
        _case("step_warped_16cubed_n3", "curved", "step", 3, 3, (16, 16, 16), "ranocha", "ranocha",
              "manufactured"),
        # MHD, the paper's weak-form solver with HLL faces
        _case("step_mhd_weak_32cubed_n3", "mhd", "step", 3, 3, (32, 32, 32), "central", "hll",
              "alfven"),
        # MHD, entropy-conservative flux differencing
        _case("rhs_mhd_ec_20cubed_n4", "mhd", "rhs", 3, 4, (20, 20, 20), "ec", "ec", "alfven"),
    ]


def draw(rng):
    kind = rng.choice(("euler", "euler", "euler", "euler", "weak", "ensemble", "grad", "curved",
                       "mhd", "mhd"))
    if kind == "ensemble":
        lo = rng.randint(5, 12)
        return {"eq": "euler", "do": "ensemble", "sims": rng.randint(3, 40), "n_lo": lo,
                "n_hi": lo + rng.randint(1, 11), "prec": rng.choice(("fp64", "fp64", "fp32"))}
    d = rng.choice((2, 3, 3)) if kind in ("euler", "weak") else 3
    N = rng.choice((1, 2, 3, 3, 3, 4, 5, 6, 7))
    most = {"euler": 6e6, "weak": 6e6, "grad": 8e5, "curved": 1.5e6, "mhd": 3e6}[kind]
    nodes = math.exp(rng.uniform(math.log(3e3), math.log(most)))
    n1 = max(2.0, (nodes / (N + 1) ** d) ** (1.0 / d))
    n = [max(2, int(round(n1 * rng.uniform(0.75, 1.25)))) for _ in range(d)]
    do = "grad" if kind == "grad" else rng.choice(("rhs", "step"))
    prec = rng.choice(("fp64", "fp64", "fp64", "fp32")) if kind in ("euler", "weak") else "fp64"
    graph = do == "step" and rng.random() < 0.4
    if kind == "mhd":
        vf, sf, state = rng.choice((("central", "hll"), ("central", "llf"), ("ec", "ec"),
                                    ("ec", "llf"))) + ("alfven",)
    elif kind == "weak":
        vf, sf, state = "central", "hll", rng.choice(("wave", "noisy"))
    elif kind == "curved":
        vf, sf, state = rng.choice((("ranocha", "ranocha"), ("ranocha", "llf"))) + ("manufactured",)
    else:
        vf, sf = rng.choice((("ranocha", "llf"), ("ranocha", "llf"), ("ranocha", "hll"),
                             ("ranocha", "ranocha")))
        state = rng.choice(("wave", "noisy", "noisy", "random" if do == "rhs" else "noisy"))
    c = _case("", "euler" if kind in ("weak", "grad") else kind, do, d, N, n, vf, sf, state, prec,
              graph)
    del c["name"]
    return c


# ---- inputs ----
def _lgl(N):
    """LGL nodes, weights and differentiation matrix (numpy long double)."""
    ld = np.longdouble
    x = -np.cos(np.pi * np.arange(N + 1) / N).astype(ld)

    def legendre(n, t):
        a, b = np.ones_like(t), t
        if n == 0:
            return a
        for k in range(1, n):
            a, b = b, ((2 * k + 1) * t * b - k * a) / ld(k + 1)
        return b

    for _ in range(100):
        q = legendre(N + 1, x) - legendre(N - 1, x)
        s = q / ((2 * N + 1) * legendre(N, x))
        s[0] = s[-1] = 0
        x = x - s
    x[0], x[-1] = ld(-1), ld(1)
    pn = legendre(N, x)
    w = ld(2) / (N * (N + 1) * pn * pn)
    D = np.zeros((N + 1, N + 1), dtype=ld)
    for i in range(N + 1):
        for j in range(N + 1):
            if i != j:
                D[i, j] = pn[i] / (pn[j] * (x[i] - x[j]))
    D[0, 0], D[N, N] = -ld(N * (N + 1)) / 4, ld(N * (N + 1)) / 4
    return x, w, D


def _counts(c):
    return (c["nx"], c["ny"], c["nz"])[:c["d"]]


def _coordinates(n, N, xi, np_type=np.float64):
    """Box coordinates of the nodes, one array [elements, (N+1)^d] per direction."""
    d = len(n)
    e = np.indices(n[::-1]).reshape(d, -1)[::-1]
    k = np.indices((N + 1,) * d).reshape(d, -1)[::-1]
    xi = np.asarray(xi, dtype=np_type)
    return [-1 + (e[r][:, None] + (xi[k[r]][None, :] + 1) / 2) * (np_type(2) / n[r])
            for r in range(d)]


def _warp(X):
    """The paper's warping of the box, amplitude 0.15 (long double)."""
    a, pi = np.longdouble(3) / 20, np.arccos(np.longdouble(-1))
    y = X[1] + a * np.cos(1.5 * pi * X[0]) * np.cos(0.5 * pi * X[1]) * np.cos(0.5 * pi * X[2])
    x = X[0] + a * np.cos(0.5 * pi * X[0]) * np.cos(2 * pi * y) * np.cos(0.5 * pi * X[2])
    z = X[2] + a * np.cos(0.5 * pi * x) * np.cos(pi * y) * np.cos(0.5 * pi * X[2])
    return [x, y, z]


def _euler_cons(rho, v, p):
    v2 = sum(vk * vk for vk in v)
    return torch.stack([rho] + [rho * vk for vk in v] + [p / 0.4 + 0.5 * rho * v2], dim=1)


def _state(c, seed):
    """The conserved state, float64 on the GPU, layout u[e][v][nodes]."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    r = np.random.default_rng(int(seed))
    n, N, d = _counts(c), c["N"], c["d"]
    if c["state"] == "manufactured":
        X = _warp(_coordinates(n, N, _lgl(N)[0], np.longdouble))
        s = torch.from_numpy(sum(X).astype(np.float64)).cuda()
        rho = 2.0 + 0.1 * torch.sin(math.pi * s)
        u = torch.stack([rho, rho, rho, rho, rho * rho], dim=1)
        noise = torch.rand(u.shape, generator=g, device="cuda", dtype=torch.float64)
        return (u + 1e-3 * (2.0 * noise - 1.0)).reshape(-1)
    X = [torch.from_numpy(x).cuda() for x in _coordinates(n, N, _lgl(N)[0])]
    s = math.pi * sum(X)

    def uniform(lo, hi):
        return lo + (hi - lo) * torch.rand(s.shape, generator=g, device="cuda",
                                           dtype=torch.float64)

    if c["state"] == "alfven":  # the circularly polarised wave at a drawn phase
        A, phi = 0.1, s + r.uniform(0, 2 * math.pi)
        nv = np.ones(3) / math.sqrt(3.0)
        e1 = np.array([1.0, -1.0, 0.0]) / math.sqrt(2.0)
        e2 = np.cross(nv, e1)
        sn, cs = torch.sin(phi), torch.cos(phi)
        B = [nv[k] + A * (sn * e1[k] + cs * e2[k]) for k in range(3)]
        v = [-A * (sn * e1[k] + cs * e2[k]) for k in range(3)]
        rho = 1.0 + 1e-2 * uniform(-1, 1)
        p = 0.1 + 1e-3 * uniform(-1, 1)
        E = p / (5.0 / 3.0 - 1.0) + 0.5 * rho * sum(a * a for a in v) + 0.5 * sum(b * b for b in B)
        return torch.stack([rho] + [rho * a for a in v] + [E] + B, dim=1).reshape(-1)
    if c["state"] == "random":
        return _euler_cons(uniform(0.5, 2.0), [uniform(-0.5, 0.5) for _ in range(d)],
                           uniform(0.5, 3.0)).reshape(-1)
    vel = r.uniform(-0.3, 0.3, size=d)
    A, ph = r.uniform(0.5, 0.98), r.uniform(0, 2 * math.pi)
    if c["state"] == "noisy":
        A = min(A, 0.9)
    rho, p = 1.0 + A * torch.sin(s + ph), torch.full_like(s, 20.0)
    v = [torch.full_like(s, float(a)) for a in vel]
    if c["state"] == "noisy":
        rho = rho + 1e-2 * uniform(-1, 1)
        v = [a + 1e-2 * uniform(-1, 1) for a in v]
        p = p + 1e-2 * uniform(-1, 1)
    return _euler_cons(rho, v, p).reshape(-1)


def _members(c, seed):
    """(degree, elements per direction) of each member: the ensemble's make-up
    belongs to the case; the seed draws the members' waves."""
    r = np.random.default_rng([17, c["sims"], c["n_lo"], c["n_hi"]])
    m = [(int(r.choice((3, 4, 5))), int(r.integers(c["n_lo"], c["n_hi"] + 1)))
         for _ in range(c["sims"])]
    u = [_state({"state": "wave", "d": 3, "N": N, "nx": n, "ny": n, "nz": n}, seed * 1000 + i)
         for i, (N, n) in enumerate(m)]
    return m, u


def _mesh(c):
    kw = {}
    if c["eq"] == "curved":
        kw["warp"] = 0.15
    if c["eq"] == "mhd":
        kw["equations"] = "mhd"
    m = Mesh(c["d"], c["N"], _counts(c), volume_flux=c["vf"], surface_flux=c["sf"],
             precision=c["prec"], **kw)
    if c["eq"] == "curved":
        m.set_source("manufactured")
    return m


def prepare(case, seed):
    if case["do"] == "ensemble":
        m, u = _members(case, seed)
        ens = Ensemble([N for N, _ in m], [n for _, n in m], precision=case["prec"])
        u0 = torch.cat(u)
        return {"case": case, "ens": ens, "u0": u0, "u": u0.clone()}
    u0 = _state(case, seed)
    st = {"case": case, "mesh": _mesh(case), "u0": u0}
    if case["do"] == "step":
        st["u"] = u0.clone()
    else:
        st["du"] = st["mesh"].empty_rhs()
    if case["do"] == "grad":
        g = torch.Generator(device="cuda").manual_seed(int(seed) + 1)
        st["w"] = torch.randn(u0.shape, generator=g, device="cuda", dtype=torch.float64)
    return st


def run(state):
    c = state["case"]
    if c["do"] == "rhs":
        return state["mesh"].rhs(state["u0"], state["du"])
    if c["do"] == "grad":
        u = state["u0"].detach().requires_grad_(True)
        du = dg_autograd.rhs(state["mesh"], u)
        du.backward(state["w"])
        return {"du": du.detach(), "ubar": u.grad}
    # one step from the same initial state (an in-place step on a working copy)
    u = state["u"]
    u.copy_(state["u0"])
    if c["do"] == "ensemble":
        state["ens"].step(u, CFL)
        return u
    if c["eq"] == "curved":
        state["mesh"].set_time(0.0)
    state["mesh"].step_cfl(u, CFL, graph=c["graph"])
    return u


def work(case):
    # one rhs per node: primitives, d N / 2 two-point fluxes with both nodes'
    # accumulation, lifting; a step is five of them with the stage update
    def per_node(d, N, kind):
        pair = {"ranocha": 88.0, "ec": 190.0, "central": 30.0}[kind]
        return 14.0 + 0.5 * d * N * pair + 15.0

    if case["do"] == "ensemble":
        r = np.random.default_rng([17, case["sims"], case["n_lo"], case["n_hi"]])
        m = [(int(r.choice((3, 4, 5))), int(r.integers(case["n_lo"], case["n_hi"] + 1)))
             for _ in range(case["sims"])]
        nodes = sum((n * (N + 1)) ** 3 for N, n in m)
        flops = sum((n * (N + 1)) ** 3 * 5 * (per_node(3, N, "ranocha") + 25) for N, n in m)
        return {"bytes": 80.0 * nodes, "flops": flops}
    d, N = case["d"], case["N"]
    nodes = float(np.prod(_counts(case))) * (N + 1) ** d
    nv = 8 if case["eq"] == "mhd" else d + 2
    one = per_node(d, N, case["vf"])
    out = 4.0 if case["prec"] == "fp32" and case["do"] == "rhs" else 8.0
    if case["do"] == "rhs":
        return {"bytes": nodes * nv * (8.0 + out), "flops": nodes * one}
    if case["do"] == "grad":  # the rhs, then each pair's flux and its adjoint
        return {"bytes": nodes * nv * 32.0, "flops": nodes * one * 3.5}
    return {"bytes": nodes * nv * 16.0, "flops": nodes * 5.0 * (one + 5.0 * nv)}


# ---- the same discretisation in plain torch ----
class DD:
    """Unevaluated sum hi + lo of two float64 tensors (double-double)."""

    def __init__(self, hi, lo=None):
        self.hi, self.lo = hi, torch.zeros_like(hi) if lo is None else lo

    @staticmethod
    def of(x, like):
        return x if isinstance(x, DD) else DD(torch.as_tensor(x, dtype=torch.float64,
                                                              device=like.hi.device))

    @staticmethod
    def norm(s, e):
        hi = s + e
        return DD(hi, e - (hi - s))

    def __add__(self, o):
        o = DD.of(o, self)
        s = self.hi + o.hi
        b = s - self.hi
        e = (self.hi - (s - b)) + (o.hi - b)
        t = self.lo + o.lo
        b = t - self.lo
        f = (self.lo - (t - b)) + (o.lo - b)
        r = DD.norm(s, e + t)
        return DD.norm(r.hi, r.lo + f)

    def __neg__(self):
        return DD(-self.hi, -self.lo)

    def __sub__(self, o):
        return self + (-DD.of(o, self))

    def __rsub__(self, o):
        return DD.of(o, self) + (-self)

    def __mul__(self, o):
        o = DD.of(o, self)
        p = self.hi * o.hi

        def split(x):
            y = 134217729.0 * x
            h = y - (y - x)
            return h, x - h

        (a, b), (c, d) = split(self.hi), split(o.hi)
        e = ((a * c - p) + a * d + b * c) + b * d
        return DD.norm(p, e + (self.hi * o.lo + self.lo * o.hi))

    def __truediv__(self, o):
        o = DD.of(o, self)
        q = DD(self.hi / o.hi)
        for _ in range(2):
            r = self - o * q
            q = q + DD(r.hi / o.hi)
        return q

    __radd__, __rmul__ = __add__, __mul__

    def __rtruediv__(self, o):
        return DD.of(o, self) / self

    def map(self, f):
        return DD(f(self.hi), f(self.lo))


def _map(x, f):
    return x.map(f) if isinstance(x, DD) else f(x)


def _hi(x):
    return x.hi if isinstance(x, DD) else x


def _stack(xs, dim):
    if isinstance(xs[0], DD):
        return DD(torch.stack([x.hi for x in xs], dim), torch.stack([x.lo for x in xs], dim))
    return torch.stack(xs, dim)


def _where(m, x, y):
    if isinstance(x, DD):
        return DD(torch.where(m, x.hi, y.hi), torch.where(m, x.lo, y.lo))
    return torch.where(m, x, y)


def _max(x, y):
    return _where(_hi(x) >= _hi(y), x, y)


def _abs(x):
    return _where(_hi(x) >= 0, x, -x)


def _sqrt(x):
    if not isinstance(x, DD):
        return torch.sqrt(x)
    s = DD(torch.sqrt(x.hi))
    return (s + x / s) * 0.5


def _atanh_over(t2):
    """atanh(t)/t = sum t^(2k)/(2k+1), enough terms for the largest t."""
    m = min(float(_hi(t2).max().detach()), 0.98)
    K = max(4, int(math.ceil(-46.0 / math.log(max(m, 1e-12)))))
    if not isinstance(t2, DD):
        K = max(4, (K * 5 + 5) // 6)
    r = None
    for k in range(K, -1, -1):
        c = 1.0 / (DD.of(2.0 * k + 1.0, t2)) if isinstance(t2, DD) else 1.0 / (2 * k + 1)
        r = t2 * 0.0 + c if r is None else r * t2 + c
    return r


def _ln_mean(x, y):
    s = x + y
    t = (y - x) / s
    return s * 0.5 / _atanh_over(t * t)


def _inv_ln_mean(x, y):
    s = x + y
    t = (y - x) / s
    return _atanh_over(t * t) * 2.0 / s


class Euler:
    gamma = 1.4

    def prim(self, u):
        d = len(u) - 2
        v = [u[1 + k] / u[0] for k in range(d)]
        m = u[1] * v[0]
        for k in range(1, d):
            m = m + u[1 + k] * v[k]
        p = (u[d + 1] - m * 0.5) * (self.gamma - 1.0 if not isinstance(m, DD) else self._gm1(m))
        return [u[0]] + v + [p]

    def _gm1(self, like):
        return DD.of(self.gamma, like) - 1.0

    def directed(self, g, w):
        """sum_k g_k w_k; g is a direction index or a list of components."""
        if isinstance(g, int):
            return w[g]
        r = g[0] * w[0]
        for k in range(1, len(w)):
            r = r + g[k] * w[k]
        return r

    def add_p(self, f, g, p):
        for k in range(len(f) - 2):
            if not isinstance(g, int):
                f[1 + k] = f[1 + k] + p * g[k]
            elif k == g:
                f[1 + k] = f[1 + k] + p
        return f

    def flux(self, u, q, g):
        d = len(u) - 2
        vn = self.directed(g, q[1:1 + d])
        f = self.add_p([x * vn for x in u], g, q[d + 1])
        f[d + 1] = f[d + 1] + q[d + 1] * vn
        return f

    def two_point(self, kind, uL, qL, uR, qR, g):
        if kind == "central":
            return [(a + b) * 0.5 for a, b in zip(self.flux(uL, qL, g), self.flux(uR, qR, g))]
        d = len(uL) - 2
        gm1 = self._gm1(qL[0]) if isinstance(qL[0], DD) else self.gamma - 1.0
        vL, vR, pL, pR = qL[1:1 + d], qR[1:1 + d], qL[d + 1], qR[d + 1]
        va = [(a + b) * 0.5 for a, b in zip(vL, vR)]
        rho = _ln_mean(qL[0], qR[0])
        vv = vL[0] * vR[0]
        for k in range(1, d):
            vv = vv + vL[k] * vR[k]
        f0 = rho * self.directed(g, va)
        f = self.add_p([f0] + [f0 * a for a in va] + [f0], g, (pL + pR) * 0.5)
        e = vv * 0.5 + pL * pR * _inv_ln_mean(qL[0] * pR, qR[0] * pL) / gm1
        f[d + 1] = f0 * e + (pL * self.directed(g, vR) + pR * self.directed(g, vL)) * 0.5
        return f

    def speed(self, u, q, g):
        return _sqrt(q[-1] * self.gamma / q[0])

    def surface(self, kind, uL, qL, uR, qR, g):
        if kind not in ("llf", "hll"):
            return self.two_point(kind, uL, qL, uR, qR, g)
        norm, gu = None, g
        if not isinstance(g, int):
            norm = _sqrt(self.directed(g, g))
            gu = [x / norm for x in g]
        fL, fR = self.flux(uL, qL, gu), self.flux(uR, qR, gu)
        d = 3 if len(uL) == 8 else len(uL) - 2
        vL, vR = self.directed(gu, qL[1:1 + d]), self.directed(gu, qR[1:1 + d])
        cL, cR = self.speed(uL, qL, gu), self.speed(uR, qR, gu)
        if kind == "llf":
            lam = _max(_abs(vL), _abs(vR)) + _max(cL, cR)
            f = [(a + b - lam * (y - x)) * 0.5 for a, b, x, y in zip(fL, fR, uL, uR)]
        else:
            sL, sR = -_max(cL - vL, cR - vR), _max(vL + cL, vR + cR)
            f = []
            for a, b, x, y in zip(fL, fR, uL, uR):
                m = (sR * a - sL * b + sL * sR * (y - x)) / (sR - sL)
                f.append(_where(_hi(sL) >= 0, a, _where(_hi(sR) <= 0, b, m)))
        return f if norm is None else [x * norm for x in f]


class MHD(Euler):
    gamma = 5.0 / 3.0

    def prim(self, u):
        v = [u[1 + k] / u[0] for k in range(3)]
        m = u[1] * v[0] + u[2] * v[1] + u[3] * v[2] + u[5] * u[5] + u[6] * u[6] + u[7] * u[7]
        return [u[0]] + v + [(u[4] - m * 0.5) * self._gm1(m)]

    def flux(self, u, q, n):
        v, B, p = q[1:4], u[5:8], q[4]
        pt = p + (B[0] * B[0] + B[1] * B[1] + B[2] * B[2]) * 0.5
        vB = v[0] * B[0] + v[1] * B[1] + v[2] * B[2]
        f = [u[1 + n]] + [u[1 + n] * v[k] - B[n] * B[k] for k in range(3)]
        f[1 + n] = f[1 + n] + pt
        zero = p * 0.0
        return f + [v[n] * (u[4] + pt) - B[n] * vB] + [
            zero if k == n else v[n] * B[k] - B[n] * v[k] for k in range(3)]

    def speed(self, u, q, n):
        B = u[5:8]
        a2 = q[4] * self.gamma / q[0]
        s = a2 + (B[0] * B[0] + B[1] * B[1] + B[2] * B[2]) / q[0]
        return _sqrt((s + _sqrt(s * s - a2 * (B[n] * B[n] / q[0]) * 4.0)) * 0.5)

    def two_point(self, kind, uL, qL, uR, qR, n):
        if kind == "central":
            return [(a + b) * 0.5 for a, b in zip(self.flux(uL, qL, n), self.flux(uR, qR, n))]
        vL, vR, BL, BR = qL[1:4], qR[1:4], uL[5:8], uR[5:8]
        bL, bR = qL[0] / (qL[4] * 2.0), qR[0] / (qR[4] * 2.0)

        def dot(a, b):
            return a[0] * b[0] + a[1] * b[1] + a[2] * b[2]

        va = [(a + b) * 0.5 for a, b in zip(vL, vR)]
        Ba = [(a + b) * 0.5 for a, b in zip(BL, BR)]
        v2, B2 = (dot(vL, vL) + dot(vR, vR)) * 0.5, (dot(BL, BL) + dot(BR, BR)) * 0.5
        vB = (dot(vL, BL) + dot(vR, BR)) * 0.5
        bB2 = (bL * dot(BL, BL) + bR * dot(BR, BR)) * 0.5
        f0 = _ln_mean(qL[0], qR[0]) * va[n]
        fm = [f0 * va[k] - Ba[n] * Ba[k] for k in range(3)]
        fm[n] = fm[n] + ((qL[0] + qR[0]) * 0.5 + bB2) / (bL + bR)
        fB = [va[n] * Ba[k] - Ba[n] * va[k] for k in range(3)]
        fB[n] = va[n] * 0.0
        fE = (f0 * (_inv_ln_mean(bL, bR) * 0.5 / self._gm1(bL) - v2 * 0.5) + dot(fm, va)
              + dot(fB, Ba) - va[n] * B2 * 0.5 + Ba[n] * vB)
        return [f0] + fm + [fE] + fB


def _dd_of(a):
    """A long double array as a DD of float64 CUDA tensors."""
    hi = a.astype(np.float64)
    return DD(torch.from_numpy(hi).cuda(),
              torch.from_numpy((a - hi.astype(np.longdouble)).astype(np.float64)).cuda())


def _geometry(n, N):
    """Metric terms (J a^r)_m, 1/J (DD) and x+y+z of the warped box."""
    xi, _, D = _lgl(N)
    shape = (-1,) + (N + 1,) * 3
    X = [x.reshape(shape) for x in _warp(_coordinates(n, N, xi, np.longdouble))]

    def der(f, r):
        return np.moveaxis(np.tensordot(f, D, axes=([3 - r], [1])), -1, 3 - r)

    a = [[der(X[k], r) for k in range(3)] for r in range(3)]
    J = sum(a[0][k] * (a[1][(k + 1) % 3] * a[2][(k + 2) % 3] - a[1][(k + 2) % 3] * a[2][(k + 1) % 3])
            for k in range(3))
    Ja = [[None] * 3 for _ in range(3)]
    for m in range(3):
        v = [X[(m + 2) % 3] * der(X[(m + 1) % 3], b) for b in range(3)]
        for i in range(3):
            Ja[i][m] = _dd_of(der(v[(i + 1) % 3], (i + 2) % 3) - der(v[(i + 2) % 3], (i + 1) % 3))
    return Ja, _dd_of(1 / J), torch.from_numpy(sum(X).astype(np.float64)).cuda()


class Operator:
    """The rhs of one case on values of either arithmetic (float64 or DD)."""

    def __init__(self, c, dd=True):
        self.c, self.dd = c, dd
        self.eq = MHD() if c["eq"] == "mhd" else Euler()
        self.n, self.N, self.d = _counts(c), c["N"], c["d"]
        x, w, D = _lgl(self.N)
        Dt = 2 * D
        Dt[0, 0] += 1 / w[0]
        Dt[-1, -1] -= 1 / w[-1]
        self.D, self.lift = Dt, 1 / w[0]
        if c["eq"] == "curved":
            self.Ja, self.invJ, self.s = _geometry(self.n, self.N)
        self.nv = 8 if c["eq"] == "mhd" else self.d + 2

    def num(self, x, like):
        if not self.dd:
            return float(x)
        hi = np.float64(x)
        dev = like.hi.device
        return DD(torch.tensor(float(hi), dtype=torch.float64, device=dev),
                  torch.tensor(float(x - np.longdouble(hi)), dtype=torch.float64, device=dev))

    def split(self, u):
        shape = (-1, self.nv) + (self.N + 1,) * self.d
        return [_map(u, lambda t, v=v: t.reshape(shape)[:, v]) for v in range(self.nv)]

    def pairs(self, u, q, r, acc, scale):
        """acc += scale sum_m Dt_im f#(u_i, u_m) along direction r."""
        eq, ax, NP = self.eq, -1 - r, self.N + 1

        def at(xs, i):
            return [_map(x, lambda t: t.select(ax, i)) for x in xs]

        U, Q = [at(u, i) for i in range(NP)], [at(q, i) for i in range(NP)]
        G = [at(self.Ja[r], i) for i in range(NP)] if self.c["eq"] == "curved" else None
        mhd = self.c["eq"] == "mhd"
        out, div = [None] * NP, [None] * NP

        def add(store, i, j, f):
            k = self.num(scale * self.D[i, j], f[0])
            store[i] = [x * k for x in f] if store[i] is None else [
                s + x * k for s, x in zip(store[i], f)]

        for i in range(NP):
            for j in range(i, NP):
                if self.D[i, j] == 0 or (i == j and abs(self.D[i, i]) < 1e-15):
                    continue
                g = r if G is None else [(a + b) * 0.5 for a, b in zip(G[i], G[j])]
                f = eq.two_point(self.c["vf"], U[i], Q[i], U[j], Q[j], g)
                b = [(U[i][5 + r] + U[j][5 + r]) * 0.5] if mhd else None
                for a, e in ((i, j), (j, i)):
                    add(out, a, e, f)
                    if mhd:
                        add(div, a, e, b)
        # faces: this element's right one (and its left neighbour's)
        fax = self.d - 1 - r  # axis of the element counter after unflattening

        def shift(x, s):
            def f(t):
                e = t.reshape(tuple(self.n[::-1]) + t.shape[1:])
                return torch.roll(e, s, dims=fax).reshape(t.shape)
            return _map(x, f)

        UL, QL = U[NP - 1], Q[NP - 1]
        UR, QR = [shift(x, -1) for x in U[0]], [shift(x, -1) for x in Q[0]]
        g = r if G is None else G[NP - 1]
        fs = eq.surface(self.c["sf"], UL, QL, UR, QR, g)
        bs = [(UL[5 + r] + UR[5 + r]) * 0.5] if mhd else None
        k = self.num(scale * self.lift, fs[0])
        out[NP - 1] = [o + f * k for o, f in zip(out[NP - 1], fs)]
        out[0] = [o - shift(f, 1) * k for o, f in zip(out[0], fs)]
        if mhd:
            div[NP - 1] = [div[NP - 1][0] + bs[0] * k]
            div[0] = [div[0][0] - shift(bs[0], 1) * k]
        part = [_stack([out[i][v] for i in range(NP)], ax) for v in range(self.nv)]
        if mhd:  # the Powell term
            db = _stack([div[i][0] for i in range(NP)], ax)
            B, v = u[5:8], q[1:4]
            vB = v[0] * B[0] + v[1] * B[1] + v[2] * B[2]
            for m, x in zip(range(1, 8), B + [vB] + v):
                part[m] = part[m] + x * db
        return part if acc is None else [a + b for a, b in zip(acc, part)]

    def rhs(self, u, t=0.0):
        u = self.split(u)
        q, acc = self.eq.prim(u), None
        for r in range(self.d):
            scale = -np.longdouble(1) if self.c["eq"] == "curved" else -np.longdouble(self.n[r])
            acc = self.pairs(u, q, r, acc, scale)
        if self.c["eq"] == "curved":
            acc = [a * self.invJ for a in acc]
            phi = math.pi * (self.s - t)
            rho, dr = 2.0 + 0.1 * torch.sin(phi), 0.1 * math.pi * torch.cos(phi)
            dp = 0.4 * (2.0 * rho - 1.5) * dr
            src = [2 * dr, 2 * dr + dp, 2 * dr + dp, 2 * dr + dp, 4 * rho * dr + 3 * dp]
            acc = [a + DD(s) for a, s in zip(acc, src)]
        return _map(_stack(acc, 1), lambda x: x.reshape(-1))

    def dt(self, u):
        u = self.split(DD(u) if not isinstance(u, DD) else u)
        q = self.eq.prim(u)
        dims = tuple(range(1, self.d + 1))
        s = 0.0
        for r in range(self.d):
            if self.c["eq"] == "curved":
                g = self.Ja[r]
                lam = (_abs(self.eq.directed(g, q[1:4])) + self.eq.speed(u, q, r)
                       * _sqrt(self.eq.directed(g, g))) * self.invJ
                s = s + torch.amax(lam.hi, dims)
            else:
                lam = _abs(q[1 + r]) + self.eq.speed(u, q, r)
                s = s + self.n[r] * torch.amax(lam.hi, dims)
        return CFL * 2.0 / ((self.N + 1) * float(s.max()))

    def step(self, u):
        dt = self.dt(u)
        u, k = DD(u), None
        for a, b, cs in zip(RK_A, RK_B, RK_C):
            du = self.rhs(u, cs * dt) * dt
            k = du if k is None else k * a + du
            u = u + k * b
        return u.hi


def _exact_cost(c):
    if c["do"] == "ensemble":
        w = work(c)
        return w["flops"]
    return work(c)["flops"] * (2.0 if c["eq"] == "mhd" else 1.0)


def exact(case, seed):
    if _exact_cost(case) > 4.5e10:  # minutes of double-double work
        return None
    if case["do"] == "ensemble":
        m, us = _members(case, seed)
        out = []
        for (N, n), u in zip(m, us):
            c = _case("", "euler", "step", 3, N, (n, n, n), "ranocha", "llf", "wave")
            out.append(Operator(c).step(u))
        return torch.cat(out)
    u0 = _state(case, seed)
    if case["do"] == "rhs":
        return Operator(case).rhs(DD(u0)).hi
    if case["do"] == "grad":
        g = torch.Generator(device="cuda").manual_seed(int(seed) + 1)
        w = torch.randn(u0.shape, generator=g, device="cuda", dtype=torch.float64)
        u = u0.requires_grad_(True)
        Operator(case, dd=False).rhs(u).backward(w)
        return {"du": Operator(case).rhs(DD(u0.detach())).hi, "ubar": u.grad}
    return Operator(case).step(u0)
