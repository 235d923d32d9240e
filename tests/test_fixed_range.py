"""The integer kernels on data that spans many orders of magnitude.

Each variable is compared with the oracle node by node or plane by plane of an
element, relative to the largest entry there: a strong trace or node must not
cost a weak one its digits. The bar is the project's 1e-12 (some hundreds of
operations of 2^-53 on data whose sums do not cancel by more than a factor of a
hundred).
"""
import numpy as np
import pytest

BAR = 1e-12


def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import oracle
    oracle.build()
    return torch


def _mhd(rho, v, p, B):
    E = p / (5.0 / 3.0 - 1.0) + 0.5 * rho * (v ** 2).sum(0) + 0.5 * (B ** 2).sum(0)
    return np.ascontiguousarray(np.stack([rho, *(rho * v), E, *B], axis=1))


def _euler(rho, v, p):
    E = p / 0.4 + 0.5 * rho * (v ** 2).sum(0)
    return np.ascontiguousarray(np.stack([rho, *(rho * v), E], axis=1))


def _rhs(torch, eq, d, N, n, vf, sf, u):
    import oracle
    from paper_2108_06476_gb300 import Mesh, workloads as W
    m = Mesh(d, N, n, volume_flux=vf, surface_flux=sf, equations=eq)
    got = m.rhs(torch.from_numpy(u.reshape(-1)).cuda()).cpu().numpy().reshape(u.shape)
    assert m.check() == 0
    if eq == "mhd":
        ref = oracle.mhd_rhs(N, n, W.box(3), u.reshape(-1), sflux=sf, vflux=vf)
    else:
        ref = oracle.rhs(d, N, n, W.box(d), u.reshape(-1),
                         vflux={"ranocha": 0, "central": 2}[vf],
                         sflux={"llf": 0, "ranocha": 1, "hll": 2}[sf])
    return got, ref.reshape(u.shape)


@pytest.mark.gpu
@pytest.mark.parametrize("eq,d,vf,sf", [("euler", 3, "ranocha", "hll"), ("euler", 3, "central", "hll"),
                                        ("euler", 2, "central", "hll"), ("euler", 3, "ranocha", "llf"),
                                        ("mhd", 3, "central", "hll"), ("mhd", 3, "central", "llf")])
@pytest.mark.parametrize("ratio", [1.0, 60.0, 1e3, 1e6, 1e8])
@pytest.mark.parametrize("flow", ["right", "left", "slow"])
def test_faces_between_traces_of_different_size(eq, d, vf, sf, ratio, flow):
    # element by element along x cold and hot gas, both supersonic by their own
    # sound speeds (HLL: the face flux is the upwind trace's own) or slow; the
    # planes of nodes x = const of an element each by themselves (only the two
    # outer ones see a face's flux)
    torch = _gpu()
    N, n = 2, ((6, 11, 10) if d == 3 else (26, 24))
    ne, P = int(np.prod(n)), (N + 1) ** d
    rng = np.random.default_rng(int(ratio) + d)
    hot = (np.arange(ne) % n[0]) % 2 == 1
    rho = rng.uniform(0.7, 1.4, (ne, P))
    p = np.where(hot[:, None], ratio, 1.0) * rng.uniform(0.9, 1.1, (ne, P))
    c = np.sqrt(np.where(hot, ratio, 1.0))[:, None] * 1.5
    v = c * rng.uniform(-0.3, 0.3, (d, ne, P))
    if flow != "slow":
        v[0] += c * (2.0 if flow == "right" else -2.0)
    if eq == "mhd":
        u = _mhd(rho, v, p, 0.2 * c * rng.uniform(-1, 1, (3, ne, P)))
    else:
        u = _euler(rho, v, p)
    got, ref = _rhs(torch, eq, d, N, n, vf, sf, u)
    err, size = (np.abs(x).reshape(ne, u.shape[1], -1, N + 1).max(axis=2) for x in (got - ref, ref))
    err = err / size
    assert err.max() <= BAR, (err.max(axis=(0, 2)), np.unravel_index(err.argmax(), err.shape))


@pytest.mark.gpu
@pytest.mark.parametrize("N,n", [(1, (12, 11, 10)), (2, (4, 3, 3)), (3, (9, 9, 8)), (3, (3, 3, 3)),
                                 (4, (9, 9, 8)), (5, (3, 3, 2)), (7, (2, 2, 3))])
def test_mhd_lifting_cancels_before_it_is_rounded(N, n):
    # a nearly uniform flow, supersonic in every direction: the mass flux of
    # HLL at a face is the left trace's momentum, so the volume sum and the lifting nearly cancel. In integers
    # the 3 (N + 1) + 3 products of a node are each truncated by at most two
    # halves of a unit about their mean (0.41 units rms), units of 2^-60 times
    # the element's powers of two (at most 4 |D_01| and 2 |m|): below 2.1 units
    # = 2^-55.9 |D_01| |m| rms. Rounded to FP64 in between the sums would be
    # off by 0.29 2^-52 lift |m| = 2^-53.2 |D_01| |m| and more.
    torch = _gpu()
    from perf.cases import _lgl
    ne, P = int(np.prod(n)), (N + 1) ** 3
    rng = np.random.default_rng(N)
    rho, p = np.full((ne, P), 1.0), rng.uniform(0.99, 1.01, (ne, P))
    v = np.array([4.1, 5.3, 4.7])[:, None, None] * (1.0 + 1e-3 * rng.uniform(-1, 1, (3, ne, P)))
    u = _mhd(rho, v, p, np.array([0.3, 0.2, 0.1])[:, None, None] * np.ones((3, ne, P)))
    from paper_2108_06476_gb300 import Mesh
    m = Mesh(3, N, n, equations="mhd", volume_flux="central", surface_flux="hll")
    got = m.rhs(torch.from_numpy(u.reshape(-1)).cuda()).cpu().numpy().reshape(u.shape)[:, 0]
    _, w, D = _lgl(N)
    ref, size = 0, 0.0
    for r in range(3):
        a = 3 - r  # node axis of direction r in [e, k, j, i]
        mr = u[:, 1 + r].astype(np.longdouble).reshape(ne, N + 1, N + 1, N + 1)
        d = np.moveaxis(np.tensordot(mr, D, axes=([a], [1])), -1, a)
        e = mr.reshape(n[::-1] + mr.shape[1:])
        last = np.take(e, [N], axis=a + 2)
        from_left = np.roll(last, 1, axis=2 - r).reshape(np.take(mr, [0], axis=a).shape)
        first = [slice(None)] * 4
        first[a] = slice(0, 1)
        d[tuple(first)] -= (from_left - mr[tuple(first)]) / w[0]
        ref = ref - n[r] * d
        size = max(size, float(n[r] * abs(D[0, 1]) * np.abs(mr).max()))
    rms = float(np.sqrt(np.mean((got.reshape(ref.shape) - ref) ** 2)))
    assert rms <= 2.0 ** -55 * size, rms / size


@pytest.mark.gpu
@pytest.mark.parametrize("sf", ["llf", "hll"])
@pytest.mark.parametrize("field", [(1.0, 0.0, 0.0), (1.29, 1e-3, 0.0), (0.0, 0.0, 1.0), (1e-4, 1e-5, 0.0)])
@pytest.mark.parametrize("flow", [(3.0, 0.3, 0.3), (30.0, 3.0, 3.0), (300.0, 30.0, 30.0),
                                  (1000.0, 100.0, 100.0), (0.3, 3.0, 0.0)])
def test_fast_speed_where_kinetic_energy_dominates(sf, field, flow):
    # p = 1, so the energy is up to 1e6 p; B = 1.29: sound and Alfven speeds
    # nearly equal, where the discriminant of the fast speed nearly vanishes.
    # Velocities vary by 30%, so nothing cancels by more than a factor of ten.
    # lambda = |v_n| + c_f carries the pressure's error 2^-53 E/p times
    # c_f/(2 lambda): below 2e-13 for every flow here
    torch = _gpu()
    N, n = 3, (4, 3, 3)
    ne, P = 36, 64
    rng = np.random.default_rng(5)
    rho, p = np.ones((ne, P)), rng.uniform(0.99, 1.01, (ne, P))
    v = np.array(flow)[:, None, None] * (1.0 + 0.3 * rng.uniform(-1, 1, (3, ne, P)))
    u = _mhd(rho, v, p, np.array(field)[:, None, None] * np.ones((3, ne, P)))
    got, ref = _rhs(torch, "mhd", 3, N, n, "central", sf, u)
    size = np.abs(ref).max(axis=2)
    err = np.abs(got - ref).max(axis=2) / np.where(size > 0, size, 1.0)
    assert err.max() <= BAR, err.max(axis=0)


def _corner(eq, d, N, ne, kind, rng, factor=1e8):
    # random states with one corner node of every element, or all the others,
    # far away; and the nodes whose lines do not reach that corner or a face
    P = (N + 1) ** d
    rho, p = rng.uniform(0.8, 1.2, (2, ne, P))
    v, B = rng.uniform(-0.3, 0.3, (d, ne, P)), rng.uniform(-0.5, 0.5, (3, ne, P))
    last = P - 1
    if kind == "pressure":
        p[:, last] *= factor
    if kind == "density":  # the same momentum
        rho[:, last] *= factor
        v[:, :, last] /= factor
    if kind == "velocity":
        v[:, :, :last] /= factor
    if kind == "field":
        B[:, :, :last] /= factor
    if kind == "all":
        rho[:, last] *= factor
        p[:, last] *= factor
    if kind == "rest":  # exact zeros in place of small values
        v[:, :, :last] = 0.0
    if kind == "vacuum field":
        B[:, :, :last] = 0.0
    i = np.arange(P)
    inner = np.ones(P, bool)
    for k in range(d):
        c = i // (N + 1) ** k % (N + 1)
        inner &= (c != 0) & (c != N)
    return (_mhd(rho, v, p, B) if eq == "mhd" else _euler(rho, v, p)), inner


def _check_corner(torch, eq, d, N, n, vf, sf, kind):
    ne = int(np.prod(n))
    u, inner = _corner(eq, d, N, ne, kind, np.random.default_rng([d, N, 3]))
    got, ref = _rhs(torch, eq, d, N, n, vf, sf, u)
    size = np.abs(ref[:, :, inner]).max(axis=(0, 2))
    err = np.abs(got - ref)[:, :, inner].max(axis=(0, 2))
    assert (err[size == 0.0] == 0.0).all(), err
    assert (err <= BAR * size).all(), err / np.where(size > 0, size, 1.0)


@pytest.mark.gpu
@pytest.mark.parametrize("d,N,n", [(2, 2, (26, 25)), (2, 5, (25, 26)), (3, 2, (9, 9, 8)),
                                   (3, 3, (9, 9, 8)), (3, 4, (9, 9, 8)), (3, 7, (9, 9, 8))])
@pytest.mark.parametrize("kind", ["pressure", "density", "velocity", "all", "rest"])
def test_weak_form_far_from_a_strong_corner(d, N, n, kind):
    _check_corner(_gpu(), "euler", d, N, n, "central", "hll", kind)


@pytest.mark.gpu
@pytest.mark.parametrize("N,n", [(2, (3, 2, 2)), (2, (9, 9, 8)), (3, (3, 2, 2)), (3, (9, 9, 8)),
                                 (4, (9, 9, 8)), (7, (2, 2, 2))])
@pytest.mark.parametrize("kind", ["pressure", "density", "velocity", "field", "all", "rest",
                                  "vacuum field"])
def test_mhd_weak_form_far_from_a_strong_corner(N, n, kind):
    _check_corner(_gpu(), "mhd", 3, N, n, "central", "hll", kind)


@pytest.mark.gpu
@pytest.mark.parametrize("d,N,n", [(2, 2, (3, 4)), (2, 2, (26, 25)), (2, 3, (4, 4)), (2, 3, (26, 25)),
                                   (2, 6, (25, 26)), (3, 2, (3, 2, 3)), (3, 2, (9, 9, 8)),
                                   (3, 3, (4, 3, 3)), (3, 3, (9, 9, 8)), (3, 4, (9, 9, 8)),
                                   (3, 5, (3, 2, 2)), (3, 7, (2, 2, 2)), (3, 7, (9, 9, 8))])
@pytest.mark.parametrize("kind", ["pressure", "velocity", "rest", "both ratios"])
def test_two_point_flux_far_from_a_strong_corner(d, N, n, kind):
    torch = _gpu()
    if kind != "both ratios":
        return _check_corner(torch, "euler", d, N, n, "ranocha", "llf", kind)
    # density and internal energy both 2^5.9 higher at the corner: the pressure
    # 2^11.8 times, inside the limits of the first two. The other nodes' rows of
    # momentum are sums of their pressure's rounding, 2^-53 to 2^-52 times the
    # coefficients' row sums (up to 60 in units of 2/h)
    ne, P = int(np.prod(n)), (N + 1) ** d
    rng = np.random.default_rng([d, N, 4])
    rho, p = np.ones((ne, P)), np.ones((ne, P))
    rho[:, P - 1], p[:, P - 1] = 2.0 ** 5.9, 2.0 ** 11.8
    u = _euler(rho, 1e-3 * rng.uniform(-1, 1, (d, ne, P)), p)
    inner = _corner("euler", d, N, ne, "none", rng)[1]
    got, ref = _rhs(torch, "euler", d, N, n, "ranocha", "llf", u)
    err = np.abs(got - ref)[:, 1:d + 1, inner].max()
    assert err <= 2.0 ** -51 * 60 * max(n), err


@pytest.mark.gpu
@pytest.mark.parametrize("N,n", [(2, (3, 2, 2)), (3, (9, 9, 8)), (4, (9, 9, 8)), (5, (2, 3, 2))])
@pytest.mark.parametrize("kind", ["pressure", "velocity", "rest"])
def test_warped_box_far_from_a_strong_corner(N, n, kind):
    torch = _gpu()
    import oracle
    from paper_2108_06476_gb300 import Mesh
    ne = int(np.prod(n))
    u, inner = _corner("euler", 3, N, ne, kind, np.random.default_rng([N, 6]))
    m = Mesh(3, N, n, warp=0.02, surface_flux="ranocha")
    geom = oracle.CurvedGeometry(N, n, 0.02)
    m.set_nodes(torch.from_numpy(geom.X).cuda())
    m.set_metric(torch.from_numpy(geom.Ja).cuda(), torch.from_numpy(geom.J).cuda())
    got = m.rhs(torch.from_numpy(u.reshape(-1)).cuda()).cpu().numpy().reshape(u.shape)
    ref = oracle.curved_rhs(geom, u.reshape(-1), sflux=1).reshape(u.shape)
    size = np.abs(ref[:, :, inner]).max(axis=(0, 2))
    err = np.abs(got - ref)[:, :, inner].max(axis=(0, 2))
    assert (err <= BAR * size).all(), err / np.where(size > 0, size, 1.0)


@pytest.mark.gpu
@pytest.mark.parametrize("N,n", [(2, (3, 2, 2)), (2, (9, 9, 8)), (3, (3, 2, 2)), (3, (9, 9, 8)),
                                 (4, (9, 9, 8)), (5, (3, 2, 2)), (7, (2, 2, 2))])
@pytest.mark.parametrize("kind", ["pressure", "velocity", "field", "rest", "vacuum field"])
def test_mhd_two_point_flux_far_from_a_strong_corner(N, n, kind):
    _check_corner(_gpu(), "mhd", 3, N, n, "ec", "ec", kind)


@pytest.mark.gpu
@pytest.mark.parametrize("d,N,n", [(2, 2, (3, 2)), (2, 5, (2, 2)), (3, 2, (2, 2, 2)), (3, 3, (2, 2, 1)),
                                   (3, 4, (2, 1, 1)), (3, 5, (2, 1, 1)), (3, 7, (1, 2, 1))])
@pytest.mark.parametrize("kind", ["probe", "mass probe", "spread", "momentum spread", "two probes",
                                  "slow"])
def test_gradient_far_from_a_strong_corner(d, N, n, kind):
    # the entries of J^T w at nodes whose lines do not reach the corner that
    # holds the large cotangents, each against w . (J e_j) by the oracle's exact
    # JVP; a probe's gradient is zero there
    torch = _gpu()
    import oracle
    from paper_2108_06476_gb300 import Mesh, workloads as W
    ne, P = int(np.prod(n)), (N + 1) ** d
    rng = np.random.default_rng([d, N, 8])
    u, inner = _corner("euler", d, N, ne, "velocity" if kind == "slow" else "none", rng)
    w = rng.standard_normal((ne, d + 2, P))
    if kind in ("probe", "mass probe"):
        w[:, :, :P - 1] = 0.0
    if kind == "mass probe":
        w[:, 1:] = 0.0
    if kind == "spread":
        w[:, :, :P - 1] *= 1e-9
    if kind == "momentum spread":
        w[:, 1:d + 1, :P - 1] *= 1e-9
        w[:, [0, d + 1]] = 0.0
    if kind == "two probes":  # energy cotangents everywhere, a large mass cotangent at the corner
        w[:, :d + 1] = 0.0
        w[:, 0, P - 1] = 1e9
    m = Mesh(d, N, n, surface_flux="ranocha")
    ub = m.rhs_vjp(torch.from_numpy(u.reshape(-1)).cuda(),
                   torch.from_numpy(w.reshape(-1)).cuda()).cpu().numpy().reshape(w.shape)
    if "probe" in kind and kind != "two probes":
        assert not ub[:, :, inner].any()
    at = np.flatnonzero(inner)
    for _ in range(12):
        e, v, j = rng.integers(ne), rng.integers(d + 2), rng.choice(at)
        t = np.zeros_like(u)
        t[e, v, j] = 1.0
        jv = oracle.rhs_jvp(d, N, n, W.box(d), u.reshape(-1), t.reshape(-1),
                            sflux=1).reshape(u.shape)
        size = np.abs(w * jv).sum()
        assert abs(ub[e, v, j] - (w * jv).sum()) <= BAR * size, (e, v, j, ub[e, v, j], size)


@pytest.mark.gpu
@pytest.mark.parametrize("eq,d,N,n,vf,sf", [("euler", 2, 3, (4, 4), "ranocha", "llf"),
                                            ("euler", 3, 2, (9, 9, 8), "ranocha", "ranocha"),
                                            ("euler", 3, 3, (4, 3, 3), "ranocha", "hll"),
                                            ("euler", 3, 3, (9, 9, 8), "ranocha", "llf"),
                                            ("euler", 3, 5, (9, 9, 8), "ranocha", "llf"),
                                            ("euler", 2, 4, (26, 25), "central", "hll"),
                                            ("euler", 3, 4, (9, 9, 8), "central", "llf"),
                                            ("mhd", 3, 2, (3, 3, 2), "central", "hll"),
                                            ("mhd", 3, 3, (9, 9, 8), "central", "llf"),
                                            ("mhd", 3, 4, (9, 9, 8), "ec", "ec"),
                                            ("mhd", 3, 5, (2, 3, 2), "ec", "ec")])
@pytest.mark.parametrize("units", [(1.0, 1.0), (1e-20, 1e6), (1e18, 1e-4), (1.0, 1e9)])
def test_each_variable_by_itself_in_any_units(eq, d, N, n, vf, sf, units):
    # density and velocity units: the variables' sizes lie up to 18 orders of
    # magnitude apart, and every one has exponents of its own
    torch = _gpu()
    ne, P = int(np.prod(n)), (N + 1) ** d
    rng = np.random.default_rng([d, N, 11])
    r, c = units
    rho = r * np.exp(rng.uniform(-0.5, 0.5, (ne, P)))
    p = r * c * c * np.exp(rng.uniform(-0.5, 0.5, (ne, P)))
    v = c * rng.uniform(-0.8, 0.8, (d, ne, P))
    if eq == "mhd":
        u = _mhd(rho, v, p, np.sqrt(r) * c * rng.uniform(-0.8, 0.8, (3, ne, P)))
    else:
        u = _euler(rho, v, p)
    got, ref = _rhs(torch, eq, d, N, n, vf, sf, u)
    err = np.abs(got - ref).max(axis=2) / np.abs(ref).max(axis=2)
    assert err.max() <= BAR, err.max(axis=0)
