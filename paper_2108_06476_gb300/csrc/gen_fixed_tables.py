"""Writes dg_fixed_tables.cuh: the constants of the fixed-point flux kernels
(dg_fixed.cuh), from 60-digit arithmetic (mpmath).

* kLog: for the i-th of 128 equal intervals of [1, 2), an integer r with r/256
  near the reciprocal of the interval's midpoint, and -ln(r/256) as a 64-bit
  integer in units of 2^-60. With z = m r/256 - 1 (|z| < 2^-7) the kernel
  forms ln(m) = -ln(r/256) + ln(1 + z).
* TanhShort/TanhMid: the polynomial p with 1 - tanh(D/2)/(D/2) = x p(x),
  x = D^2, interpolated at the Chebyshev points of x in [0, 1/16] (|D| < 1/4)
  and [0, 1] (|D| < 1); coefficient k (of x^(k-1), k = 1, 2, ...) is negated
  and stored in units of 2^-(64 + 2k).
* SinhShort/SinhMid: the same for 1 - D/sinh(D), in units of 2^-(63 + 2k).
  The short polynomials' coefficients from the fourth on are 32-bit integers
  (units of 2^-(32 + 2k), one bit less for sinh).

* TanhFar/SinhFar: 1 - tanh(D/2)/(D/2) and 1 - D/sinh(D) on x in [0, 17.5]
  (|D| < 4.18, a ratio of 2^6) as polynomials in z = (x - 8.75)/16; the
  coefficients are negated and stored in units of 2^-61.

* TanhD*/SinhD*: the derivatives with respect to D of tanh(D/2)/(D/2) and
  D/sinh(D), divided by D, as polynomials in the same variables; coefficient k
  of x^k in units of 2^-(63 + 2k), far ones in 2^-61, all negated.

Usage: python gen_fixed_tables.py > dg_fixed_tables.cuh
"""
import mpmath as mp

mp.mp.dps = 60


def tanhc(x):
    if x == 0:
        return mp.mpf(1) / 12
    d = mp.sqrt(x)
    return (1 - mp.tanh(d / 2) / (d / 2)) / x


def sinhc(x):
    if x == 0:
        return mp.mpf(1) / 6
    d = mp.sqrt(x)
    return (1 - d / mp.sinh(d)) / x


def tanhd(x):  # -(d/dD tanh(D/2)/(D/2))/D
    if x < mp.mpf(10) ** -20:
        return mp.mpf(1) / 6
    d = mp.sqrt(x)
    return -(mp.sech(d / 2) ** 2 / d - 2 * mp.tanh(d / 2) / x) / d


def sinhd(x):  # -(d/dD D/sinh(D))/D
    if x < mp.mpf(10) ** -20:
        return mp.mpf(1) / 3
    d = mp.sqrt(x)
    return -(1 / mp.sinh(d) - d * mp.cosh(d) / mp.sinh(d) ** 2) / d


def fit(fun, a, n):
    nodes = [a * (1 + mp.cos(mp.pi * (2 * k + 1) / (2 * n))) / 2 for k in range(n)]
    V = mp.matrix([[x ** j for j in range(n)] for x in nodes])
    c = mp.lu_solve(V, mp.matrix([fun(x) for x in nodes]))
    return [c[j] for j in range(n)]


def worst(fun, c, a):
    e = mp.mpf(0)
    for k in range(1, 401):
        x = a * k / 400
        e = max(e, abs(x * (sum(cj * x ** j for j, cj in enumerate(c)) - fun(x))))
    return float(e)


def emit(name, fun, a, n, off, narrow_from=None):
    c = fit(fun, mp.mpf(a), n)
    q = [int(mp.nint(-cj * mp.mpf(2) ** (off + 2 * (k + 1)))) for k, cj in enumerate(c)]
    print(f"// x in [0, {a}], {n} coefficients: largest error {worst(fun, c, mp.mpf(a)):.1e}")
    if narrow_from is None:
        print(f"constexpr int k{name}N = {n};")
        print(f"#define DG_FX_{name} {{" + ", ".join(f"{v}LL" for v in q) + "}")
        return
    w = q[:narrow_from]
    s = [int(mp.nint(-cj * mp.mpf(2) ** (off - 32 + 2 * (k + 1)))) for k, cj in enumerate(c)]
    print(f"#define DG_FX_{name} {{" + ", ".join(f"{v}LL" for v in w) + "}")
    print(f"#define DG_FX_{name}32 {{" + ", ".join(str(v) for v in s[narrow_from:]) + "}")


def emit_far(name, fun, n, times_x=True):
    f0 = fun
    if not times_x:
        fun = lambda x: f0(x) / x if x else mp.mpf(0)  # noqa: E731
    a, h = mp.mpf("17.5"), mp.mpf("8.75")
    nodes = [a * (1 + mp.cos(mp.pi * (2 * k + 1) / (2 * n))) / 2 for k in range(n)]
    z = [(x - h) / 16 for x in nodes]
    V = mp.matrix([[y ** j for j in range(n)] for y in z])
    c = mp.lu_solve(V, mp.matrix([x * fun(x) for x in nodes]))
    e = max(abs(sum(c[j] * ((a * k / 400 - h) / 16) ** j for j in range(n))
                - (a * k / 400) * fun(a * k / 400)) for k in range(1, 401))
    q = [int(mp.nint(-c[k] * mp.mpf(2) ** 61)) for k in range(n)]
    assert sum(abs(v) * 0.547 ** k for k, v in enumerate(q)) < 2 ** 62.5
    print(f"// z = (x - 8.75)/16, {n} coefficients: largest error {float(e):.1e}")
    print(f"constexpr int kFarN = {n};" if name == "TanhFar"
          else f'static_assert(kFarN == {n}, "");')
    print(f"#define DG_FX_{name} {{" + ", ".join(f"{v}LL" for v in q) + "}")


def main():
    print("// written by gen_fixed_tables.py")
    print("#pragma once")
    print("namespace dg {\nnamespace fx {")
    emit("TanhShort", tanhc, "0.0625", 6, 64, 3)
    emit("SinhShort", sinhc, "0.0625", 6, 63, 3)
    emit("TanhMid", tanhc, "1", 11, 64)
    emit("SinhMid", sinhc, "1", 11, 63)
    emit_far("TanhFar", tanhc, 32)
    emit_far("SinhFar", sinhc, 32)
    emit("TanhDShort", tanhd, "0.0625", 6, 61, 3)
    emit("SinhDShort", sinhd, "0.0625", 6, 61, 3)
    emit("TanhDMid", tanhd, "1", 11, 61)
    emit("SinhDMid", sinhd, "1", 11, 61)
    emit_far("TanhDFar", tanhd, 32, False)
    emit_far("SinhDFar", sinhd, 32, False)
    print("struct __align__(16) LogEntry {\n  long long l;\n  int r, pad;\n};")
    rows, zmax = [], 0.0
    for i in range(128):
        r = int(mp.nint(256 / (1 + (mp.mpf(i) + 0.5) / 128)))
        if i == 0:
            r = 256  # 1 - z exact at 1: ln(1) = 0
        for e in (i, i + 1):
            zmax = max(zmax, abs(float((1 + mp.mpf(e) / 128) * r / 256 - 1)))
        rows.append("{%dLL, %d, 0}" % (int(mp.nint(-mp.log(mp.mpf(r) / 256) * mp.mpf(2) ** 60)), r))
    print(f"// largest |z|: {zmax:.5f}")
    print("#define DG_FX_LOG_ROWS \\\n  " + ", \\\n  ".join(
        ", ".join(rows[i:i + 3]) for i in range(0, 128, 3)))
    print("constexpr long long kLn2 = %dLL;  // 2^-60" % int(mp.nint(mp.log(2) * mp.mpf(2) ** 60)))
    print("}  // namespace fx\n}  // namespace dg")


if __name__ == "__main__":
    main()
