// The adjoint of Ranocha's volume flux in 64-bit fixed point (FP64 meshes), in
// the layout and with the scales of dg_fixed_volume.cuh. In FP64 a pair costs
// 376 instructions of the FP64 unit (64 cycles each): 1.98 ms of the 2.07 ms
// that one call takes at 16^3 N = 4. Here it costs none: 0.244 ms, the warps'
// issue slots 44% busy (16 warps per SM by registers and shared memory). The
// gradient of one rhs there (rhs, face adjoints, this) went from 2.07 to 0.46
// ms.
//
// With T(D) = tanh(D/2)/(D/2), S(D) = D/sinh(D), D the difference of ln rho or
// of ln e, means rho_m, e_m, v_m of the two nodes and R = rho_m T, the flux is
//   f_0 = R v_m,n,   f_k = f_0 v_m,k + delta_kn p_m,
//   f_E = f_0 eps + (p_a v_b,n + p_b v_a,n)/2,   eps = v_a.v_b/2 + e_m S,
// as a function of rho, v, p and e taken as independent. For the cotangent g,
//   F = g_0 + sum_k g_k v_m,k + g_E eps          (of f_0)
//   v_a,k:  g_k f_0/2 + g_E f_0 v_b,k/2, and for n also F R/2 + g_E p_b/2
//   p_a:    g_n/2 + g_E v_b,n/2
//   rho_a:  F v_m,n T/2 -+ F v_m,n rho_m T'/rho_a
//   e_a:    g_E f_0 S/2 -+ g_E f_0 e_m S'/e_a       (- for a, + for b)
// The sums of the terms over rho_a and e_a are kept apart and divided once per
// node, in FP64, where e = p/((gamma-1) rho) is differentiated too. T' and S'
// come from polynomials for T'/D and S'/D, as T and S do.
//
// Included by dg_vjp_kernels.cuh.
#pragma once

namespace dg {
namespace fx {

static __constant__ i64 kTanhDFar[] = DG_FX_TanhDFar, kSinhDFar[] = DG_FX_SinhDFar;

// a mean factor 1 + c (c in 2^-63) and its derivative with respect to D (2^-64)
struct Mean {
  i64 c, d;
};
__device__ __forceinline__ Mean tanh_short_d(i64 D) {
  const i64 k[] = DG_FX_TanhDShort;
  const int k32[] = DG_FX_TanhDShort32;
  const Limbs d = limbs(D << 3), x = limbs(sqr(d));
  return {tanh_short(x) >> 1, mul(d, limbs(short_poly(x, k, k32))) << 2};
}
__device__ __forceinline__ Mean sinh_short_d(i64 D) {
  const i64 k[] = DG_FX_SinhDShort;
  const int k32[] = DG_FX_SinhDShort32;
  const Limbs d = limbs(D << 3), x = limbs(sqr(d));
  return {sinh_short(x), mul(d, limbs(short_poly(x, k, k32))) << 2};
}
__device__ __forceinline__ Mean tanh_any_d(i64 D) {
  if (!d_mid((int)(D >> 32)))
    return {far_poly(D, kTanhFar) << 2, mul(limbs(D), limbs(far_poly(D, kTanhDFar))) << 7};
  const i64 c[] = DG_FX_TanhMid, k[] = DG_FX_TanhDMid;
  const Limbs d = limbs(D << 3), x = limbs(sqr(d));
  return {mul(x, limbs(mid_poly<kTanhMidN>(x, c))) >> 1,
          mul(d, limbs(mid_poly<kTanhDMidN>(x, k))) << 2};
}
__device__ __forceinline__ Mean sinh_any_d(i64 D) {
  if (!d_mid((int)(D >> 32)))
    return {far_poly(D, kSinhFar) << 2, mul(limbs(D), limbs(far_poly(D, kSinhDFar))) << 7};
  const i64 c[] = DG_FX_SinhMid, k[] = DG_FX_SinhDMid;
  const Limbs d = limbs(D << 3), x = limbs(sqr(d));
  return {mul(x, limbs(mid_poly<kSinhMidN>(x, c))),
          mul(d, limbs(mid_poly<kSinhDMidN>(x, k))) << 2};
}

// Exponents of an element's cotangents and sums. |D_ab| < 2^ed, |w| of mass,
// momenta, energy < 2^x; with d the largest coefficient, a pair's |g| stays
// below 1.25 d |w| (2 d |w| at N = 1, where ed is one more) and the sum over a
// node's pairs below 2.5 d |w| per direction (row and column sums). A sum's
// exponent comes from the product of the element's largest values (FP64, one
// thread per element), not from the product of their powers of two, which
// would cost it 4 bits; it is raised where a term's own format needs it.
//   F (of f_0)        63 - F
//   A1 rho directly   63 - a     A2 over rho  62 - (F + ev + er)
//   B1 e directly     63 - b     B2 over e    61 - (ed + x_E + er + ev + ee)
//   p                 63 - p     v            63 - v
constexpr int kNone = -1000;  // the exponent of zero
struct VScale {
  Scale u;
  int x[3], F, a, b, p, v;
  int e2;              // of B2's format
  int sm, sv, se, ue;  // g_0, g_k v_m, g_E eps to F (ue: upwards)
  int vF, vg, ve, vp;  // F R, g_k f_0, g_E f_0 v, g_E p to v
  int pg, pe;          // g_n, g_E v to p
  int sa, sb;          // to A1, B1
  int zero;            // no cotangent: nothing to sum
};
__device__ __forceinline__ int exp_of(double x) {
  return x > 0.0 ? exp_above((unsigned)__double2hiint(x)) : kNone;
}
template <int D>
__device__ __forceinline__ VScale vjp_scale(const unsigned* key, const int* c, int ed,
                                            double dmax) {
  VScale s;
  s.u = element_scale(key, c);
  const unsigned lo = (kBias - 150u) << 20, hi = (kBias + 150u) << 20;
  auto up = [](unsigned k) { return k ? __hiloint2double((int)k + 1, 0) : 0.0; };
  double W[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const unsigned w = key[8 + k];
    s.x[k] = w ? exp_above(w) : kNone;
    W[k] = up(w);
    if (w && !(w > lo && w < hi)) s.u.ok = 0;
  }
  s.zero = s.x[0] == kNone && s.x[1] == kNone && s.x[2] == kNone;
  if (ed > 300 || ed < -300 || energy_far(s.u.em, key[7])) s.u.ok = 0;
  if (!s.u.ok || s.zero) return s;
  // pressures and energies by themselves (the scales that momentum and energy
  // fluxes need would cost them bits). Where kinetic energies exceed the
  // internal ones, from a Mach number between 1.3 and 2.6, the common exponents
  // cost more bits than FP64 loses (at Mach 3, N = 4 an error of 2.7e-15
  // against 1.0e-15): FP64 there
  const int er = s.u.er, ev = s.u.ev, em = exp_above(key[5]);
  const int ee = exp_above(key[2]) + 1;
  s.u.em = em;
  s.u.ee = ee;
  s.u.kv = ee - 2 * ev - 2;
  const int xm = ed + s.x[0], xv = ed + s.x[1], xe = ed + s.x[2];
  const double r = up(key[0]), e = up(key[2]), v = up(key[4]), p = up(key[5]);
  const double wv = W[1] + W[2] * v;
  const double Fb = dmax * (W[0] + (double)D * W[1] * v + W[2] * (e + 0.5 * D * v * v));
  s.F = max(max(exp_of(1.25 * Fb), xm + 1), xv + ev + 2);
  s.v = exp_of(1.25 * dmax * (D * wv * r * v + W[2] * p) + 1.25 * Fb * r);
  s.v = max(max(s.v, s.F + er), max(max(xv + er + ev + 1, xe + er + 2 * ev + 2), xe + em + 1));
  s.p = max(max(exp_of(1.25 * D * dmax * wv), xv), xe + ev + 1);
  s.a = max(exp_of(1.25 * D * Fb * v), s.F + ev);
  s.b = max(exp_of(1.25 * D * dmax * W[2] * r * v), xe + er + ev + 1);
  s.e2 = xe + er + ev + ee;
  auto cap = [](int n) { return n < 63 ? n : 63; };
  const int ne = s.F - xe - ee - 2;
  s.sm = cap(s.F - xm - 1);
  s.sv = cap(s.F - xv - ev - 2);
  s.se = cap(ne > 0 ? ne : 0);
  s.ue = ne < 0 ? -ne : 0;
  s.vF = cap(s.v - s.F - er);
  s.vg = cap(s.v - xv - er - ev - 1);
  s.ve = cap(s.v - xe - er - 2 * ev - 2);
  s.vp = cap(s.v - xe - em - 1);
  s.pg = cap(s.p - xv);
  s.pe = cap(s.p - xe - ev - 1);
  s.sa = cap(s.a - s.F - ev);
  s.sb = cap(s.b - xe - er - ev - 1);
  if (s.ue > 31 || s.u.kv < 0 || s.u.kv > 62 || max(s.v, max(s.a, s.e2)) > 900) s.u.ok = 0;
  return s;
}

// adjoints of one pair: what a node's sums gain (A2 and B2: minus for a, plus
// for b)
template <int D>
struct PairAdj {
  i64 A1, A2, B1, B2, pa, pb, va[D], vb[D];
};
// g: mass, momenta (normal first), energy, 62 - (ed + x)
template <int D>
__device__ __forceinline__ PairAdj<D> pair_adjoint(const Node<D>& a, const Node<D>& b,
                                                   const i64* g, const VScale& s) {
  PairAdj<D> o;
  const i64 dr = b.lr - a.lr, de = b.le - a.le;
  Mean t, h;
  if (d_short((int)(dr >> 32)) && d_short((int)(de >> 32))) {
    t = tanh_short_d(dr);
    h = sinh_short_d(de);
  } else {
    t = tanh_any_d(dr);
    h = sinh_any_d(de);
  }
  const i64 sr = a.r + b.r, se = a.e + b.e;
  const Limbs rm = limbs(sr), em = limbs(se), tc = limbs(t.c), hc = limbs(h.c);
  const Limbs R = limbs(sr + (mul(rm, tc) << 1));
  const i64 vm0 = a.v[0] + b.v[0];
  const Limbs vn = limbs(vm0), gE = limbs(g[D + 1]);
  const Limbs f0 = limbs(mul(R, vn) << 1);  // 63 - er - ev
  Limbs xa[D], xb[D];
  i64 some = g[0] | g[D + 1];
#pragma unroll
  for (int k = 0; k < D; ++k) some |= g[1 + k];
  // D: the shifted products' mean loss (where there is nothing but zeros, zero)
  i64 vv = 0, F = (g[0] >> s.sm) + (some ? D : 0);
#pragma unroll
  for (int k = 0; k < D; ++k) {
    xa[k] = limbs(a.v[k]);
    xb[k] = limbs(b.v[k]);
    vv = fma64(xa[k], xb[k], vv);
    const Limbs gk = limbs(g[1 + k]);
    F += mul(gk, k == 0 ? vn : limbs(a.v[k] + b.v[k])) >> s.sv;
    o.va[k] = mul(gk, f0) >> s.vg;
  }
  F += mul_up(gE, limbs(se + (mul(em, hc) << 1) + (vv >> s.u.kv)), s.ue) >> s.se;
  const Limbs Fl = limbs(F);
  const i64 E = mul(gE, f0);  // g_E f_0, 61 - (ed + x_E + er + ev)
  const Limbs E2 = limbs(E << 1);
#pragma unroll
  for (int k = 0; k < D; ++k) {
    o.vb[k] = o.va[k] + (mul(E2, xa[k]) >> s.ve);
    o.va[k] += mul(E2, xb[k]) >> s.ve;
  }
  const i64 FR = mul(Fl, R) >> s.vF;
  o.va[0] += FR + (mul(gE, limbs(b.p << 1)) >> s.vp);
  o.vb[0] += FR + (mul(gE, limbs(a.p << 1)) >> s.vp);
  const i64 gp = g[1] >> s.pg;
  o.pa = gp + (mul(gE, limbs(b.v[0] << 1)) >> s.pe);
  o.pb = gp + (mul(gE, limbs(a.v[0] << 1)) >> s.pe);
  const i64 Rb = mul(Fl, vn);
  const Limbs R2 = limbs(Rb << 1);
  o.A1 = fma64(R2, tc, Rb) >> s.sa;
  o.A2 = mul(limbs(mul(R2, limbs(t.d))), rm);
  o.B1 = fma64(E2, hc, E) >> s.sb;
  o.B2 = mul(limbs(mul(E2, limbs(h.d))), em);
  return o;
}

}  // namespace fx

// slots of a node: the staged values of fx_stage_node or rho, e, p, v (FP64),
// then w; sums A1, A2, B1, B2, p, v (fixed point) or rho, -, -, -, p, v (FP64)
template <int D, int N>
struct VjpFx {
  using T = Tourney<N>;
  static constexpr int NV = D + 2, P = Shape<D, N>::P, LINES = Shape<D, N>::LINES;
  static constexpr int W = 5 + D, SL = W + NV, ELEM = (SL + 5 + D) * P * 8;
  static constexpr int threads(int epb) { return 32 * ((epb * LINES + T::LPW - 1) / T::LPW); }
  // elements per CTA: the count for which the warps an SM holds (shared
  // memory, 20 warps at 100 registers) have the most lines; of equals the one
  // with a tenth more of its lanes in use (3D N = 4: 5 elements in 8 warps, not
  // 2 in 4), else the smallest
  static constexpr int score(int epb) {
    const int warps = threads(epb) / 32;
    const int by_smem = 229376 / (epb * ELEM + 2048), by_warps = 20 / warps;
    const int ctas = by_smem < by_warps ? by_smem : by_warps;
    return ctas * epb * LINES;
  }
  static constexpr bool fuller(int e, int b) {
    return e * threads(b) * 10 > b * threads(e) * 11 && score(e) * 21 >= score(b) * 20;
  }
  static constexpr int best() {
    int b = 1;
    for (int e = 2; e <= 16; ++e)
      if (threads(e) <= 512 && e * ELEM <= 200000 &&
          (score(e) * 20 > score(b) * 21 || fuller(e, b)))
        b = e;
    return b;
  }
  static constexpr int EPB = best();
  // where sum j starts: the units by which its truncated products and shifts
  // fall short on average (A2 and B2: none on average)
  __device__ __forceinline__ static constexpr int start(int j) {
    return j == 1 || j == 3 ? 0 : j < 5 ? 3 * D * N / 2 : (2 * D + 3) * N / 2;
  }
};

// Whether what a node's sums come from lies too far below the units of its
// element (at sp; cross_far): its velocities, or any class of cotangents while
// another one on its lines is not zero (the classes' terms share exponents)
template <int D, int N>
__device__ __forceinline__ bool vjp_far_node(const double* sp, const unsigned* key, int node) {
  using V = VjpFx<D, N>;
  auto most = [&](int at, int n, int cnt) {
    unsigned m = 0;
    for (int j = 0; j < cnt; ++j)
      m = max(m, (unsigned)__double2hiint(sp[(at + j) * V::P + n]) & 0x7fffffffu);
    return m;
  };
  const int at[4] = {3, V::W, V::W + 1, V::W + 1 + D}, cnt[4] = {D, 1, D, 1};
  // most nodes, or one of the first on their lines, are near enough themselves
  bool near = true;
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const unsigned top = key[c ? 7 + c : 4];
    near = near &&
           (top - most(at[c], node, cnt[c]) <= (kCrossBits << 20) ||
            cross_max<D, N>(node, [&](int n) { return most(at[c], n, cnt[c]); }, top) != 0u);
  }
  if (near) return false;
  bool some = false, far = false;
#pragma unroll 1
  for (int c = 0; c < 4; ++c) {
    const unsigned top = key[c ? 7 + c : 4];
    const unsigned m = cross_max<D, N>(node, [&](int n) { return most(at[c], n, cnt[c]); });
    if (c == 0) {
      if (cross_far(top, m)) return true;
    } else {
      some = some || m != 0u;
      far = far || top - m > (kCrossBits << 20);
    }
  }
  return some && far;
}

template <int D, int N>
__device__ __forceinline__ void vjp_fx_pair(unsigned char* elem, const fx::VScale& sc,
                                            const fx::Limbs (*ds)[kNPMax],
                                            const double (*ds64)[kNPMax], double gm1inv, int dir,
                                            int l, int a, int b) {
  using V = VjpFx<D, N>;
  constexpr int P = V::P, NV = V::NV;
  const int na = line_node_rt<D, N>(dir, l, a), nb = line_node_rt<D, N>(dir, l, b);
  const int t1 = dir + 1 == D ? 0 : dir + 1, t2 = D == 2 ? t1 : (t1 + 1 == D ? 0 : t1 + 1);
  const int dk[3] = {dir, t1, t2};
  int comp[NV];  // of each normal-first variable
  comp[0] = 0;
#pragma unroll
  for (int k = 0; k < D; ++k) comp[1 + k] = (1 + dk[k]) * P;
  comp[D + 1] = (D + 1) * P;
  if (sc.u.ok) {
    const fx::i64* sx = reinterpret_cast<const fx::i64*>(elem);
    fx::i64* sa = reinterpret_cast<fx::i64*>(elem) + V::SL * P;
    const fx::Limbs dab = ds[a][b], dba = ds[b][a];
    fx::i64 g[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const fx::i64* sw = sx + V::W * P + comp[v];
      g[v] = fx::fma64(dab, fx::limbs(sw[na]), fx::mul(dba, fx::limbs(sw[nb])));
    }
    const fx::PairAdj<D> o = fx::pair_adjoint<D>(fx_node<D, N>(sx, dir, t1, t2, na),
                                                 fx_node<D, N>(sx, dir, t1, t2, nb), g, sc);
    sa[na] += o.A1;
    sa[nb] += o.A1;
    sa[P + na] -= o.A2;
    sa[P + nb] += o.A2;
    sa[2 * P + na] += o.B1;
    sa[2 * P + nb] += o.B1;
    sa[3 * P + na] -= o.B2;
    sa[3 * P + nb] += o.B2;
    sa[4 * P + na] += o.pa;
    sa[4 * P + nb] += o.pb;
#pragma unroll
    for (int k = 0; k < D; ++k) {
      sa[(5 + dk[k]) * P + na] += o.va[k];
      sa[(5 + dk[k]) * P + nb] += o.vb[k];
    }
  } else {
    const double* sp = reinterpret_cast<const double*>(elem);
    double* sa = reinterpret_cast<double*>(elem) + V::SL * P;
    const double dab = ds64[a][b], dba = ds64[b][a];
    double qa[NV], qb[NV], g[NV], ga[NV], gb[NV];
    qa[0] = sp[na];
    qb[0] = sp[nb];
    qa[D + 1] = sp[2 * P + na];
    qb[D + 1] = sp[2 * P + nb];
#pragma unroll
    for (int k = 0; k < D; ++k) {
      qa[1 + k] = sp[(3 + dk[k]) * P + na];
      qb[1 + k] = sp[(3 + dk[k]) * P + nb];
    }
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const double* sw = sp + V::W * P + comp[v];
      g[v] = dab * sw[na] + dba * sw[nb];
      ga[v] = gb[v] = 0.0;
    }
    ranocha_pair_rev<double, D>(qa, qb, g, gm1inv, ga, gb);
    sa[na] += ga[0];
    sa[nb] += gb[0];
    sa[4 * P + na] += ga[D + 1];
    sa[4 * P + nb] += gb[D + 1];
#pragma unroll
    for (int k = 0; k < D; ++k) {
      sa[(5 + dk[k]) * P + na] += ga[1 + k];
      sa[(5 + dk[k]) * P + nb] += gb[1 + k];
    }
  }
}

template <int D, int N>
__global__ void __launch_bounds__(VjpFx<D, N>::threads(VjpFx<D, N>::EPB),
                                  640 / VjpFx<D, N>::threads(VjpFx<D, N>::EPB) < 1
                                      ? 1
                                      : 640 / VjpFx<D, N>::threads(VjpFx<D, N>::EPB))
    vjp_volume_fx_kernel(const double* __restrict__ u, const double* __restrict__ w,
                         double* __restrict__ ubar, const double* __restrict__ fb, Geom g,
                         Tables<double> tb) {
  using V = VjpFx<D, N>;
  using T = Tourney<N>;
  constexpr int NP = N + 1, P = V::P, NV = V::NV, LINES = V::LINES, EPB = V::EPB;
  extern __shared__ __align__(16) unsigned char dg_smem[];
  __shared__ fx::Limbs s_d[D][kNPMax][kNPMax];  // 63 - ed
  __shared__ double s_d64[D][kNPMax][kNPMax];
  __shared__ fx::VScale s_scale[EPB];
  __shared__ unsigned s_key[EPB][11];  // those of FxShared, then the cotangents'
  const int e0 = blockIdx.x * EPB;
  const int count = (int)g.nelem - e0 < EPB ? (int)g.nelem - e0 : EPB;
  const int t = threadIdx.x;
  if (t < count) {
    fx_clear_key(s_key[t]);
    s_key[t][8] = s_key[t][9] = s_key[t][10] = 0u;
  }
  const int ed = fx_table_exponent<D>(tb) + (N == 1);
  for (int i = t; i < D * NP * NP; i += blockDim.x) {
    const int k = i / (NP * NP), r = i / NP % NP, c = i % NP;
    s_d64[k][r][c] = tb.Ds[k][r][c];
    s_d[k][r][c] = fx::limbs(fx::half_fixed(tb.Ds[k][r][c], ed) << 1);
  }
  int cb[2];
  fx::scale_bits(g.gm1, cb);
  __syncthreads();
  unsigned bad = 0;
  for (int t0 = t & ~31; t0 < count * P; t0 += blockDim.x) {
    const int i = t0 + (t & 31);
    const bool in = i < count * P;
    const int el = i / P, node = i % P;
    FxKeys k = {};
    unsigned kw[3] = {0u, 0u, 0u};
    if (in) {
      double c[NV];
      double* sp = reinterpret_cast<double*>(dg_smem + el * V::ELEM) + node;
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        const long long idx = ((long long)(e0 + el) * NV + v) * P + node;
        c[v] = u[idx];
        const double x = w[idx];
        const int cl = v == 0 ? 0 : v <= D ? 1 : 2;
        sp[(V::W + v) * P] = x;
        kw[cl] = max(kw[cl], (unsigned)__double2hiint(x) & 0x7fffffffu);
      }
      const FxPrim<D> q = fx_prim<D>(c, g, bad);
      k = fx_keys<D>(q);
      sp[0] = q.rho;
      sp[P] = q.e;
      sp[2 * P] = q.p;
#pragma unroll
      for (int j = 0; j < D; ++j) sp[(3 + j) * P] = q.v[j];
    }
    const int last = (t0 + 31 < count * P ? t0 + 31 : count * P - 1) / P;
    for (int ek = t0 / P; ek <= last; ++ek) {
      const bool mine = in && el == ek;
      fx_merge_keys(k, mine, s_key[ek]);
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        const unsigned m = __reduce_max_sync(0xffffffffu, mine ? kw[j] : 0u);
        if ((t & 31) == 0) atomicMax(&s_key[ek][8 + j], m);
      }
    }
  }
  __syncthreads();
  if (t < count) {
    double dmax = 0.0;
#pragma unroll
    for (int k = 0; k < D; ++k) dmax = ::fmax(dmax, ::fabs(tb.Ds[k][0][1]));
    s_scale[t] = fx::vjp_scale<D>(s_key[t], cb, ed, N == 1 ? 2.0 * dmax : dmax);
  }
  __syncthreads();
  for (int i = t; i < count * P; i += blockDim.x) {
    const int el = i / P;
    if (vjp_far_node<D, N>(reinterpret_cast<const double*>(dg_smem + el * V::ELEM), s_key[el],
                           i % P))
      s_scale[el].u.ok = 0;
  }
  __syncthreads();
  for (int i = t; i < count * P; i += blockDim.x) {
    const int el = i / P;
    const fx::VScale& sc = s_scale[el];
    double* sp = reinterpret_cast<double*>(dg_smem + el * V::ELEM) + i % P;
    fx::i64* sx = reinterpret_cast<fx::i64*>(sp);
    if (sc.u.ok) {
      const double rho = sp[0], e = sp[P], p = sp[2 * P];
      double v[D];
#pragma unroll
      for (int j = 0; j < D; ++j) v[j] = sp[(3 + j) * P];
      sx[0] = fx::half_fixed(rho, sc.u.er);
      sx[P] = fx::ln_fixed(rho, sc.u.er);
      sx[2 * P] = fx::half_fixed(e, sc.u.ee);
      sx[3 * P] = fx::ln_fixed(e, sc.u.ee);
      sx[4 * P] = fx::half_fixed(p, sc.u.em);
#pragma unroll
      for (int j = 0; j < D; ++j) sx[(5 + j) * P] = fx::half_fixed(v[j], sc.u.ev);
#pragma unroll
      for (int j = 0; j < NV; ++j) {
        const int x = sc.x[j == 0 ? 0 : j <= D ? 1 : 2];
        sx[(V::W + j) * P] = x == fx::kNone ? 0 : fx::half_fixed(sp[(V::W + j) * P], x) << 1;
      }
    }
    fx::i64* sa = sx + V::SL * P;
#pragma unroll
    for (int j = 0; j < 5 + D; ++j) sa[j * P] = sc.u.ok ? V::start(j) : 0;
  }
  __syncthreads();
  const int lane = t & 31, slot = lane / T::LPW;
  const int ln = (t >> 5) * T::LPW + lane % T::LPW;
  const bool in = slot < T::T && ln < count * LINES;
  const int el = ln / LINES, l = ln % LINES;
#pragma unroll 1
  for (int dir = 0; dir < D; ++dir) {
#pragma unroll 1
    for (int m = 0; m < T::ROUNDS; ++m) {
      if (in && !(s_scale[el].u.ok && s_scale[el].zero)) {
        int a, b;
        tourney_pair<N>(m, slot, a, b);
        vjp_fx_pair<D, N>(dg_smem + el * V::ELEM, s_scale[el], s_d[dir], s_d64[dir], g.gm1inv,
                          dir, l, a, b);
      }
      __syncwarp();
    }
    __syncthreads();
  }
  const double gm1 = g.gm1;
  const int nelem = (int)g.nelem;
  for (int i = t; i < count * P; i += blockDim.x) {
    const int ell = i / P, node = i % P, e = e0 + ell;
    const fx::VScale& sc = s_scale[ell];
    const double* sp = reinterpret_cast<const double*>(dg_smem + ell * V::ELEM) + node;
    const fx::i64* sx = reinterpret_cast<const fx::i64*>(sp);
    const fx::i64* sa = sx + V::SL * P;
    double irho, v[D], vb[D], pb, rb;
    if (sc.u.ok) {
      const int er = sc.u.er, ev = sc.u.ev, ee = sc.u.ee;
      const double en = fx::to_double_int(sx[2 * P], ee - 62);
      irho = rcp(fx::to_double_int(sx[0], er - 62));
      // (a sum still at its start saw nothing but zeros)
      auto sum = [&](int j, int x) {
        return sa[j * P] == V::start(j) ? 0.0 : fx::to_double_int(sa[j * P], x);
      };
      const double eb = sum(2, sc.b - 63) + sum(3, sc.e2 - 61) * rcp(en);
      const double eir = eb * irho;
      pb = sum(4, sc.p - 63) + eir * g.gm1inv;
      rb = sum(0, sc.a - 63) + sum(1, sc.F + ev + er - 62) * irho - eir * en;
#pragma unroll
      for (int k = 0; k < D; ++k) {
        v[k] = fx::to_double_int(sx[(5 + k) * P], ev - 62);
        vb[k] = sum(5 + k, sc.v - 63);
      }
    } else {
      irho = 1.0 / sp[0];
      rb = __longlong_as_double(sa[0]);
      pb = __longlong_as_double(sa[4 * P]);
#pragma unroll
      for (int k = 0; k < D; ++k) {
        v[k] = sp[(3 + k) * P];
        vb[k] = __longlong_as_double(sa[(5 + k) * P]);
      }
    }
    // the adjoint of the conserved variables: ubar_rho = rhobar - sum_k
    // vbar_k v_k/rho + pbar (gamma-1) |v|^2/2, ubar_m_k = vbar_k/rho - pbar
    // (gamma-1) v_k, ubar_E = pbar (gamma-1)
    double val[NV], v2 = 0.0;
    const double pg = pb * gm1;
#pragma unroll
    for (int k = 0; k < D; ++k) {
      const double m = vb[k] * irho;
      v2 += v[k] * v[k];
      rb -= m * v[k];
      val[1 + k] = m - pg * v[k];
    }
    val[0] = rb + pg * half(v2);
    val[D + 1] = pg;
    const int c[3] = {node % NP, (node / NP) % NP, node / (NP * NP)};
#pragma unroll
    for (int dir = 0; dir < D; ++dir) {
      if (c[dir] != N && c[dir] != 0) continue;
      const int lf = (D == 2) ? ((dir == 0) ? c[1] : c[0])
                              : (dir == 0) ? (c[1] + NP * c[2])
                              : (dir == 1) ? (c[0] + NP * c[2]) : (c[0] + NP * c[1]);
      const long long ef = c[dir] == N ? e : neighbour32(g, e, dir, -1);
      const double* s = fb + (((long long)(dir * 2 + (c[dir] == 0)) * NV) * nelem + ef) * LINES + lf;
#pragma unroll
      for (int j = 0; j < NV; ++j) val[j] += s[(long long)j * nelem * LINES];
    }
#pragma unroll
    for (int j = 0; j < NV; ++j) ubar[((long long)e * NV + j) * P + node] = val[j];
  }
}

}  // namespace dg
