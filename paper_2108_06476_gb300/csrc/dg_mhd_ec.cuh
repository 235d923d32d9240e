// EC flux differencing for MHD in 64-bit fixed point: the two-point flux of
// mhd_ec_flux on integers scaled by per-element powers of two (dg_fixed.cuh;
// in FP64 a pair takes about 100 instructions, 64 cycles each of the
// sub-partition's FP64 unit), the pairs of a line spread over (N + 1)/2
// threads as in dg_fixed_volume.cuh.
//
// The flux's quotient needs no division: with beta = rho/(2p) = 1/(2
// (gamma-1) e), e the internal energy and D = ln e_b - ln e_a,
//   ({rho} + {beta |B|^2})/(2 {beta}) = {p_t} - [[p_t]]/2 tanh(D/2),
// p_t = p + |B|^2/2, [[a]] = a_b - a_a (beta_a/(beta_a + beta_b) = (1 +
// tanh(D/2))/2), and 1/(2 (gamma-1) beta_ln) = {e} D/sinh(D).
//
// Included by dg_mhd.cu. 20^3 N = 4: volume kernel 1.13 ms in FP64, 0.33 here,
// faces 0.18 and 0.07 ms; 4^3 N = 7 (directions on warps of their own): 144 and
// 42 us.
#pragma once

// rho < 2^er, |v_k| < 2^ev, |B_k| < 2^eb, e < 2^(ee - 1), pressures and
// momentum fluxes by em, energy fluxes by em + ev
struct MEScale {
  int er, ev, eb, ee, em;
  int ok;
};

// node values: r = rho/2 (63 - er), e/2 (63 - ee), pt/2 (63 - em), v/2 (63 -
// ev), B/2 (63 - eb), |v|^2/4 (62 - 2 ev), |B|^2/4 (62 - 2 eb), v.B/2 (61 - ev
// - eb), and ln rho, ln e (60)
struct MENode {
  fx::i64 r, lr, e, le, pt, v[3], B[3], v2, b2, vb;
};
constexpr int kMESlots = 14;

struct MEPrim {
  double rho, e, p, v[3], B[3];
  unsigned E;  // high word of the total energy
};

__device__ __forceinline__ MEPrim me_prim(const double* c, double gm1, double gm1inv,
                                          unsigned& bad) {
  MEPrim q;
  const double rr = rcp(c[0]);
  double mv = 0.0;
  q.rho = c[0];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    q.v[k] = c[1 + k] * rr;
    q.B[k] = c[5 + k];
    mv = fma(c[1 + k], q.v[k], mv);
    mv = fma(q.B[k], q.B[k], mv);
  }
  q.p = gm1 * fma(-0.5, mv, c[4]);
  q.e = q.p * rr * gm1inv;
  q.E = (unsigned)__double2hiint(c[4]);
  Prim<double, 3> t;
  t.rho = q.rho;
  t.p = q.p;
  bad |= prim_check(t);
  return q;
}

// keys: rho max and min, e max and min, |v| max, p max, |B| max (then, not used
// here, |v| min, |B| min, total energy min)
__device__ __forceinline__ MEScale me_scale(const unsigned* key, const int* c, bool usable) {
  const unsigned rmax = key[0], rmin = key[1], emax = key[2], emin = key[3], vmax = key[4],
                 pmax = key[5], bmax = key[6];
  MEScale s;
  s.er = fx::exp_above(rmax);
  s.ev = fx::exp_above(vmax);
  s.eb = fx::exp_above(bmax);
  if (s.eb < -400) s.eb = -400;
  const int ee = fx::exp_above(emax);
  s.em = fx::exp_above(pmax) + (rmax - rmin < (1u << 20) ? c[0] : c[1]);
  if (s.em < 2 * s.eb + 4) s.em = 2 * s.eb + 4;
  const int floor_ev = (s.em - s.er - 60) >> 1;
  if (s.ev < floor_ev) s.ev = floor_ev;
  if (s.em < s.er + 2 * s.ev + 4) s.em = s.er + 2 * s.ev + 4;
  s.ee = ee + 1;
  if (s.ee < 2 * s.ev + 2) s.ee = 2 * s.ev + 2;
  if (s.ee < s.em - s.er) s.ee = s.em - s.er;
  const unsigned lo = (fx::kBias - 150u) << 20, hi = (fx::kBias + 150u) << 20;
  s.ok = usable && rmax < hi && rmin > lo && emax < hi && emin > lo && vmax < hi && pmax < hi &&
         bmax < hi && rmax - rmin < (6u << 20) && emax - emin < (6u << 20) &&
         (int)((emax - emin) >> 20) + s.ee - ee <= 8 && s.er + s.ee - s.em < 16;
  return s;
}

__device__ __forceinline__ MENode me_node(const MEPrim& q, const MEScale& s) {
  MENode n;
  n.r = fx::half_fixed(q.rho, s.er);
  n.lr = fx::ln_fixed(q.rho, s.er);
  n.e = fx::half_fixed(q.e, s.ee);
  n.le = fx::ln_fixed(q.e, s.ee);
  n.v2 = n.b2 = n.vb = 0;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    n.v[k] = fx::half_fixed(q.v[k], s.ev);
    n.B[k] = fx::half_fixed(q.B[k], s.eb);
    const fx::Limbs v = fx::limbs(n.v[k]), B = fx::limbs(n.B[k]);
    n.v2 = fx::fma64(v, v, n.v2);
    n.b2 = fx::fma64(B, B, n.b2);
    n.vb = fx::fma64(v, B, n.vb);
  }
  n.pt = fx::half_fixed(q.p, s.em) + shr(n.b2, s.em - 2 * s.eb - 1);
  return n;
}

// tanh(D/2) - D/2 from the short or general polynomials: c = tanh(D/2)/(D/2) - 1
// in 2^-63
__device__ __forceinline__ fx::i64 me_tanhc(fx::i64 D, bool is_short, fx::Limbs x) {
  if (is_short) return fx::tanh_short(x) >> 1;
  if (fx::d_mid((int)(D >> 32))) {
    const fx::i64 c[] = DG_FX_TanhMid;
    return fx::mul(x, fx::limbs(fx::mid_poly<fx::kTanhMidN>(x, c))) >> 1;
  }
  return fx::far_poly(D, fx::kTanhFar) << 2;
}

// The flux, normal component first: f[0] mass (62 - er - ev), f[1..3] momenta
// (63 - em), f[4] energy (61 - em - ev), f[5..7] induction (61 - ev - eb; zero
// in the normal component), f[8] {B_n} (62 - eb); all below 2^62.1.
__device__ __forceinline__ void me_flux(const MENode& a, const MENode& b, const MEScale& s,
                                        fx::i64* f) {
  using namespace fx;
  const i64 de = b.le - a.le;
  i64 rho, e;
  both_means(a.r + b.r, b.lr - a.lr, a.e + b.e, de, rho, e);
  const bool sh = d_short((int)(de >> 32));
  // {p_t} - [[p_t]]/2 tanh(D/2), D/2 = de in 2^-61
  const i64 th = de + (mul(limbs(de), limbs(me_tanhc(de, sh, square_of(de)))) << 1);  // 2^-61
  const i64 ph = a.pt + b.pt - (mul(limbs(b.pt - a.pt), limbs(th)) << 3);             // 63 - em
  Limbs v[3], B[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    v[k] = limbs(a.v[k] + b.v[k]);
    B[k] = limbs(a.B[k] + b.B[k]);
  }
  const i64 f0 = mul(limbs(rho), v[0]);
  f[0] = f0;
  const Limbs g = limbs(shr(f0, s.em - s.er - 2 * s.ev - 2));
  const int kb = s.em - 2 * s.eb;
  i64 en = 0;  // f_m . {v}, 62 - em - ev
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    f[1 + k] = mul(g, v[k]) - shr(mul(B[0], B[k]), kb - 1);
    if (k == 0) f[1] += ph;
    en = fma64(limbs(f[1 + k]), v[k], en);
    f[5 + k] = k == 0 ? 0 : (mul(v[0], B[k]) >> 1) - (mul(B[0], v[k]) >> 1);
  }
  const i64 eps = e - shr(a.v2 + b.v2, s.ee - 2 * s.ev - 1);  // 63 - ee
  i64 mag = fma64(limbs(f[6]), B[1], mul(limbs(f[7]), B[2]));  // 60 - ev - 2 eb
  mag = fma64(B[0], limbs(a.vb + b.vb), mag);
  mag -= mul(v[0], limbs(a.b2 + b.b2)) >> 1;
  f[4] = mul_up(limbs(f0), limbs(eps), s.er + s.ee - s.em) + (en >> 1) + shr(mag, kb - 1);
  f[8] = (a.B[0] + b.B[0]) >> 1;
}

// exponents of the sums of products with coefficients in 62 - ed (v: variable,
// 8: div B)
__device__ __forceinline__ int me_exponent(int v, const MEScale& s) {
  return v == 0 ? s.er + s.ev - 60
                : v <= 3 ? s.em - 61 : v == 4 ? s.em + s.ev - 59 : v < kMV ? s.ev + s.eb - 59
                                                                          : s.eb - 60;
}

constexpr int kMEKeys = 10;
__device__ __forceinline__ constexpr bool me_key_is_min(int j) {
  return j == 1 || j == 3 || j > 6;
}
__device__ __forceinline__ void me_keys(const MEPrim& q, unsigned* k) {
  auto hw = [](double x) { return (unsigned)__double2hiint(x); };
  k[0] = k[1] = hw(q.rho);
  k[2] = k[3] = hw(q.e);
  k[4] = k[6] = 0u;
  k[5] = hw(q.p);
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    k[4] = max(k[4], hw(q.v[j]) & 0x7fffffffu);
    k[6] = max(k[6], hw(q.B[j]) & 0x7fffffffu);
  }
  k[7] = k[4];
  k[8] = k[6];
  k[9] = q.E;
}

// the EC face flux (normal component first) from the conserved traces; false
// if the FP64 form is due
__device__ __forceinline__ bool mhd_ec_face_fixed(const double* cl, const double* cr, const Geom& g,
                                                  unsigned& bad, double* f) {
  const MEPrim L = me_prim(cl, g.gm1, g.gm1inv, bad), R = me_prim(cr, g.gm1, g.gm1inv, bad);
  unsigned kl[kMEKeys], kr[kMEKeys];
  me_keys(L, kl);
  me_keys(R, kr);
#pragma unroll
  for (int j = 0; j < 7; ++j) kl[j] = me_key_is_min(j) ? min(kl[j], kr[j]) : max(kl[j], kr[j]);
  int c[2];
  fx::scale_bits(g.gm1, c);
  const MEScale s = me_scale(kl, c, true);
  if (!s.ok) return false;
  fx::i64 x[kMQ];
  me_flux(me_node(L, s), me_node(R, s), s, x);
  const int ex[kMV] = {s.er + s.ev - 62, s.em - 63, s.em - 63, s.em - 63,
                       s.em + s.ev - 61, s.ev + s.eb - 61, s.ev + s.eb - 61, s.ev + s.eb - 61};
#pragma unroll
  for (int v = 0; v < kMV; ++v) f[v] = fx::to_double_int(x[v], ex[v]);
  return true;
}

template <int N>
struct MELaunch {
  using T = Tourney<N>;
  static constexpr int P = (N + 1) * (N + 1) * (N + 1), LINES = (N + 1) * (N + 1);
  static constexpr int ELEM = (kMESlots + kMQ) * P * 8;
  // a warp owns an element at N = 3, else the block its elements
  static constexpr bool WARP = LINES == T::LPW && P % 32 == 0;
  static constexpr int BY_THREADS = 8 * T::LPW / LINES > 0 ? 8 * T::LPW / LINES : 1;
  static constexpr int BY_SMEM = 98304 / ELEM > 0 ? 98304 / ELEM : 1;
  static constexpr int MOST = BY_THREADS < BY_SMEM ? BY_THREADS : BY_SMEM;
  // 3D N = 4: three elements fill 94% of their warps' lanes, four 89%
  static constexpr int EPB = N == 4 && MOST == 4 ? 3 : MOST < 16 ? MOST : 16;
  static constexpr int threads(int epb) { return 32 * ((epb * LINES + T::LPW - 1) / T::LPW); }
  // SPREAD (small meshes): one element per CTA with warps and sums of their own
  // for each direction
  static constexpr int ELEM_SPREAD = (kMESlots + 3 * kMQ) * P * 8;
};

// one pair of the element at elem: the flux and both nodes' sums
template <int N>
__device__ __forceinline__ void me_pair(unsigned char* elem, const MEScale& sc,
                                        const fx::Limbs (*ds)[kNPMax],
                                        const double (*ds64)[kNPMax], double hgm1inv, int dir,
                                        int l, int a, int b, int set) {
  constexpr int P = MELaunch<N>::P;
  const int t1 = dir == 2 ? 0 : dir + 1, t2 = t1 == 2 ? 0 : t1 + 1;
  const int X[3] = {dir, t1, t2};
  const int na = fx_place<3, N>(line_node_rt<3, N>(dir, l, a));
  const int nb = fx_place<3, N>(line_node_rt<3, N>(dir, l, b));
  const int comp[kMQ] = {0, 1 + dir, 1 + t1, 1 + t2, 4, 5 + dir, 5 + t1, 5 + t2, 8};
  fx::i64* sa = reinterpret_cast<fx::i64*>(elem) + (kMESlots + set * kMQ) * P;
  if (sc.ok) {
    const fx::i64* sx = reinterpret_cast<const fx::i64*>(elem);
    auto load = [&](int n) {
      MENode q;
      q.r = sx[n];
      q.lr = sx[P + n];
      q.e = sx[2 * P + n];
      q.le = sx[3 * P + n];
      q.pt = sx[4 * P + n];
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        q.v[k] = sx[(5 + X[k]) * P + n];
        q.B[k] = sx[(8 + X[k]) * P + n];
      }
      q.v2 = sx[11 * P + n];
      q.b2 = sx[12 * P + n];
      q.vb = sx[13 * P + n];
      return q;
    };
    fx::i64 f[kMQ];
    me_flux(load(na), load(nb), sc, f);
    const fx::Limbs dab = ds[a][b], dba = ds[b][a];
#pragma unroll
    for (int v = 0; v < kMQ; ++v) {
      if (v == 5) continue;  // the normal induction flux is zero
      const fx::Limbs fl = fx::limbs(f[v]);
      fx::i64* s = sa + comp[v] * P;
      s[na] = fx::fma64(dab, fl, s[na]);
      s[nb] = fx::fma64(dba, fl, s[nb]);
    }
  } else {
    const double* sp = reinterpret_cast<const double*>(elem);
    auto load = [&](int n) {
      ECq q;
      q.rho = sp[n];
      q.beta = sp[P + n];
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        q.hv[k] = sp[(2 + X[k]) * P + n];
        q.hB[k] = sp[(5 + X[k]) * P + n];
      }
      q.pm = sp[8 * P + n];
      q.qv2 = sp[9 * P + n];
      q.qB2 = sp[10 * P + n];
      q.hvB = sp[11 * P + n];
      return q;
    };
    const ECq qa = load(na), qb = load(nb);
    double f[kMQ];
    mhd_ec_flux<0>(qa, qb, hgm1inv, f);
    f[8] = qa.hB[0] + qb.hB[0];
    const double dab = ds64[a][b], dba = ds64[b][a];
#pragma unroll
    for (int v = 0; v < kMQ; ++v) {
      double* s = reinterpret_cast<double*>(sa) + comp[v] * P;
      s[na] = fma(dab, f[v], s[na]);
      s[nb] = fma(dba, f[v], s[nb]);
    }
  }
}

// the units by which a sum's truncated products fall short (fx_stage_node)
template <int N>
__device__ __forceinline__ constexpr int me_start(int v) {
  return v >= 5 && v < kMV ? 2 * N : 3 * N;
}

// stage a node's slots in its element's form and start its sums
template <int N, bool SPREAD>
__device__ __forceinline__ void me_stage(const MEPrim& q, const MEScale& sc, unsigned char* elem,
                                         int pl) {
  constexpr int P = MELaunch<N>::P;
  fx::i64* sx = reinterpret_cast<fx::i64*>(elem);
  if (sc.ok) {
    const MENode n = me_node(q, sc);
    sx[pl] = n.r;
    sx[P + pl] = n.lr;
    sx[2 * P + pl] = n.e;
    sx[3 * P + pl] = n.le;
    sx[4 * P + pl] = n.pt;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      sx[(5 + k) * P + pl] = n.v[k];
      sx[(8 + k) * P + pl] = n.B[k];
    }
    sx[11 * P + pl] = n.v2;
    sx[12 * P + pl] = n.b2;
    sx[13 * P + pl] = n.vb;
  } else {
    // as ec_of, from the primitives at hand
    const double beta = 0.5 * q.rho * rcp(q.p);
    double v2 = 0.0, b2 = 0.0, vb = 0.0;
    double* sp = reinterpret_cast<double*>(elem);
    sp[pl] = q.rho;
    sp[P + pl] = beta;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      v2 = fma(q.v[k], q.v[k], v2);
      b2 = fma(q.B[k], q.B[k], b2);
      vb = fma(q.v[k], q.B[k], vb);
      sp[(2 + k) * P + pl] = half(q.v[k]);
      sp[(5 + k) * P + pl] = half(q.B[k]);
    }
    sp[8 * P + pl] = 0.5 * fma(beta, b2, q.rho);
    sp[9 * P + pl] = 0.25 * v2;
    sp[10 * P + pl] = 0.25 * b2;
    sp[11 * P + pl] = half(vb);
  }
#pragma unroll
  for (int v = 0; v < kMQ; ++v) {
    sx[(kMESlots + v) * P + pl] = sc.ok ? me_start<N>(v) : 0;
    if (SPREAD) {
      sx[(kMESlots + kMQ + v) * P + pl] = 0;
      sx[(kMESlots + 2 * kMQ + v) * P + pl] = 0;
    }
  }
}

template <int N, int EPB, bool SPREAD>
__global__ void __launch_bounds__((SPREAD ? 3 : 1) * MELaunch<N>::threads(EPB),
                                  512 / ((SPREAD ? 3 : 1) * MELaunch<N>::threads(EPB)) < 1
                                      ? 1
                                      : 512 / ((SPREAD ? 3 : 1) * MELaunch<N>::threads(EPB)))
    mhd_volume_ec_fx_kernel(double* u, double* __restrict__ du, const double* __restrict__ fs,
                            Geom g, Tables<double> tbg, int powell, unsigned* __restrict__ err,
                            StageFuse fz) {
  using L = MELaunch<N>;
  using T = Tourney<N>;
  constexpr int NP = N + 1, P = L::P, LINES = L::LINES;
  constexpr int ELEM = SPREAD ? L::ELEM_SPREAD : L::ELEM;
  static_assert(!SPREAD || EPB == 1, "");
  extern __shared__ __align__(16) unsigned char dg_smem[];
  __shared__ Tables<double> tb;
  __shared__ fx::Limbs s_d[3][kNPMax][kNPMax];
  __shared__ MEScale s_scale[EPB];
  __shared__ unsigned s_key[EPB][kMEKeys];
  const int e0 = blockIdx.x * EPB;
  const int count = (int)g.nelem - e0 < EPB ? (int)g.nelem - e0 : EPB;
  const int t = threadIdx.x;
  if (t < count) {
#pragma unroll
    for (int j = 0; j < kMEKeys; ++j) s_key[t][j] = me_key_is_min(j) ? 0xffffffffu : 0u;
  }
  stage_tables<3, N, double>(tb, tbg, fz.k ? *fz.dt : 1.0);
  __syncthreads();
  const int ed = fx_table_exponent<3>(tb);
  for (int i = t; i < 3 * NP * NP; i += blockDim.x) {
    const int dir = i / (NP * NP), a = (i / NP) % NP, b = i % NP;
    s_d[dir][a][b] = fx::limbs(fx::half_fixed(tb.Ds[dir][a][b], ed));
  }
  const bool usable = ed <= 300 && ed >= -300;
  int cb[2];
  fx::scale_bits(g.gm1, cb);
  unsigned bad = 0;
  // keys of the elements' scales, over all nodes of the batch
  for (int t0 = t & ~31; t0 < count * P; t0 += blockDim.x) {
    const int i = t0 + (t & 31);
    const bool in = i < count * P;
    const int el = i / P, node = i % P;
    unsigned k[kMEKeys] = {};
    if (in) {
      double c[kMV];
#pragma unroll
      for (int v = 0; v < kMV; ++v) c[v] = u[((long long)(e0 + el) * kMV + v) * P + node];
      const MEPrim q = me_prim(c, g.gm1, g.gm1inv, bad);
      me_keys(q, k);
      double* sp = reinterpret_cast<double*>(dg_smem + el * ELEM) + fx_place<3, N>(node);
      sp[0] = q.rho;
      sp[P] = q.e;
      sp[2 * P] = q.p;
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        sp[(3 + j) * P] = q.v[j];
        sp[(6 + j) * P] = q.B[j];
      }
    }
    const int last = (t0 + 31 < count * P ? t0 + 31 : count * P - 1) / P;
    for (int ek = t0 / P; ek <= last; ++ek) {
      const bool mine = in && el == ek;
#pragma unroll
      for (int j = 0; j < kMEKeys; ++j) {
        if (me_key_is_min(j)) {
          const unsigned m = __reduce_min_sync(0xffffffffu, mine ? k[j] : 0xffffffffu);
          if ((t & 31) == 0) atomicMin(&s_key[ek][j], m);
        } else {
          const unsigned m = __reduce_max_sync(0xffffffffu, mine ? k[j] : 0u);
          if ((t & 31) == 0) atomicMax(&s_key[ek][j], m);
        }
      }
    }
  }
  if (bad) atomicOr(err, bad);
  __syncthreads();
  bool weak = false;
  if (t < count) {
    const unsigned* k = s_key[t];
    s_scale[t] = me_scale(k, cb, usable);
    if (energy_far(s_scale[t].em, k[9])) s_scale[t].ok = 0;
    weak = s_scale[t].ok && (k[4] - k[7]) + (k[6] - k[8]) > (kCrossBits << 20);
  }
  if (__syncthreads_or(weak)) {  // some node may lie too far below
    for (int i = t; i < count * P; i += blockDim.x) {
      const int el = i / P;
      const double* sp = reinterpret_cast<const double*>(dg_smem + el * ELEM);
      auto size = [&](int at, int n) {
        unsigned m = 0;
#pragma unroll
        for (int j = 0; j < 3; ++j)
          m = max(m, (unsigned)__double2hiint(sp[(at + j) * P + fx_place<3, N>(n)]) & 0x7fffffffu);
        return m;
      };
      const unsigned mv = s_key[el][4], mb = s_key[el][6];
      if ((mv - size(3, i % P)) + (mb - size(6, i % P)) <= (kCrossBits << 20)) continue;
      const unsigned cv = cross_max<3, N>(i % P, [&](int n) { return size(3, n); });
      const unsigned cb2 = cross_max<3, N>(i % P, [&](int n) { return size(6, n); });
      // the induction rows hold products of v and B
      if (cross_far(mv, cv) || (cv && cb2 && (mv - cv) + (mb - cb2) > (kCrossBits << 20)))
        s_scale[el].ok = 0;
    }
    __syncthreads();
  }
  for (int i = t; i < count * P; i += blockDim.x) {
    const int el = i / P, node = i % P, pl = fx_place<3, N>(node);
    const double* sp = reinterpret_cast<const double*>(dg_smem + el * ELEM) + pl;
    MEPrim q;
    q.rho = sp[0];
    q.e = sp[P];
    q.p = sp[2 * P];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      q.v[j] = sp[(3 + j) * P];
      q.B[j] = sp[(6 + j) * P];
    }
    me_stage<N, SPREAD>(q, s_scale[el], dg_smem + el * ELEM, pl);
  }
  __syncthreads();
  const int lane = t & 31, slot = lane / T::LPW;
  const int WPD = (int)blockDim.x / 96;  // warps per direction (SPREAD)
#pragma unroll 1
  for (int dir = SPREAD ? (t >> 5) / WPD : 0; dir < 3; dir += SPREAD ? 3 : 1) {
    for (int w = SPREAD ? (t >> 5) % WPD : t >> 5; w * T::LPW < count * LINES;
         w += SPREAD ? WPD : blockDim.x >> 5) {
      const int ln = w * T::LPW + lane % T::LPW;
      const bool in = slot < T::T && ln < count * LINES;
      const int el = ln / LINES, l = ln % LINES;
#pragma unroll 1
      for (int r = 0; r < T::ROUNDS; ++r) {
        if (in) {
          int a, b;
          tourney_pair<N>(r, slot, a, b);
          me_pair<N>(dg_smem + el * ELEM, s_scale[el], s_d[dir], tb.Ds[dir], 0.5 * g.gm1inv, dir,
                     l, a, b, SPREAD ? dir : 0);
        }
        __syncwarp();
      }
    }
    // at N = 3 each warp works on one element
    if (!SPREAD && !L::WARP) __syncthreads();
  }
  if (SPREAD || L::WARP) __syncthreads();
  const long long base = g.nelem * LINES;
  for (int i = t; i < count * P; i += blockDim.x) {
    const int el = i / P, node = i % P, e = e0 + el;
    const MEScale sc = s_scale[el];
    const fx::i64* sa =
        reinterpret_cast<const fx::i64*>(dg_smem + el * ELEM) + kMESlots * P + fx_place<3, N>(node);
    double val[kMQ];
#pragma unroll
    for (int v = 0; v < kMQ; ++v) {
      if (sc.ok) {
        fx::i64 a = sa[v * P];
        if (SPREAD) a += sa[(kMQ + v) * P] + sa[(2 * kMQ + v) * P];
        val[v] = a == me_start<N>(v) ? 0.0  // nothing but zeros
                                     : fx::to_double_int(a, ed + me_exponent(v, sc));
      } else {
        val[v] = __longlong_as_double(sa[v * P]);
        if (SPREAD)
          val[v] = (val[v] + __longlong_as_double(sa[(kMQ + v) * P])) +
                   __longlong_as_double(sa[(2 * kMQ + v) * P]);
      }
    }
#pragma unroll
    for (int dir = 0; dir < 3; ++dir) {
      int l, j;
      line_of<N>(dir, node, l, j);
      if (j == N || j == 0) {
        const long long ef = j == N ? e : neighbour32(g, e, dir, -1);
        const double lift = j == N ? tb.liftR[dir] : tb.liftL[dir];
        const double* src = fs + (long long)dir * kMQ * base + ef * LINES + l;
#pragma unroll
        for (int v = 0; v < kMQ; ++v) val[v] = fma(lift, src[v * base], val[v]);
      }
    }
    double c[kMV];
#pragma unroll
    for (int v = 0; v < kMV; ++v) c[v] = u[((long long)e * kMV + v) * P + node];
    if (powell) {
      const double rr = rcp(c[0]);
      double vb = 0.0;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const double v = c[1 + k] * rr;
        vb = fma(v, c[5 + k], vb);
        val[1 + k] = fma(c[5 + k], val[kMV], val[1 + k]);
        val[5 + k] = fma(v, val[kMV], val[5 + k]);
      }
      val[4] = fma(vb, val[kMV], val[4]);
    }
    double* const uo = fz.u_out ? fz.u_out : u;
#pragma unroll
    for (int v = 0; v < kMV; ++v) {
      const long long idx = ((long long)e * kMV + v) * P + node;
      if (fz.k) {
        double kk = val[v];
        if (fz.a != 0.0) kk = fma(fz.a, fz.k[idx], kk);
        fz.k[idx] = kk;
        uo[idx] = c[v] + fz.b * kk;
      } else {
        du[idx] = val[v];
      }
    }
  }
}
