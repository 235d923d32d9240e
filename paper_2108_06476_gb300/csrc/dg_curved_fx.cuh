// The warped box with Ranocha's flux in 64-bit fixed point: the contravariant
// two-point flux of ranocha_contra on integers scaled by per-element powers of
// two (dg_fixed.cuh), the pairs of a line spread over (N + 1)/2 threads
// (dg_fixed_volume.cuh); in FP64 the volume kernel kept the FP64 unit 87%
// busy. Small meshes take one element per CTA with a set of warps and of sums
// for each direction (SPREAD). Volume kernel with the source, FP64 and here:
// 40^3 N = 3 2.78 and 0.92 ms, 14^3 N = 5 0.86 and 0.22 ms, 4^3 N = 7 146 and
// 42 us; EC faces at 40^3 N = 3 0.53 and 0.27 ms.
//
// Included by dg_curved.cuh.
#pragma once

namespace dg {

// the metric vectors: |J a^r_n| < 2^eg
struct CScale {
  fx::Scale u;
  int eg;
};
constexpr int kCSlots = 8 + 9;  // r, ln rho, e, ln e, p, v[3] and (J a^r)_n/2 by r, n

__device__ __forceinline__ CScale cfx_scale(const unsigned* key, const int* cb) {
  CScale s;
  s.u = fx::element_scale(key, cb);
  s.eg = fx::exp_above(key[8]);
  const unsigned lo = (fx::kBias - 150u) << 20, hi = (fx::kBias + 150u) << 20;
  if (!(key[8] < hi && key[8] > lo)) s.u.ok = 0;
  return s;
}

// The flux along the mean metric vector, from the halved metric vectors ga, gb
// (62 - eg): f[0] mass (60 - er - ev - eg), f[1..3] momenta (61 - em - eg),
// f[4] energy (60 - em - ev - eg); all below 2^62.
__device__ __forceinline__ void contra_flux_fx(const fx::Node<3>& a, const fx::Node<3>& b,
                                               const fx::i64* ga, const fx::i64* gb,
                                               const CScale& sc, fx::i64* f) {
  using namespace fx;
  const Scale& s = sc.u;
  i64 rho, ee;
  both_means(a.r + b.r, b.lr - a.lr, a.e + b.e, b.le - a.le, rho, ee);
  Limbs g[3];
  i64 va = 0, vb = 0, vv = 0;  // v_a.g/2, v_b.g/2 (61 - ev - eg); v_a.v_b/4
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    g[k] = limbs(ga[k] + gb[k]);
    const Limbs x = limbs(a.v[k]), y = limbs(b.v[k]);
    va = fma64(x, g[k], va);
    vb = fma64(y, g[k], vb);
    vv = fma64(x, y, vv);
  }
  ee += vv >> s.kv;
  const i64 f0 = mul(limbs(rho), limbs(va + vb));
  f[0] = f0;
  const Limbs h = limbs(f0 >> s.km), p = limbs(a.p + b.p);
#pragma unroll
  for (int k = 0; k < 3; ++k)
    f[1 + k] = fma64(h, limbs(a.v[k] + b.v[k]), mul(p, g[k]));
  const i64 pv = fma64(limbs(a.p), limbs(vb), mul(limbs(b.p), limbs(va)));
  f[4] = (pv + mul_up(limbs(f0), limbs(ee), s.s)) << 1;
}

template <int N>
struct CFxLaunch {
  using T = Tourney<N>;
  static constexpr int P = (N + 1) * (N + 1) * (N + 1), LINES = (N + 1) * (N + 1);
  static constexpr int ELEM = (kCSlots + 5) * P * 8, ELEM_SPREAD = (kCSlots + 15) * P * 8;
  static constexpr bool WARP = LINES == T::LPW && P % 32 == 0;
  static constexpr int BY_THREADS = 8 * T::LPW / LINES > 0 ? 8 * T::LPW / LINES : 1;
  static constexpr int BY_SMEM = 98304 / ELEM > 0 ? 98304 / ELEM : 1;
  static constexpr int MOST = BY_THREADS < BY_SMEM ? BY_THREADS : BY_SMEM;
  static constexpr int EPB = MOST < 16 ? MOST : 16;
  static constexpr int threads(int epb) { return 32 * ((epb * LINES + T::LPW - 1) / T::LPW); }
};

template <int N>
__device__ __forceinline__ void cfx_pair(unsigned char* elem, const CScale& sc,
                                         const fx::Limbs (*ds)[kNPMax],
                                         const double (*ds64)[kNPMax], int r, int l, int a, int b,
                                         int set) {
  constexpr int P = CFxLaunch<N>::P;
  const int na = fx_place<3, N>(line_node_rt<3, N>(r, l, a));
  const int nb = fx_place<3, N>(line_node_rt<3, N>(r, l, b));
  fx::i64* sa = reinterpret_cast<fx::i64*>(elem) + (kCSlots + 5 * set) * P;
  if (sc.u.ok) {
    const fx::i64* sx = reinterpret_cast<const fx::i64*>(elem);
    auto load = [&](int n, fx::i64* g) {
      fx::Node<3> q;
      q.r = sx[n];
      q.lr = sx[P + n];
      q.e = sx[2 * P + n];
      q.le = sx[3 * P + n];
      q.p = sx[4 * P + n];
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        q.v[k] = sx[(5 + k) * P + n];
        g[k] = sx[(8 + 3 * r + k) * P + n];
      }
      return q;
    };
    fx::i64 ga[3], gb[3], f[5];
    const fx::Node<3> qa = load(na, ga), qb = load(nb, gb);
    contra_flux_fx(qa, qb, ga, gb, sc, f);
    const fx::Limbs dab = ds[a][b], dba = ds[b][a];
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      const fx::Limbs fl = fx::limbs(f[v]);
      sa[v * P + na] = fx::fma64(dab, fl, sa[v * P + na]);
      sa[v * P + nb] = fx::fma64(dba, fl, sa[v * P + nb]);
    }
  } else {
    const double* sp = reinterpret_cast<const double*>(elem);
    auto load = [&](int n) {
      CPrim q;
      q.s0 = sp[n];
      q.s1 = sp[P + n];
      q.hp = sp[2 * P + n];
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        q.v[k] = sp[(3 + k) * P + n];
        q.hv[k] = half(q.v[k]);
      }
      return q;
    };
    double g[3], f[5];
#pragma unroll
    for (int k = 0; k < 3; ++k)
      g[k] = sp[(8 + 3 * r + k) * P + na] + sp[(8 + 3 * r + k) * P + nb];
    ranocha_contra(load(na), load(nb), g, f);
    const double dab = ds64[a][b], dba = ds64[b][a];
    double* s = reinterpret_cast<double*>(sa);
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      s[v * P + na] = fma(dab, f[v], s[v * P + na]);
      s[v * P + nb] = fma(dba, f[v], s[v * P + nb]);
    }
  }
}

template <int N, int EPB, bool SPREAD>
__global__ void __launch_bounds__((SPREAD ? 3 : 1) * CFxLaunch<N>::threads(EPB),
                                  640 / ((SPREAD ? 3 : 1) * CFxLaunch<N>::threads(EPB)) < 1
                                      ? 1
                                      : 640 / ((SPREAD ? 3 : 1) * CFxLaunch<N>::threads(EPB)))
    curved_volume_fx_kernel(double* u, double* __restrict__ du, const double* __restrict__ fs,
                            const double* __restrict__ Ja, const double* __restrict__ invJ,
                            const double* __restrict__ X, Geom g, CTables tb,
                            unsigned* __restrict__ err, StageFuse fz, SourceArgs src) {
  using L = CFxLaunch<N>;
  using T = Tourney<N>;
  constexpr int NP = N + 1, P = L::P, LINES = L::LINES, NV = 5;
  constexpr int ELEM = SPREAD ? L::ELEM_SPREAD : L::ELEM;
  static_assert(!SPREAD || EPB == 1, "");
  extern __shared__ __align__(16) unsigned char dg_smem[];
  __shared__ fx::Limbs s_d[kNPMax][kNPMax];
  __shared__ double s_d64[kNPMax][kNPMax];
  __shared__ CScale s_scale[EPB];
  __shared__ unsigned s_key[EPB][9];  // those of FxShared, then the metric vectors'
  const int e0 = blockIdx.x * EPB;
  const int count = (int)g.nelem - e0 < EPB ? (int)g.nelem - e0 : EPB;
  const int t = threadIdx.x;
  if (t < count) {
    fx_clear_key(s_key[t]);
    s_key[t][8] = 0u;
  }
  // |Dt[0][1]| is the largest coefficient (fx_table_exponent)
  const int ed = fx::exp_above((unsigned)__double2hiint(tb.Ds[0][1]) & 0x7fffffffu);
  for (int i = t; i < NP * NP; i += blockDim.x) {
    s_d64[i / NP][i % NP] = tb.Ds[i / NP][i % NP];
    s_d[i / NP][i % NP] = fx::limbs(fx::half_fixed(tb.Ds[i / NP][i % NP], ed));
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
    unsigned kg = 0;
    if (in) {
      const long long e = e0 + el;
      double c[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) c[v] = u[(e * NV + v) * P + node];
      const FxPrim<3> q = fx_prim<3>(c, g, bad);
      k = fx_keys<3>(q);
      double* sp = reinterpret_cast<double*>(dg_smem + el * ELEM) + fx_place<3, N>(node);
      sp[0] = q.rho;
      sp[P] = q.e;
      sp[2 * P] = q.p;
#pragma unroll
      for (int j = 0; j < 3; ++j) sp[(3 + j) * P] = q.v[j];
#pragma unroll
      for (int j = 0; j < 9; ++j) {
        const double m = Ja[(e * 9 + j) * P + node];
        sp[(8 + j) * P] = m;
        kg = max(kg, (unsigned)__double2hiint(m) & 0x7fffffffu);
      }
    }
    const int last = (t0 + 31 < count * P ? t0 + 31 : count * P - 1) / P;
    for (int ek = t0 / P; ek <= last; ++ek) {
      const bool mine = in && el == ek;
      fx_merge_keys(k, mine, s_key[ek]);
      const unsigned m = __reduce_max_sync(0xffffffffu, mine ? kg : 0u);
      if ((t & 31) == 0) atomicMax(&s_key[ek][8], m);
    }
  }
  if (bad) atomicOr(err, bad);
  __syncthreads();
  bool slow = false;
  if (t < count) {
    s_scale[t] = cfx_scale(s_key[t], cb);
    if (energy_far(s_scale[t].u.em, s_key[t][7])) s_scale[t].u.ok = 0;
    slow = fx_slow(s_key[t], s_scale[t].u);
  }
  if (__syncthreads_or(slow)) {
    fx_slow_elements<3, N>(count, dg_smem, ELEM, 3, s_key,
                           [&](int el) { s_scale[el].u.ok = 0; });
    __syncthreads();
  }
  for (int i = t; i < count * P; i += blockDim.x) {
    const int el = i / P, pl = fx_place<3, N>(i % P);
    const CScale sc = s_scale[el];
    unsigned char* elem = dg_smem + el * ELEM;
    double* sp = reinterpret_cast<double*>(elem) + pl;
    fx::i64* sx = reinterpret_cast<fx::i64*>(elem) + pl;
    FxPrim<3> q;
    q.rho = sp[0];
    q.e = sp[P];
    q.p = sp[2 * P];
#pragma unroll
    for (int j = 0; j < 3; ++j) q.v[j] = sp[(3 + j) * P];
    if (sc.u.ok) {
      sx[0] = fx::half_fixed(q.rho, sc.u.er);
      sx[P] = fx::ln_fixed(q.rho, sc.u.er);
      sx[2 * P] = fx::half_fixed(q.e, sc.u.ee);
      sx[3 * P] = fx::ln_fixed(q.e, sc.u.ee);
      sx[4 * P] = fx::half_fixed(q.p, sc.u.em);
#pragma unroll
      for (int j = 0; j < 3; ++j) sx[(5 + j) * P] = fx::half_fixed(q.v[j], sc.u.ev);
#pragma unroll
      for (int j = 0; j < 9; ++j) sx[(8 + j) * P] = fx::half_fixed(sp[(8 + j) * P], sc.eg) >> 1;
    } else {
      node_slots<kVRanocha, double>(q.rho, q.p, g.gm1, sp[0], sp[P]);
      sp[2 * P] = 0.5 * q.p;
#pragma unroll
      for (int j = 0; j < 9; ++j) sp[(8 + j) * P] *= 0.5;
    }
    // the units by which truncated products fall short (fx_stage_node)
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      sx[(kCSlots + v) * P] = sc.u.ok ? 3 * N : 0;
      if (SPREAD) sx[(kCSlots + 5 + v) * P] = sx[(kCSlots + 10 + v) * P] = 0;
    }
  }
  __syncthreads();
  const int lane = t & 31, slot = lane / T::LPW;
  const int wpd = (int)blockDim.x / 96;  // warps per direction (SPREAD)
#pragma unroll 1
  for (int r = SPREAD ? (t >> 5) / wpd : 0; r < 3; r += SPREAD ? 3 : 1) {
    for (int w = SPREAD ? (t >> 5) % wpd : t >> 5; w * T::LPW < count * LINES;
         w += SPREAD ? wpd : blockDim.x >> 5) {
      const int ln = w * T::LPW + lane % T::LPW;
      const bool in = slot < T::T && ln < count * LINES;
      const int el = ln / LINES, l = ln % LINES;
#pragma unroll 1
      for (int m = 0; m < T::ROUNDS; ++m) {
        if (in) {
          int a, b;
          tourney_pair<N>(m, slot, a, b);
          cfx_pair<N>(dg_smem + el * ELEM, s_scale[el], s_d, s_d64, r, l, a, b, SPREAD ? r : 0);
        }
        __syncwarp();
      }
    }
    if (!SPREAD && !L::WARP) __syncthreads();
  }
  if (SPREAD || L::WARP) __syncthreads();
  const double dtv = fz.k ? *fz.dt : 0.0;
  double* const uo = fz.u_out ? fz.u_out : u;
  const double ts = src.kind ? source_time(src) : 0.0;
  const long long base = g.nelem * LINES;
  for (int i = t; i < count * P; i += blockDim.x) {
    const int el = i / P, node = i % P, e = e0 + el;
    const CScale sc = s_scale[el];
    const fx::i64* sa =
        reinterpret_cast<const fx::i64*>(dg_smem + el * ELEM) + kCSlots * P + fx_place<3, N>(node);
    double val[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      if (sc.u.ok) {
        fx::i64 a = sa[v * P];
        if (SPREAD) a += sa[(5 + v) * P] + sa[(10 + v) * P];
        const int x = v == 0 ? sc.u.er + sc.u.ev - 58 : v < 4 ? sc.u.em - 59 : sc.u.em + sc.u.ev - 58;
        val[v] = a == 3 * N ? 0.0 : fx::to_double_int(a, ed + sc.eg + x);  // 3 N: only zeros
      } else {
        val[v] = __longlong_as_double(sa[v * P]);
        if (SPREAD)
          val[v] = (val[v] + __longlong_as_double(sa[(5 + v) * P])) +
                   __longlong_as_double(sa[(10 + v) * P]);
      }
    }
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      int l, j;
      line_of<N>(r, node, l, j);
      if (j == N || j == 0) {
        const long long ef = j == N ? e : neighbour32(g, e, r, -1);
        const double lift = j == N ? tb.liftR : tb.liftL;
        const double* s = fs + (long long)r * NV * base + ef * LINES + l;
#pragma unroll
        for (int v = 0; v < NV; ++v) val[v] = fma(lift, s[v * base], val[v]);
      }
    }
    const double ij = invJ[(long long)e * P + node];
    double S[NV] = {0.0, 0.0, 0.0, 0.0, 0.0};
    if (src.kind == kSourceManufactured)
      manufactured_source(X[((long long)e * 3 + 0) * P + node], X[((long long)e * 3 + 1) * P + node],
                          X[((long long)e * 3 + 2) * P + node], ts, g.gm1, S);
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const double d = fma(ij, val[v], S[v]);
      const long long idx = ((long long)e * NV + v) * P + node;
      if (fz.k) {
        double kk = dtv * d;
        if (fz.a != 0.0) kk = fma(fz.a, fz.k[idx], kk);
        fz.k[idx] = kk;
        uo[idx] = u[idx] + fz.b * kk;
      } else {
        du[idx] = d;
      }
    }
  }
}

// Ranocha's face flux along the metric vector g from the conserved traces;
// false if the FP64 form is due
__device__ __forceinline__ bool curved_face_fixed(const double* cl, const double* cr,
                                                  const double* gv, const Geom& g, double* f) {
  unsigned bad = 0;
  const FxPrim<3> L = fx_prim<3>(cl, g, bad), R = fx_prim<3>(cr, g, bad);
  const FxKeys a = fx_keys<3>(L), b = fx_keys<3>(R);
  unsigned key[9] = {max(a.r, b.r), min(a.r, b.r), max(a.e, b.e), min(a.e, b.e),
                     max(a.v, b.v), max(a.p, b.p), 0u, 0u, 0u};
#pragma unroll
  for (int k = 0; k < 3; ++k) key[8] = max(key[8], (unsigned)__double2hiint(gv[k]) & 0x7fffffffu);
  int cb[2];
  fx::scale_bits(g.gm1, cb);
  const CScale sc = cfx_scale(key, cb);
  if (!sc.u.ok) return false;
  auto node = [&](const FxPrim<3>& q) {
    fx::Node<3> n;
    n.r = fx::half_fixed(q.rho, sc.u.er);
    n.lr = fx::ln_fixed(q.rho, sc.u.er);
    n.e = fx::half_fixed(q.e, sc.u.ee);
    n.le = fx::ln_fixed(q.e, sc.u.ee);
    n.p = fx::half_fixed(q.p, sc.u.em);
#pragma unroll
    for (int k = 0; k < 3; ++k) n.v[k] = fx::half_fixed(q.v[k], sc.u.ev);
    return n;
  };
  fx::i64 hg[3], x[5];
#pragma unroll
  for (int k = 0; k < 3; ++k) hg[k] = fx::half_fixed(gv[k], sc.eg) >> 1;
  contra_flux_fx(node(L), node(R), hg, hg, sc, x);
#pragma unroll
  for (int v = 0; v < 5; ++v)
    f[v] = fx::to_double_int(x[v], sc.eg + (v == 0 ? sc.u.er + sc.u.ev - 60
                                            : v < 4 ? sc.u.em - 61 : sc.u.em + sc.u.ev - 60));
  return true;
}

}  // namespace dg
