// The weak-form MHD volume term in 64-bit fixed point (dg_fixed.cuh), one
// thread per node as mhd_volume_kernel did in FP64 (191 FP64 instructions per
// node, 64 cycles of the sub-partition's FP64 unit each). The primitives, the
// nodal fluxes, the product with the derivative rows and the lifting of the face
// values run on integers scaled by per-element powers of two; the reciprocal of
// the density, the Powell term and the stage update stay in FP64, so that both
// pipes are busy. The lifting's - lift f(u_i) at the line ends is part of the
// diagonal (M_00 = -liftL/2, M_NN = -liftR/2, the rows of the derivative matrix
// summing to zero), and + lift F* is added before the sum is rounded to FP64:
// the two cancel (added afterwards in FP64, the error of smooth data was up to
// 2.2 times that of lift (F* - f(u_i)), at a supersonic outflow 25 times). A
// face value beyond the element's units (a strong jump's dissipation) is added
// in FP64, which costs a tenth of the rhs where most are. The same steps run in
// FP64 in elements with non-finite values, non-positive densities or densities
// spread over more than 2^6, and with nodes whose energy lies far below the
// element's units or whose lines hold far smaller momenta, velocities or fields
// than the element (energy_far, cross_far).
//
// Included by dg_mhd.cu. 48^3 N = 3, rhs only: 2.68 ms in FP64, 1.11 here (0.98
// with the lifting in FP64); HLL faces 1.81 and 0.61 ms, LLF 1.55 and 0.55.
#pragma once

// |m_k| < 2^em, |v_k| < 2^ev, |B_k| < 2^eb, energies below 2^(ee - 1), 1/rho < 2^e1
struct MWScale {
  int em, ev, eb, ee, e1;
  int ok;
};

// fixed-point values of a node: m (63 - em), v (62 - ev), B (62 - eb),
// H = E + p_t and p_t (62 - ee), v.B (60 - ev - eb)
struct MWNode {
  fx::i64 m[3], v[3], B[3], H, pt, vb;
  fx::i64 p, hb2;  // p and |B|^2/2 (62 - ee)
};

// from the high words of the largest and smallest density and the largest
// |m_k|, |B_k|, E and |v_k|. ee covers the energies, m.v/2 and |B|^2/2, so that
// E - m.v/2 - |B|^2/2 stays in range also where the pressure is negative.
__device__ __forceinline__ MWScale mw_scale(const unsigned* key, double gm1, bool usable) {
  MWScale w;
  const unsigned rmax = key[0], rmin = key[1], km = key[2], kb = key[3], ke = key[4], kv = key[5];
  const unsigned hi = (fx::kBias + 150u) << 20, lo = (fx::kBias - 150u) << 20;
  w.ok = usable && rmax < hi && rmin > lo && rmax - rmin < (6u << 20) && km < hi && kb < hi &&
         ke < hi && ke > lo && kv < hi;
  const int eg = fx::exp_above((unsigned)__double2hiint(gm1));
  w.em = fx::exp_above(km);
  w.eb = fx::exp_above(kb);
  if (w.em < -400) w.em = -400;
  if (w.eb < -400) w.eb = -400;
  w.e1 = 2 - fx::exp_above(rmin);  // rmin >= 2^(exp - 1) (1 - 2^-20)
  w.ev = fx::exp_above(kv);
  if (w.ev < -400) w.ev = -400;
  w.ee = fx::exp_above(ke);
  if (w.ee < w.em + w.ev) w.ee = w.em + w.ev;
  if (w.ee < 2 * w.eb + 1) w.ee = 2 * w.eb + 1;
  w.ee += 1 + (eg > 0 ? eg : 0);
  return w;
}

// The halves of a unit that a product with the coefficient k loses on average to
// truncation (fma64: one for each limb), and in the upper 16 bits those with a
// factor of 53 bits (momenta and B_n): its low 8 bits are zeros, so a high limb
// of 8 bits loses nothing (N = 1 and 2, where the rows are few-bit numbers).
__device__ __forceinline__ int mw_cut(fx::Limbs k) {
  return (k.h != 0) + (k.l != 0) + (((k.h & 0xffffff) != 0) + (k.l != 0)) * 65536;
}

// a sum's start from mw_cut over its products (v: variable, kMV: div B)
__device__ __forceinline__ int mw_start(int cut, int v) {
  return ((v == 0 || v == kMV ? cut >> 16 : cut & 0xffff) + 1) / 2;
}

__device__ __forceinline__ fx::i64 shr(fx::i64 a, int n) { return a >> (n < 63 ? n : 63); }

// (v: the velocities in FP64)
__device__ __forceinline__ MWNode mw_node(const double* c, const double* v, const MWScale& w,
                                          double gm1) {
  MWNode q;
  fx::i64 ke2 = 0, b2 = 0;
  q.vb = 0;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    q.m[k] = fx::half_fixed(c[1 + k], w.em - 1);
    q.B[k] = fx::half_fixed(c[5 + k], w.eb);
    const fx::Limbs m = fx::limbs(q.m[k]), B = fx::limbs(q.B[k]);
    q.v[k] = fx::half_fixed(v[k], w.ev);
    const fx::Limbs x = fx::limbs(q.v[k]);
    ke2 = fx::fma64(m, x, ke2);    // 61 - em - ev
    b2 = fx::fma64(B, B, b2);      // 60 - 2 eb
    q.vb = fx::fma64(x, B, q.vb);  // 60 - ev - eb
  }
  const fx::i64 E = fx::half_fixed(c[4], w.ee);
  const fx::i64 hb2 = shr(b2, w.ee - 2 * w.eb - 1);
  const int eg = fx::exp_above((unsigned)__double2hiint(gm1));
  const fx::i64 p = fx::mul(fx::limbs(E - shr(ke2, w.ee - w.em - w.ev) - hb2),
                            fx::limbs(fx::half_fixed(gm1, eg - 1)));  // 61 - ee - eg
  q.p = eg >= -1 ? p << (1 + eg) : shr(p, -1 - eg);
  q.hb2 = hb2;
  q.pt = q.p + hb2;
  q.H = E + q.pt;
  return q;
}

// the physical flux in direction dir: f0 mass (62 - em), momenta (61 - ee),
// energy (61 - ev - ee), induction (61 - ev - eb; zero in direction dir)
__device__ __forceinline__ void mw_flux(const MWNode& q, const MWScale& w, int dir, fx::i64* f) {
  const fx::Limbs mn = fx::limbs(q.m[dir]), vn = fx::limbs(q.v[dir]), bn = fx::limbs(q.B[dir]),
                  nbn = fx::limbs(-q.B[dir]);
  f[0] = q.m[dir] >> 1;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const fx::Limbs vk = fx::limbs(q.v[k]), bk = fx::limbs(q.B[k]);
    f[1 + k] = shr(fx::mul(mn, vk), w.ee - w.em - w.ev) - shr(fx::mul(bn, bk), w.ee - 2 * w.eb - 1);
    if (k == dir) f[1 + k] += q.pt >> 1;
    f[5 + k] = k == dir ? 0 : fx::fma64(vn, bk, fx::mul(nbn, vk)) << 1;
  }
  f[4] = (fx::mul(vn, fx::limbs(q.H)) - shr(fx::mul(bn, fx::limbs(q.vb)), w.ee - 2 * w.eb - 2)) << 1;
}

// half the squared fast speed of the normal (first) direction times the
// density, and that over the density: c_f^2/2 in 61 - ee - e1. With a = gamma p,
// b_n and b_t the squares of the normal and transverse field, the discriminant
// (a + b_n + b_t)^2 - 4 a b_n is taken as (a - b_n)^2 + b_t (b_t + 2 (a + b_n)),
// whose terms do not cancel, and from operands shifted up to their leading bit:
// where kinetic energy makes up most of the units 2^ee, squares of unshifted
// ones would lose twice the bits (c_f off by 4e-9 at 100 times the sound
// speed).
__device__ __forceinline__ fx::i64 mw_fast2(const MWNode& q, const MWScale& w, fx::Limbs gamma,
                                            int egam, fx::Limbs r) {
  const fx::Limbs B0 = fx::limbs(q.B[0]), B1 = fx::limbs(q.B[1]), B2 = fx::limbs(q.B[2]);
  // quarters: gamma p (62 - ee; gamma > 1 in 62 - egam), the squares (62 - 2 eb)
  fx::i64 a = fx::mul(fx::limbs(q.p), gamma) << egam;
  fx::i64 bn = fx::mul(B0, B0), bt = fx::fma64(B1, B1, fx::mul(B2, B2));
  if (bn < 0) bn = 0;  // truncation (fma64)
  if (bt < 0) bt = 0;
  const int sh = w.ee - 2 * w.eb;  // >= 1
  // shifted up by n: a, b_n and b_t below 2^59 each, their sum below 2^61
  const int na = __clzll(a) - 5, nb = __clzll(bn + bt) - 5 + sh;
  const int n = na < nb ? (na > 0 ? na : 0) : (nb > 0 ? nb : 0);
  a <<= n;
  bn = n < sh ? shr(bn, sh - n) : bn << (n - sh);
  bt = n < sh ? shr(bt, sh - n) : bt << (n - sh);
  const fx::Limbs d = fx::limbs(a - bn), t = fx::limbs(bt);
  const fx::i64 disc = fx::fma64(t, fx::limbs(bt + 2 * (a + bn)), fx::sqr(d));
  const fx::i64 k = a + bn + bt + fx::sqrt_fixed(disc << 2);  // half of rho c_f^2, halved again
  return fx::mul(fx::limbs(k >> n), r);
}

// LLF or HLL from the conserved traces in normal-first order (rho, m, E, B),
// into f in the same order. Returns false (f not written) if the FP64 form is
// due.
__device__ __forceinline__ bool mhd_face_fixed(bool hll, const double* cl, const double* cr,
                                               double gamma, double gm1, double* f) {
  auto hw = [](double x) { return (unsigned)__double2hiint(x); };
  unsigned key[6] = {max(hw(cl[0]), hw(cr[0])), min(hw(cl[0]), hw(cr[0])), 0u, 0u,
                     max(hw(cl[4]), hw(cr[4])), 0u};
  const double il = rcp(cl[0]), ir = rcp(cr[0]);
  double vl[3], vr[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    vl[k] = cl[1 + k] * il;
    vr[k] = cr[1 + k] * ir;
    key[5] = max(key[5], max(hw(vl[k]) & 0x7fffffffu, hw(vr[k]) & 0x7fffffffu));
    key[2] = max(key[2], max(hw(cl[1 + k]) & 0x7fffffffu, hw(cr[1 + k]) & 0x7fffffffu));
    key[3] = max(key[3], max(hw(cl[5 + k]) & 0x7fffffffu, hw(cr[5 + k]) & 0x7fffffffu));
  }
  // energies more than 2^6 apart: the weaker trace would keep fewer bits than
  // FP64 has
  const unsigned kd = key[4] - min(hw(cl[4]), hw(cr[4]));
  const MWScale w = mw_scale(key, gm1, kd < (6u << 20));
  if (!w.ok) return false;
  const MWNode L = mw_node(cl, vl, w, gm1), R = mw_node(cr, vr, w, gm1);
  if (L.p <= 0 || R.p <= 0) return false;
  const int egam = fx::exp_above(hw(gamma));
  const fx::Limbs gam = fx::limbs(fx::half_fixed(gamma, egam));
  const fx::i64 xl = mw_fast2(L, w, gam, egam, fx::limbs(fx::half_fixed(il, w.e1 - 1)));
  const fx::i64 xr = mw_fast2(R, w, gam, egam, fx::limbs(fx::half_fixed(ir, w.e1 - 1)));
  // c_f = sqrt(x 2^(ee + e1 - 60)), the exponent made even
  int ec = w.ee + w.e1;
  const int odd = ec & 1;
  ec = (ec + odd) / 2;
  fx::i64 ca, cb;
  if (!hll) {
    ca = cb = fx::sqrt_fixed(((xl > xr ? xl : xr) >> odd) << 2);
  } else {
    ca = fx::sqrt_fixed((xl >> odd) << 2);
    cb = fx::sqrt_fixed((xr >> odd) << 2);
  }
  fx::FaceBlend blend;
  blend.speeds(hll, L.v[0], R.v[0], w.ev, ca, cb, ec);
  if (blend.side) {  // one trace's own flux, in FP64 whatever the other's size
    double c[kMV];
#pragma unroll
    for (int v = 0; v < kMV; ++v) c[v] = blend.side == 1 ? cl[v] : cr[v];
    unsigned dummy = 0;
    mhd_flux<0>(mhd_state(c, gm1, dummy), c, f);
    return true;
  }
  fx::i64 fl[kMV], fr[kMV];
  mw_flux(L, w, 0, fl);
  mw_flux(R, w, 0, fr);
  const int er = fx::exp_above(key[0]);
  f[0] = blend(fl[0], fr[0], w.em - 62, fx::full_fixed(cr[0], er) - fx::full_fixed(cl[0], er),
               er - 63);
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    f[1 + k] = blend(fl[1 + k], fr[1 + k], w.ee - 61, (R.m[k] >> 1) - (L.m[k] >> 1), w.em - 62);
    f[5 + k] = blend(fl[5 + k], fr[5 + k], w.ev + w.eb - 61, R.B[k] - L.B[k], w.eb - 62);
  }
  f[4] = blend(fl[4], fr[4], w.ev + w.ee - 61, (R.H - R.pt) - (L.H - L.pt), w.ee - 62);
  return true;
}

// shared slots of an element: its fluxes, then the lifting of its face nodes
template <int N>
struct MWElem {
  static constexpr int LINES = (N + 1) * (N + 1);
  static constexpr int SLOTS =
      kMV * LINES * (N + 1) > 6 * (kMV + 1) * LINES ? kMV * LINES * (N + 1) : 6 * (kMV + 1) * LINES;
};

template <int N, int EPB>
__global__ void __launch_bounds__(32 * ((EPB * (N + 1) * (N + 1) * (N + 1) + 31) / 32),
                                  (EPB * (N + 1) * (N + 1) * (N + 1) <= kMhdThreads) ? kMhdMinBlocks
                                                                                   : 1)
    mhd_volume_weak_kernel(double* u, double* __restrict__ du, const double* __restrict__ fs,
                           Geom g, Tables<double> tb, int powell, unsigned* __restrict__ err,
                           StageFuse fz) {
  constexpr int NP = N + 1, P = NP * NP * NP, LINES = NP * NP;
  extern __shared__ __align__(16) unsigned char dg_smem[];
  fx::i64* sf = reinterpret_cast<fx::i64*>(dg_smem);  // [el][8][P] (MWElem)
  __shared__ fx::Limbs s_m[3][NP][NP + 1];            // M, format 62 - ed
  __shared__ double s_m64[3][NP][NP + 1];
  __shared__ double s_lift[2][3];
  __shared__ fx::Limbs s_liftx[2][3];                 // 62 - ed
  __shared__ int s_cut[3][NP];  // mw_cut over a row and its lifting
  __shared__ unsigned s_key[EPB][6];                  // see mw_scale
  __shared__ int s_far[EPB];
  const int e0 = blockIdx.x * EPB;
  const int count = (int)g.nelem - e0 < EPB ? (int)g.nelem - e0 : EPB;
  const double sc = fz.k ? *fz.dt : 1.0;
  const int t = threadIdx.x;
  const bool in = t < count * P;
  const int el = in ? t / P : 0, node = in ? t % P : 0, e = e0 + el;
  double c[kMV];
#pragma unroll
  for (int v = 0; v < kMV; ++v)
    c[v] = in ? u[((long long)e * kMV + v) * P + node] : (v == 0 || v == 4 ? 1.0 : 0.0);
  // the largest coefficient is that of D_01, the lifting's at most twice it;
  // with the diagonal the absolute row sums stay below 8.2 times it, with the
  // lifting of three directions below 12.6 times (of the 16 that fit)
  unsigned mk = 0;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const unsigned h = (unsigned)__double2hiint(sc * tb.Ds[k][0][1]) & 0x7fffffffu;
    mk = h > mk ? h : mk;
  }
  const int ed = fx::exp_above(mk) + 1;
  for (int i = t; i < 3 * NP * NP; i += blockDim.x) {
    const int dir = i / (NP * NP), a = (i / NP) % NP, b = i % NP;
    double m = sc * tb.Ds[dir][a][b];
    if (a == b) m = a == 0 ? -0.5 * sc * tb.liftL[dir] : (a == N ? -0.5 * sc * tb.liftR[dir] : 0.0);
    s_m64[dir][a][b] = m;
    s_m[dir][a][b] = fx::limbs(fx::half_fixed(m, ed));  // the diagonal: below
  }
  if (t < 3) {
    s_lift[0][t] = sc * tb.liftL[t];
    s_lift[1][t] = sc * tb.liftR[t];
    s_liftx[0][t] = fx::limbs(fx::half_fixed(s_lift[0][t], ed));
    s_liftx[1][t] = fx::limbs(fx::half_fixed(s_lift[1][t], ed));
  }
  if (t < count) {
#pragma unroll
    for (int k = 0; k < 6; ++k) s_key[t][k] = k == 1 ? 0xffffffffu : 0u;
    s_far[t] = 0;
  }
  const double rr = rcp(c[0]);
  const double vel[3] = {c[1] * rr, c[2] * rr, c[3] * rr};
  __syncthreads();
  if (t < 3 * NP) {
    // the rows with their lifting sum to zero exactly (the coefficients'
    // roundings would leave 2^-53 of a constant flux or field)
    const int dir = t / NP, a = t % NP;
    fx::i64 x = 0;
    int cut = 0;
    auto take = [&](fx::Limbs k) {
      x -= (fx::i64)k.h * (1LL << 32) + k.l;
      cut += mw_cut(k);
    };
    for (int b = 0; b < NP; ++b)
      if (b != a) take(s_m[dir][a][b]);
    if (a == 0) take(s_liftx[0][dir]);
    if (a == N) take(s_liftx[1][dir]);
    s_m[dir][a][a] = fx::limbs(x);
    s_cut[dir][a] = cut + mw_cut(fx::limbs(x));
  }
  unsigned km = 0, kb = 0, kv = 0;  // of the node
  {
    auto hw = [](double x) { return (unsigned)__double2hiint(x); };
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      kv = max(kv, hw(vel[k]) & 0x7fffffffu);
      km = max(km, hw(c[1 + k]) & 0x7fffffffu);
      kb = max(kb, hw(c[5 + k]) & 0x7fffffffu);
    }
    const unsigned kr = hw(c[0]), ke = hw(c[4]);
    const int last = (t | 31) < count * P ? (t | 31) : count * P - 1;
    for (int ek = (t & ~31) / P; ek <= last / P; ++ek) {
      const bool mine = in && el == ek;
      const unsigned a = __reduce_max_sync(0xffffffffu, mine ? kr : 0u);
      const unsigned b = __reduce_min_sync(0xffffffffu, mine ? kr : 0xffffffffu);
      const unsigned m = __reduce_max_sync(0xffffffffu, mine ? km : 0u);
      const unsigned bb = __reduce_max_sync(0xffffffffu, mine ? kb : 0u);
      const unsigned ee = __reduce_max_sync(0xffffffffu, mine ? ke : 0u);
      const unsigned vv = __reduce_max_sync(0xffffffffu, mine ? kv : 0u);
      if ((t & 31) == 0) {
        atomicMax(&s_key[ek][0], a);
        atomicMin(&s_key[ek][1], b);
        atomicMax(&s_key[ek][2], m);
        atomicMax(&s_key[ek][3], bb);
        atomicMax(&s_key[ek][4], ee);
        atomicMax(&s_key[ek][5], vv);
      }
    }
  }
  __syncthreads();
  MWScale w = mw_scale(s_key[el], g.gm1, ed <= 300 && ed >= -300);
  {
    const unsigned mm = s_key[el][2], mb = s_key[el][3], mv = s_key[el][5];
    const bool low = in && w.ok && energy_far(w.ee, (unsigned)__double2hiint(c[4]));
    const bool weak = in && w.ok && (mm - km > (kCrossBits << 20) ||
                                     (mv - kv) + (mb - kb) > (kCrossBits << 20));
    if (__syncthreads_or(low || weak)) {  // some node may lie too far below
      uint3* sk = reinterpret_cast<uint3*>(sf + el * MWElem<N>::SLOTS);
      if (in) sk[node] = make_uint3(km, kv, kb);
      __syncthreads();
      bool far = low;
      if (weak) {
        const unsigned cm = cross_max<3, N>(node, [&](int n) { return sk[n].x; });
        const unsigned cv = cross_max<3, N>(node, [&](int n) { return sk[n].y; });
        const unsigned cb = cross_max<3, N>(node, [&](int n) { return sk[n].z; });
        // the induction rows hold products of v and B
        far = far || cross_far(mm, cm) || cross_far(mv, cv) || cross_far(mb, cb) ||
              (cv && cb && (mv - cv) + (mb - cb) > (kCrossBits << 20));
      }
      if (far) s_far[el] = 1;
      __syncthreads();
      if (s_far[el]) w.ok = 0;
    }
  }
  MWNode q;
  MState s;
  unsigned bad = 0;
  if (w.ok) {
    q = mw_node(c, vel, w, g.gm1);
    if (q.p <= 0) bad |= kErrP;
  } else {
    s = mhd_state(c, g.gm1, bad);
  }
  if (in && bad) atomicOr(err, bad);
  fx::i64 acc[kMV + 1];
  // truncation (fma64): the sums start from what their products lose on average
  int cut = 0;
#pragma unroll
  for (int dir = 0; dir < 3; ++dir) {
    int l, a;
    line_of<N>(dir, node, l, a);
    cut += s_cut[dir][a];
  }
#pragma unroll
  for (int v = 0; v <= kMV; ++v) {
    acc[v] = w.ok ? mw_start(cut, v) : 0;
  }
#pragma unroll
  for (int dir = 0; dir < 3; ++dir) {
    int l, a;
    line_of<N>(dir, node, l, a);
    if (in) {
      fx::i64* f = sf + el * MWElem<N>::SLOTS + node;
      if (w.ok) {
        fx::i64 d[kMV];
        mw_flux(q, w, dir, d);
        d[5 + dir] = q.B[dir];  // 62 - eb, the slot of B_n
#pragma unroll
        for (int v = 0; v < kMV; ++v) f[v * P] = d[v];
      } else {
        double d[kMV];
        if (dir == 0) mhd_flux<0>(s, c, d);
        else if (dir == 1) mhd_flux<1>(s, c, d);
        else mhd_flux<2>(s, c, d);
        d[5 + dir] = s.B[dir];
#pragma unroll
        for (int v = 0; v < kMV; ++v) f[v * P] = __double_as_longlong(d[v]);
      }
    }
    __syncthreads();
    if (in) {
      const int ns = dir == 0 ? 1 : (dir == 1 ? NP : LINES);
      const fx::i64* f = sf + el * MWElem<N>::SLOTS + line_node_rt<3, N>(dir, l, 0);
      if (w.ok) {
#pragma unroll
        for (int b = 0; b < NP; ++b) {
          const fx::Limbs m = s_m[dir][a][b];
#pragma unroll
          for (int v = 0; v < kMV; ++v) {
            const int to = v == 5 + dir ? kMV : v;
            acc[to] = fx::fma64(m, fx::limbs(f[v * P + b * ns]), acc[to]);
          }
        }
      } else {
        for (int b = 0; b < NP; ++b) {
          const double m = s_m64[dir][a][b];
#pragma unroll
          for (int v = 0; v < kMV; ++v) {
            const int to = v == 5 + dir ? kMV : v;
            acc[to] = __double_as_longlong(
                fma(m, __longlong_as_double(f[v * P + b * ns]), __longlong_as_double(acc[to])));
          }
        }
      }
    }
    if (dir < 2) __syncthreads();
  }
  // exponents of the fluxes' units: below 2^62 for values below 2^x
  auto unit = [&](int v) {
    return v == 0 ? w.em : v <= 3 ? w.ee + 1 : v == 4 ? w.ev + w.ee + 1
                                     : v < kMV ? w.ev + w.eb + 1 : w.eb;
  };
  const long long base = g.nelem * LINES;
  auto face = [&](int dir, int i, int l) {
    const long long ef = i == N ? e : neighbour32(g, e, dir, -1);
    return fs + (long long)dir * kMQ * base + ef * LINES + l;
  };
  // lift F*: a thread takes every P-th of its element's face nodes; the products
  // go to shared memory by variable. (By nodes, nearly every warp ran all three
  // directions for a part of its lanes: 64^3 N = 3 2.75 ms, now 2.62; 16^3 N = 5
  // with faces 0.29 and 0.23)
  constexpr int FACES = 6 * LINES;
  constexpr fx::i64 kTooLarge = (fx::i64)(1ULL << 63);
  fx::i64* sl = sf + el * MWElem<N>::SLOTS;
  __syncthreads();
  if (in && w.ok) {
#pragma unroll 1
    for (int m = node; m < FACES; m += P) {
      const int dir = m / (2 * LINES), right = m / LINES % 2, l = m % LINES;
      const double* src = face(dir, right ? N : 0, l);
      const fx::Limbs lift = s_liftx[right][dir];
#pragma unroll
      for (int v = 0; v <= kMV; ++v) {
        const double f = src[v * base];
        const unsigned most = (unsigned)(unit(v) + (int)fx::kBias) << 20;
        sl[v * FACES + m] = ((unsigned)__double2hiint(f) & 0x7fffffffu) < most
                                ? fx::mul(lift, fx::limbs(fx::half_fixed(f, unit(v))))
                                : kTooLarge;
      }
    }
  }
  __syncthreads();
  if (!in) return;
  // face values that are added in FP64: bit 9 dir + variable
  static_assert(kMV + 1 == 9, "");
  unsigned late = w.ok ? 0u : 0x7ffffffu;
  if (w.ok) {
#pragma unroll
    for (int dir = 0; dir < 3; ++dir) {
      int l, i;
      line_of<N>(dir, node, l, i);
      if (i == N || i == 0) {
        const fx::i64* x = sl + (2 * dir + (i == N)) * LINES + l;
#pragma unroll
        for (int v = 0; v <= kMV; ++v) {
          const fx::i64 p = x[v * FACES];
          if (p != kTooLarge) acc[v] += p;
          else late |= 1u << (9 * dir + v);
        }
      }
    }
  }
  double val[kMV + 1];
#pragma unroll
  for (int v = 0; v <= kMV; ++v)
    val[v] = !w.ok                       ? __longlong_as_double(acc[v])
             : acc[v] == mw_start(cut, v) ? 0.0  // nothing but zeros
                                          : fx::to_double_int(acc[v], ed + unit(v) - 60);
  for (int dir = 0; late && dir < 3; ++dir, late >>= 9) {
    int l, i;
    line_of<N>(dir, node, l, i);
    if ((late & 511u) && (i == N || i == 0)) {
      const double lift = s_lift[i == N][dir];
      const double* src = face(dir, i, l);
#pragma unroll
      for (int v = 0; v <= kMV; ++v)
        if (late >> v & 1u) val[v] = fma(lift, src[v * base], val[v]);
    }
  }
  if (powell) {
    // Phi = (0, B, v.B, v)
    double vb = 0.0;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      vb = fma(vel[k], c[5 + k], vb);
      val[1 + k] = fma(c[5 + k], val[kMV], val[1 + k]);
      val[5 + k] = fma(vel[k], val[kMV], val[5 + k]);
    }
    val[4] = fma(vb, val[kMV], val[4]);
  }
  double* const uo = fz.u_out ? fz.u_out : u;
#pragma unroll
  for (int v = 0; v < kMV; ++v) {
    const long long i = ((long long)e * kMV + v) * P + node;
    if (fz.k) {
      // the first stage (A = 0) neither reads k nor lets stale k values in
      double kk = val[v];
      if (fz.a != 0.0) kk = fma(fz.a, fz.k[i], kk);
      fz.k[i] = kk;
      uo[i] = c[v] + fz.b * kk;
    } else {
      du[i] = val[v];
    }
  }
}
