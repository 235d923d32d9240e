// The volume term of the weak form (central volume flux) on FP64 meshes. The
// central two-point flux makes the split form a derivative of the nodal flux:
// with f_a the flux of node a along a line and F* the face fluxes,
//   du_a += sum_b Ds_ab (f_a + f_b)/2 + lifting
//         = sum_b M_ab f_b + lifting,
// M_ab = Ds_ab/2 off the diagonal and, since the rows of Dt sum to -(W^-1
// B)_aa, M_00 = -liftL/2 and M_NN = -liftR/2. So each node's flux is evaluated
// once per direction instead of once per pair, and what remains is the
// product with M, in 64-bit fixed point like the pair fluxes of dg_fixed.cuh
// (same rates, same per-element scales). Elements with non-finite values, with
// nodes whose energy lies far below the element's largest, or whose lines hold
// far smaller momenta or velocities than the element (cross_far, energy_far)
// take FP64.
//
// One thread per node, its primitives and sums in registers, the fluxes of one
// direction in shared memory. 32^3 N = 4: rhs 2.11 ms with a pair flux per pair
// in FP64, 0.92 ms here with the same (HLL) faces, 0.50 with faces on integers and
// the sums made doubles on the integer pipe (0.54 by FP64 additions: the FP64
// unit, 77% busy with prologue, lifting and stage update, bounds the kernel).
#pragma once

namespace dg {

template <int D, int N>
struct WeakLaunch {
  static constexpr int P = Shape<D, N>::P;
  static constexpr int EPB = 256 / P < 1 ? 1 : (256 / P > 32 ? 32 : 256 / P);
  static constexpr int THREADS = 32 * ((EPB * P + 31) / 32);
  static constexpr int SMEM = EPB * (D + 2) * P * 8;
};

// exponents of an element: |m_k| < 2^em, |v_k| < 2^ev, |E + p| < 2^eh, fluxes
// of momentum below 2^ef
struct WeakScale {
  int em, ev, eh, ef, k, ok;
};

template <int D, int N, int EPB>
__global__ void __launch_bounds__(WeakLaunch<D, N>::THREADS)
    volume_weak_kernel(double* u, double* __restrict__ du, const double* __restrict__ fs, Geom g,
                       Tables<double> tbg, unsigned* __restrict__ err, StageFuse fz) {
  constexpr int NP = N + 1, P = Shape<D, N>::P, NV = D + 2, LINES = Shape<D, N>::LINES;
  extern __shared__ __align__(16) unsigned char dg_smem[];
  __shared__ fx::Limbs s_m[D][NP][NP + 1];    // M, format 62 - ed
  __shared__ double s_m64[D][NP][NP + 1];
  __shared__ double s_lift[2][D];             // left, right
  __shared__ unsigned s_key[EPB][4];          // |m|, |v|, |E + p|, |p|
  __shared__ int s_far[EPB];
  __shared__ int s_left[EPB][D];
  fx::i64* sf = reinterpret_cast<fx::i64*>(dg_smem);  // [el][NV][P]
  const int e0 = blockIdx.x * EPB;
  const int count = (int)g.nelem - e0 < EPB ? (int)g.nelem - e0 : EPB;
  const double sc = fz.k ? *fz.dt : 1.0;
  const int t = threadIdx.x;
  const bool in = t < count * P;
  const int el = in ? t / P : 0, node = in ? t % P : 0, e = e0 + el;
  double c[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) c[v] = in ? u[((long long)e * NV + v) * P + node] : 1.0;
  // the largest coefficient is Ds[0][1]/2 (fx_table_exponent); with the
  // diagonal the absolute row sums stay below 8.2 times it: one bit more
  int ed;
  {
    unsigned m = 0;
#pragma unroll
    for (int k = 0; k < D; ++k) {
      const unsigned h = (unsigned)__double2hiint(0.5 * sc * tbg.Ds[k][0][1]) & 0x7fffffffu;
      m = h > m ? h : m;
    }
    ed = fx::exp_above(m) + 1;
  }
  for (int i = t; i < D * NP * NP; i += blockDim.x) {
    const int dir = i / (NP * NP), a = (i / NP) % NP, b = i % NP;
    double m = 0.5 * sc * tbg.Ds[dir][a][b];
    if (a == b) m = a == 0 ? -0.5 * sc * tbg.liftL[dir] : (a == N ? -0.5 * sc * tbg.liftR[dir] : 0.0);
    s_m64[dir][a][b] = m;
    s_m[dir][a][b] = fx::limbs(fx::half_fixed(m, ed));
  }
  if (t < D) {
    s_lift[0][t] = sc * tbg.liftL[t];
    s_lift[1][t] = sc * tbg.liftR[t];
  }
  if (t < count) {
#pragma unroll
    for (int k = 0; k < 4; ++k) s_key[t][k] = 0u;
    s_far[t] = 0;
    for (int k = 0; k < D; ++k) s_left[t][k] = neighbour32(g, e0 + t, k, -1);
  }
  __syncthreads();
  double rr;
  const Prim<double, D> q = prim_rcp<D>(c, g.gm1, rr);
  const double H = c[NV - 1] + q.p;
  unsigned km = 0, kv = 0;  // of the node
  {
    const unsigned bad = in ? prim_check(q) : 0u;
    if (bad) atomicOr(err, bad);
#pragma unroll
    for (int k = 0; k < D; ++k) {
      const unsigned hm = (unsigned)__double2hiint(c[1 + k]) & 0x7fffffffu;
      const unsigned hv = (unsigned)__double2hiint(q.v[k]) & 0x7fffffffu;
      km = hm > km ? hm : km;
      kv = hv > kv ? hv : kv;
    }
    const unsigned kh = (unsigned)__double2hiint(H) & 0x7fffffffu;
    const unsigned kp = (unsigned)__double2hiint(q.p) & 0x7fffffffu;
    const int first = (t & ~31) / P, lastt = (t | 31) < count * P ? (t | 31) : count * P - 1;
    for (int ek = first; ek <= lastt / P; ++ek) {
      const bool mine = in && el == ek;
      const unsigned a = __reduce_max_sync(0xffffffffu, mine ? km : 0u);
      const unsigned b = __reduce_max_sync(0xffffffffu, mine ? kv : 0u);
      const unsigned h = __reduce_max_sync(0xffffffffu, mine ? kh : 0u);
      const unsigned p = __reduce_max_sync(0xffffffffu, mine ? kp : 0u);
      if ((t & 31) == 0) {
        atomicMax(&s_key[ek][0], a);
        atomicMax(&s_key[ek][1], b);
        atomicMax(&s_key[ek][2], h);
        atomicMax(&s_key[ek][3], p);
      }
    }
  }
  __syncthreads();
  WeakScale w;
  bool low, weak;
  {
    const unsigned mm = s_key[el][0], mv = s_key[el][1], kh = s_key[el][2], kp = s_key[el][3];
    w.em = fx::exp_above(mm);
    w.ev = fx::exp_above(mv);
    w.eh = fx::exp_above(kh);
    w.ef = fx::exp_above(kp) + 1;
    if (w.em < -300) w.em = -300;  // nothing moves
    if (w.ev < -300) w.ev = -300;
    if (w.ef < w.em + w.ev + 1) w.ef = w.em + w.ev + 1;
    w.k = w.ef - w.em - w.ev < 63 ? w.ef - w.em - w.ev : 63;
    const unsigned hi = (fx::kBias + 150u) << 20, lo = (fx::kBias - 150u) << 20;
    w.ok = mm < hi && mv < hi && kh < hi && kp < hi && kh > lo && kp > lo && ed <= 300 &&
           ed >= -300;
    low = in && w.ok &&
          energy_far(w.ef > w.eh ? w.ef : w.eh, (unsigned)__double2hiint(c[NV - 1]));
    weak = in && w.ok && (mm - km > (kCrossBits << 20) || mv - kv > (kCrossBits << 20));
  }
  if (__syncthreads_or(low || weak)) {  // some node may lie too far below
    uint2* sk = reinterpret_cast<uint2*>(sf + el * NV * P);
    if (in) sk[node] = make_uint2(km, kv);
    __syncthreads();
    if (low ||
        (weak &&
         (cross_far(s_key[el][0], cross_max<D, N>(node, [&](int n) { return sk[n].x; })) ||
          cross_far(s_key[el][1], cross_max<D, N>(node, [&](int n) { return sk[n].y; })))))
      s_far[el] = 1;
    __syncthreads();
    if (s_far[el]) w.ok = 0;
  }
  // fixed point: m (63 - em), v (63 - ev), p (62 - ef), E + p (63 - eh)
  fx::i64 xm[D], xv[D], xp = 0, xh = 0, acc[NV];
  if (w.ok) {
#pragma unroll
    for (int k = 0; k < D; ++k) {
      xm[k] = fx::half_fixed(c[1 + k], w.em - 1);
      xv[k] = fx::half_fixed(q.v[k], w.ev - 1);
    }
    xp = fx::half_fixed(q.p, w.ef);
    xh = fx::half_fixed(H, w.eh - 1);
  } else {
#pragma unroll
    for (int k = 0; k < D; ++k) {
      xm[k] = __double_as_longlong(c[1 + k]);
      xv[k] = __double_as_longlong(q.v[k]);
    }
    xp = __double_as_longlong(q.p);
    xh = __double_as_longlong(H);
  }
#pragma unroll
  for (int v = 0; v < NV; ++v) acc[v] = w.ok ? D * NP : 0;  // truncation, see fma64
#pragma unroll
  for (int dir = 0; dir < D; ++dir) {
    int l, a;
    pp_line_of<D, N>(dir, node, l, a);
    if (in) {
      fx::i64* f = sf + el * NV * P + node;
      if (w.ok) {
        const fx::Limbs mn = fx::limbs(xm[dir]), vn = fx::limbs(xv[dir]);
        f[0] = xm[dir] >> 1;  // 62 - em
#pragma unroll
        for (int k = 0; k < D; ++k) {
          fx::i64 r = fx::mul(mn, fx::limbs(xv[k])) >> w.k;  // 62 - ef
          if (k == dir) r += xp;
          f[(1 + k) * P] = r;
        }
        f[(NV - 1) * P] = fx::mul(fx::limbs(xh), vn);  // 62 - eh - ev
      } else {
        const double mn = __longlong_as_double(xm[dir]);
        f[0] = xm[dir];
#pragma unroll
        for (int k = 0; k < D; ++k)
          f[(1 + k) * P] = __double_as_longlong(
              fma(mn, __longlong_as_double(xv[k]), k == dir ? __longlong_as_double(xp) : 0.0));
        f[(NV - 1) * P] = __double_as_longlong(__longlong_as_double(xh) *
                                               __longlong_as_double(xv[dir]));
      }
    }
    __syncthreads();
    if (in) {
      const int n0 = line_node_rt<D, N>(dir, l, 0);
      const int ns = dir == 0 ? 1 : (dir == 1 ? NP : NP * NP);
      const fx::i64* f = sf + el * NV * P + n0;
      if (w.ok) {
#pragma unroll
        for (int b = 0; b < NP; ++b) {
          const fx::Limbs m = s_m[dir][a][b];
#pragma unroll
          for (int v = 0; v < NV; ++v) acc[v] = fx::fma64(m, fx::limbs(f[v * P + b * ns]), acc[v]);
        }
      } else {
        for (int b = 0; b < NP; ++b) {
          const double m = s_m64[dir][a][b];
#pragma unroll
          for (int v = 0; v < NV; ++v)
            acc[v] = __double_as_longlong(
                fma(m, __longlong_as_double(f[v * P + b * ns]), __longlong_as_double(acc[v])));
        }
      }
    }
    if (dir + 1 < D) __syncthreads();
  }
  if (!in) return;
  double val[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v)
    val[v] = !w.ok ? __longlong_as_double(acc[v])
             : acc[v] == D * NP  // nothing but zeros
                 ? 0.0
                 : fx::to_double_int(acc[v],
                                     ed + (v == 0 ? w.em : v <= D ? w.ef : w.eh + w.ev) - 60);
  const long long base = g.nelem * LINES;
#pragma unroll
  for (int dir = 0; dir < D; ++dir) {
    int l, i;
    pp_line_of<D, N>(dir, node, l, i);
    if (i == 0 || i == N) {
      const double lift = s_lift[i == N][dir];
      const long long off = (long long)(i == N ? e : s_left[el][dir]) * LINES + l;
#pragma unroll
      for (int v = 0; v < NV; ++v)
        val[v] = fma(lift, fs[(long long)(dir * NV + v) * base + off], val[v]);
    }
  }
#pragma unroll
  for (int v = 0; v < NV; ++v)
    fx_store<D>(u, du, fz, ((long long)e * NV + v) * P + node, val[v]);
}

}  // namespace dg
