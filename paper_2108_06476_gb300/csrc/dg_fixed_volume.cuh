// Volume term with Ranocha's flux on FP64 meshes: the pair fluxes in fixed
// point (dg_fixed.cuh), or in FP64 for elements outside its limits.
//
// Layout of the work. Integer accumulation has no order, so a line's pairs
// can be spread over threads freely: the N + 1 nodes of a line play a
// round-robin tournament, T = (N + 1)/2 (rounded down) threads per line
// taking one disjoint pair each per round and adding D_ab f and D_ba f to the
// two nodes' sums in shared memory. One pair body serves every round, so the
// code is small and a thread needs few registers (one pair's values, no line
// of nodes and no accumulators), which leaves more warps per SM: with one
// thread per line (168 registers, 12 warps per SM) the integer pipes stood at
// 37% waiting for dependent results; this layout runs 24 warps per SM. Measured
// at 64^3 N = 3, a fused stage's volume kernel: FP64 8.47 ms, fixed point with
// one thread per line 3.87, this layout 2.49; rhs at 24^3 N = 7: 8.14 ms to
// 2.0. Meshes all of whose elements take the FP64 form, against the FP64 kernels
// with one thread per line: 32^3 N = 3 supersonic 1.42 and 1.50 ms, with a node
// 150 times denser in every element 1.71 and 2.32; 24^3 N = 4 1.60 and 1.72,
// 16^3 N = 7 3.00 and 3.14, 2D 256^2 N = 3 0.48 and 0.49; a stage of 18 members
// of degree 3 to 5 6.48 and 6.28 ms. About 40 FP64 instructions per node are left (prologue, lifting, stage
// update); the sums become doubles on the integer pipe (to_double's two
// additions per value cost the step 4%: 14.98 and 14.30 ms). The threads of a line share a warp
// (32/T lines per warp), so rounds are separated by a warp barrier. At N = 3
// in 3D a warp owns a whole element (16 lines x 2) and no block barrier runs
// at all.
//
// Included by dg_rhs_kernels.cuh after ranocha_nf and the node helpers.
#pragma once

namespace dg {

template <int N>
struct Tourney {
  static constexpr int NP = N + 1;
  static constexpr int T = NP / 2;                      // pairs per round
  static constexpr int ROUNDS = NP % 2 ? NP : NP - 1;
  static constexpr int LPW = 32 / T;                    // lines per warp
};

// the pair a < b of slot t in round r (circle method; an odd number of nodes
// leaves one node out of each round)
template <int N>
__device__ __forceinline__ void tourney_pair(int r, int t, int& a, int& b) {
  constexpr int NP = N + 1;
  int x, y;
  if (NP % 2 == 0) {
    constexpr int M = NP - 1 > 0 ? NP - 1 : 1;
    x = r + t >= M ? r + t - M : r + t;
    y = r - t < 0 ? r - t + M : r - t;
    if (t == 0) x = NP - 1;
  } else {
    x = r + t + 1 >= NP ? r + t + 1 - NP : r + t + 1;
    y = r - t - 1 < 0 ? r - t - 1 + NP : r - t - 1;
  }
  a = x < y ? x : y;
  b = x < y ? y : x;
}

// place of a node in an element's shared arrays: at N = 3 in 3D rotated so
// that the 16 lines of any direction hit 16 different 8-byte columns
template <int D, int N>
__device__ __forceinline__ int fx_place(int node) {
  if (D == 3 && N == 3) {
    const int i = node & 3, j = (node >> 2) & 3, k = node >> 4;
    return ((i + k) & 3) | (((j + k) & 3) << 2) | (k << 4);
  }
  return node;
}

// staged 8-byte slots of an element: fixed point r, ln rho, e, ln e, p, v[D];
// FP64 s0, s1, p/2, v[D]; then D + 2 accumulators
template <int D, int N>
struct FxShape {
  static constexpr int SLOTS = 5 + D;
  static constexpr int ELEM = (SLOTS + D + 2) * Shape<D, N>::P * 8;  // bytes
  // a warp owns an element
  static constexpr bool WARP =
      Shape<D, N>::LINES == Tourney<N>::LPW && Shape<D, N>::P % 32 == 0;
};

// shared memory of one batch besides the slots and accumulators
template <int D, int MAXE>
struct FxShared {
  fx::Limbs Ds[D][kNPMax][kNPMax];  // format 62 - ed
  fx::Scale scale[MAXE];
  unsigned key[MAXE][8];
  int left[MAXE][D];
  int ed, far;
};

template <int D, int N>
__device__ __forceinline__ fx::Node<D> fx_node(const fx::i64* sx, int dir, int t1, int t2,
                                               int nd) {
  constexpr int P = Shape<D, N>::P;
  fx::Node<D> q;
  q.r = sx[nd];
  q.lr = sx[P + nd];
  q.e = sx[2 * P + nd];
  q.le = sx[3 * P + nd];
  q.p = sx[4 * P + nd];
  q.v[0] = sx[(5 + dir) * P + nd];
  q.v[1] = sx[(5 + t1) * P + nd];
  if (D == 3) q.v[D - 1] = sx[(5 + t2) * P + nd];
  return q;
}

template <int D, int N>
__device__ __forceinline__ LinePrim<double, D> fp64_node(const double* sp, int dir, int t1, int t2,
                                                         int nd) {
  constexpr int P = Shape<D, N>::P;
  LinePrim<double, D> q;
  q.s0 = sp[nd];
  q.s1 = sp[P + nd];
  q.hp = sp[2 * P + nd];
  q.vn = sp[(3 + dir) * P + nd];
  q.hvn = half(q.vn);
  q.vt[0] = sp[(3 + t1) * P + nd];
  q.hvt[0] = half(q.vt[0]);
  if (D == 3) {
    q.vt[D - 2] = sp[(3 + t2) * P + nd];
    q.hvt[D - 2] = half(q.vt[D - 2]);
  }
  return q;
}

// one pair of an element: the flux and both nodes' sums
template <int D, int N>
__device__ __forceinline__ void fx_pair(unsigned char* elem, const fx::Scale& sc,
                                        const fx::Limbs (*ds)[kNPMax],
                                        const double (*ds64)[kNPMax], int dir, int l, int a,
                                        int b) {
  constexpr int P = Shape<D, N>::P, NV = D + 2, SL = FxShape<D, N>::SLOTS;
  const int t1 = dir + 1 == D ? 0 : dir + 1, t2 = D == 2 ? t1 : (t1 + 1 == D ? 0 : t1 + 1);
  const int na = fx_place<D, N>(line_node_rt<D, N>(dir, l, a));
  const int nb = fx_place<D, N>(line_node_rt<D, N>(dir, l, b));
  int comp[NV];  // variable of each normal-first component, times P
  comp[0] = 0;
  comp[1] = (1 + dir) * P;
  comp[2] = (1 + t1) * P;
  if (D == 3) comp[D] = (1 + t2) * P;
  comp[D + 1] = (D + 1) * P;
  if (sc.ok) {
    const fx::i64* sx = reinterpret_cast<const fx::i64*>(elem);
    fx::i64* sa = reinterpret_cast<fx::i64*>(elem) + SL * P;
    fx::i64 f[NV];
    fx::pair_flux<D>(fx_node<D, N>(sx, dir, t1, t2, na), fx_node<D, N>(sx, dir, t1, t2, nb), sc,
                     f);
    const fx::Limbs dab = ds[a][b], dba = ds[b][a];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const fx::Limbs fl = fx::limbs(f[v]);
      sa[comp[v] + na] = fx::fma64(dab, fl, sa[comp[v] + na]);
      sa[comp[v] + nb] = fx::fma64(dba, fl, sa[comp[v] + nb]);
    }
  } else {
    const double* sp = reinterpret_cast<const double*>(elem);
    double* sa = reinterpret_cast<double*>(elem) + SL * P;
    double f[NV], an;
    ranocha_nf<double, D>(fp64_node<D, N>(sp, dir, t1, t2, na),
                          fp64_node<D, N>(sp, dir, t1, t2, nb), f, an);
    const double dab = ds64[a][b], dba = ds64[b][a];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      sa[comp[v] + na] = fma(dab, f[v], sa[comp[v] + na]);
      sa[comp[v] + nb] = fma(dba, f[v], sa[comp[v] + nb]);
    }
  }
}

// the exponent of the coefficients' format: |Dt[0][1]| is the largest
// coefficient of every degree, and the absolute row sums over the three
// directions stay below 6 times it, so that a node's sum of products with
// fluxes below 2^62 (or 1.25 2^62, pair_flux) stays below 2^63
template <int D>
__device__ __forceinline__ int fx_table_exponent(const Tables<double>& tb) {
  unsigned m = 0;
#pragma unroll
  for (int k = 0; k < D; ++k) {
    const unsigned h = (unsigned)__double2hiint(tb.Ds[k][0][1]) & 0x7fffffffu;
    m = h > m ? h : m;
  }
  return fx::exp_above(m);
}

// primitives of a node and the keys of its element's scale
template <int D>
struct FxPrim {
  double rho, e, p, v[D];
  unsigned E;  // high word of the total energy
};
template <int D>
__device__ __forceinline__ FxPrim<D> fx_prim(const double* c, const Geom& g, unsigned& bad) {
  Prim<double, D> q;
  FxPrim<D> r;
  q.rho = r.rho = c[0];
  const double rr = rcp(c[0]);
  double mv = 0.0;
#pragma unroll
  for (int k = 0; k < D; ++k) {
    q.v[k] = r.v[k] = c[1 + k] * rr;
    mv = fma(c[1 + k], r.v[k], mv);
  }
  const double i = fma(-0.5, mv, c[D + 1]);  // rho e
  q.p = r.p = g.gm1 * i;
  r.e = i * rr;
  r.E = (unsigned)__double2hiint(c[D + 1]);
  bad |= prim_check(q);
  return r;
}

struct FxKeys {
  unsigned r, e, v, p, E;
};
template <int D>
__device__ __forceinline__ FxKeys fx_keys(const FxPrim<D>& q) {
  FxKeys k;
  k.r = (unsigned)__double2hiint(q.rho);
  k.e = (unsigned)__double2hiint(q.e);
  k.p = (unsigned)__double2hiint(q.p);
  k.E = q.E;
  k.v = 0;
#pragma unroll
  for (int j = 0; j < D; ++j) {
    const unsigned h = (unsigned)__double2hiint(q.v[j]) & 0x7fffffffu;
    k.v = h > k.v ? h : k.v;
  }
  return k;
}
// the keys of one element over the warp's lanes `mine`, by lane 0 into key
// (LEAST: the least velocity and energy too)
template <bool LEAST = true>
__device__ __forceinline__ void fx_merge_keys(const FxKeys& k, bool mine, unsigned* key) {
  const unsigned a = __reduce_max_sync(0xffffffffu, mine ? k.r : 0u);
  const unsigned b = __reduce_min_sync(0xffffffffu, mine ? k.r : 0xffffffffu);
  const unsigned c = __reduce_max_sync(0xffffffffu, mine ? k.e : 0u);
  const unsigned d = __reduce_min_sync(0xffffffffu, mine ? k.e : 0xffffffffu);
  const unsigned v = __reduce_max_sync(0xffffffffu, mine ? k.v : 0u);
  const unsigned p = __reduce_max_sync(0xffffffffu, mine ? k.p : 0u);
  unsigned lv, le;
  if (LEAST) {
    lv = __reduce_min_sync(0xffffffffu, mine ? k.v : 0xffffffffu);
    le = __reduce_min_sync(0xffffffffu, mine ? k.E : 0xffffffffu);
  }
  if ((threadIdx.x & 31) == 0) {
    atomicMax(&key[0], a);
    atomicMin(&key[1], b);
    atomicMax(&key[2], c);
    atomicMin(&key[3], d);
    atomicMax(&key[4], v);
    atomicMax(&key[5], p);
    if (LEAST) {
      atomicMin(&key[6], lv);
      atomicMin(&key[7], le);
    }
  }
}

// the staged slots of a node in its element's form, and its cleared sums
template <int D, int N>
__device__ __forceinline__ void fx_stage_node(const FxPrim<D>& q, const fx::Scale& sc, double gm1,
                                              unsigned char* elem, int pl) {
  constexpr int P = Shape<D, N>::P, NV = D + 2, SL = FxShape<D, N>::SLOTS;
  double* sp = reinterpret_cast<double*>(elem);
  fx::i64* sx = reinterpret_cast<fx::i64*>(elem);
  if (sc.ok) {
    sx[pl] = fx::half_fixed(q.rho, sc.er);
    sx[P + pl] = fx::ln_fixed(q.rho, sc.er);
    sx[2 * P + pl] = fx::half_fixed(q.e, sc.ee);
    sx[3 * P + pl] = fx::ln_fixed(q.e, sc.ee);
    sx[4 * P + pl] = fx::half_fixed(q.p, sc.em);
#pragma unroll
    for (int k = 0; k < D; ++k) sx[(5 + k) * P + pl] = fx::half_fixed(q.v[k], sc.ev);
  } else {
    node_slots<kVRanocha, double>(q.rho, q.p, gm1, sp[pl], sp[P + pl]);
    sp[2 * P + pl] = half(q.p);
#pragma unroll
    for (int k = 0; k < D; ++k) sp[(3 + k) * P + pl] = q.v[k];
  }
  // the sums start at +0.0, or at the D N units by which the truncated
  // products fall short on average
#pragma unroll
  for (int v = 0; v < NV; ++v) sx[(SL + v) * P + pl] = sc.ok ? D * N : 0;
}

// whether some node of the element is so slow that its lines have to be looked
// at (fx_slow_node)
__device__ __forceinline__ bool fx_slow(const unsigned* key, const fx::Scale& sc) {
  return sc.ok && key[4] - key[6] > (kCrossBits << 20);
}
// whether the velocities on the node's lines lie too far below the element's
// units; at(n): the key of node n's largest component
template <int D, int N, typename F>
__device__ __forceinline__ bool fx_slow_node(const unsigned* key, int node, const F& at) {
  return key[4] - at(node) > (kCrossBits << 20) && cross_far(key[4], cross_max<D, N>(node, at));
}

// clears the integer form (drop(el)) of elements with a node whose velocities
// lie too far below the units; v: FP64 slots `at` on of the elements at smem,
// `stride` bytes apart; by the whole block, between barriers
template <int D, int N, int K, typename F>
__device__ __forceinline__ void fx_slow_elements(int count, const unsigned char* smem, int stride,
                                                 int at, unsigned (*key)[K], const F& drop) {
  constexpr int P = Shape<D, N>::P;
  for (int t = threadIdx.x; t < count * P; t += blockDim.x) {
    const int el = t / P;
    const double* sv = reinterpret_cast<const double*>(smem + el * stride) + at * P;
    auto speed = [&](int n) {
      unsigned k = 0;
#pragma unroll
      for (int j = 0; j < D; ++j) {
        const unsigned h = (unsigned)__double2hiint(sv[j * P + fx_place<D, N>(n)]) & 0x7fffffffu;
        k = h > k ? h : k;
      }
      return k;
    };
    if (fx_slow_node<D, N>(key[el], t % P, speed)) drop(el);
  }
}

// primitives of the batch's nodes (rho, e, p, v in FP64 slots) and the keys of
// their elements' scales, by the whole block
template <int D, int N>
__device__ __forceinline__ unsigned fx_load(const double* __restrict__ u, const Geom& g, int e0,
                                            int count, unsigned char* smem,
                                            unsigned (*key)[8]) {
  constexpr int P = Shape<D, N>::P, NV = D + 2, ELEM = FxShape<D, N>::ELEM;
  unsigned bad = 0;
  for (int t0 = threadIdx.x & ~31; t0 < count * P; t0 += blockDim.x) {
    const int t = t0 + (threadIdx.x & 31);
    const bool in = t < count * P;
    const int el = t / P, node = t % P, pl = fx_place<D, N>(node);
    FxKeys k = {};
    if (in) {
      double c[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) c[v] = u[((long long)(e0 + el) * NV + v) * P + node];
      const FxPrim<D> q = fx_prim<D>(c, g, bad);
      k = fx_keys<D>(q);
      double* sp = reinterpret_cast<double*>(smem + el * ELEM);
      sp[pl] = q.rho;
      sp[P + pl] = q.e;
      sp[2 * P + pl] = q.p;
#pragma unroll
      for (int j = 0; j < D; ++j) sp[(3 + j) * P + pl] = q.v[j];
    }
    const int last = (t0 + 31 < count * P ? t0 + 31 : count * P - 1) / P;
    for (int ek = t0 / P; ek <= last; ++ek) fx_merge_keys(k, in && el == ek, key[ek]);
  }
  return bad;
}

__device__ __forceinline__ void fx_clear_key(unsigned* key) {
  key[0] = key[2] = key[4] = key[5] = 0u;
  key[1] = key[3] = key[6] = 0xffffffffu;
  key[7] = 0x7fefffffu;  // where it is not used it refuses nothing
}

__device__ __forceinline__ fx::Scale fx_scale(const unsigned* key, const int* c, int ed) {
  fx::Scale sc = fx::element_scale(key, c);
  if (ed > 300 || ed < -300 || energy_far(sc.em, key[7])) sc.ok = 0;
  return sc;
}
// the slots of each element's form, in place, by the whole block
template <int D, int N>
__device__ __forceinline__ void fx_stage(const Geom& g, int count, unsigned char* smem,
                                         const fx::Scale* scale) {
  constexpr int P = Shape<D, N>::P, ELEM = FxShape<D, N>::ELEM;
  for (int t = threadIdx.x; t < count * P; t += blockDim.x) {
    const int el = t / P, pl = t % P;
    const double* sp = reinterpret_cast<const double*>(smem + el * ELEM);
    FxPrim<D> q;
    q.rho = sp[pl];
    q.e = sp[P + pl];
    q.p = sp[2 * P + pl];
#pragma unroll
    for (int k = 0; k < D; ++k) q.v[k] = sp[(3 + k) * P + pl];
    fx_stage_node<D, N>(q, scale[el], g.gm1, smem + el * ELEM, pl);
  }
}

// a sum of variable v as a double (D N: nothing but zeros)
template <int D, int N>
__device__ __forceinline__ double fx_value(fx::i64 a, int v, const fx::Scale& sc, int ed) {
  if (!sc.ok) return __longlong_as_double(a);
  if (a == D * N) return 0.0;
  return fx::to_double_int(a, ed + (v == 0 ? sc.er + sc.ev - 60 : v <= D ? sc.em - 61
                                                                         : sc.em + sc.ev - 59));
}

// the sums of a node as doubles, with the lifting of the faces it lies on
template <int D, int N>
__device__ __forceinline__ void fx_result(const unsigned char* elem, const fx::Scale& sc, int ed,
                                          const Tables<double>& tb, const double* __restrict__ fs,
                                          int nelem, int e, const int* left, int node,
                                          double val[D + 2]) {
  constexpr int P = Shape<D, N>::P, NV = D + 2, SL = FxShape<D, N>::SLOTS,
                LINES = Shape<D, N>::LINES;
  const fx::i64* sa = reinterpret_cast<const fx::i64*>(elem) + SL * P + fx_place<D, N>(node);
#pragma unroll
  for (int v = 0; v < NV; ++v) val[v] = fx_value<D, N>(sa[v * P], v, sc, ed);
  const long long base = (long long)nelem * LINES;
#pragma unroll
  for (int dir = 0; dir < D; ++dir) {
    int l, i;
    pp_line_of<D, N>(dir, node, l, i);
    if (i == 0 || i == N) {
      const double lift = i == N ? tb.liftR[dir] : tb.liftL[dir];
      const long long off = (long long)(i == N ? e : left[dir]) * LINES + l;
#pragma unroll
      for (int v = 0; v < NV; ++v)
        val[v] = fma(lift, fs[(long long)(dir * NV + v) * base + off], val[v]);
    }
  }
}

template <int D>
__device__ __forceinline__ void fx_store(double* u, double* __restrict__ du, const StageFuse& fz,
                                         long long i, double val) {
  if (fz.k) {
    // the first stage (A = 0) neither reads k nor lets stale k values in
    double kk = val;
    if (fz.a != 0.0) kk = fma(fz.a, fz.k[i], kk);
    fz.k[i] = kk;
    (fz.u_out ? fz.u_out : u)[i] = u[i] + fz.b * kk;
  } else {
    du[i] = val;
  }
}

// One batch of `count` (<= MAXE) elements from e0; every thread of the block
// calls it (it starts with a block barrier). smem: count x ELEM bytes. In a
// fused stage (fz.k set) tb holds the coefficients times the stage's dt.
// BLOCK: the whole block works on the batch also where a warp could own an
// element.
template <int D, int N, int MAXE, bool BLOCK = false>
__device__ __forceinline__ void fx_batch(double* u, double* __restrict__ du,
                                         const double* __restrict__ fs, const Geom& g,
                                         const Tables<double>& tb, unsigned* __restrict__ err,
                                         const StageFuse& fz, int e0, int count,
                                         unsigned char* smem, FxShared<D, MAXE>& sh) {
  using S = Shape<D, N>;
  using T = Tourney<N>;
  constexpr int P = S::P, NV = S::NV, LINES = S::LINES, NP = S::NP;
  constexpr int ELEM = FxShape<D, N>::ELEM;
  const int nelem = (int)g.nelem;
  if ((int)threadIdx.x < count) {
    fx_clear_key(sh.key[threadIdx.x]);
    for (int k = 0; k < D; ++k)
      sh.left[threadIdx.x][k] = neighbour32(g, e0 + threadIdx.x, k, -1);
  }
  __syncthreads();  // tb is in place
  const int ed = fx_table_exponent<D>(tb);
  int cb[2];
  fx::scale_bits(g.gm1, cb);
  for (int i = threadIdx.x; i < D * NP * NP; i += blockDim.x) {
    const int dir = i / (NP * NP), a = (i / NP) % NP, b = i % NP;
    sh.Ds[dir][a][b] = fx::limbs(fx::half_fixed(tb.Ds[dir][a][b], ed));
  }
  __syncthreads();
  if constexpr (FxShape<D, N>::WARP && !BLOCK) {
    const int lane = threadIdx.x & 31;
    for (int el = threadIdx.x >> 5; el < count; el += blockDim.x >> 5) {
      unsigned char* elem = smem + el * ELEM;
      const int e = e0 + el;
      constexpr int NPL = P / 32;  // nodes per lane
      FxPrim<D> q[NPL];
      unsigned bad = 0;
#pragma unroll
      for (int j = 0; j < NPL; ++j) {
        double c[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) c[v] = u[((long long)e * NV + v) * P + lane + 32 * j];
        q[j] = fx_prim<D>(c, g, bad);
      }
      if (bad) atomicOr(err, bad);
#pragma unroll
      for (int j = 0; j < NPL; ++j) fx_merge_keys<false>(fx_keys<D>(q[j]), true, sh.key[el]);
      __syncwarp();
      fx::Scale sc = fx_scale(sh.key[el], cb, ed);
      // each node against the units by itself, in place of the least keys
      bool low = false, slow = false;
#pragma unroll
      for (int j = 0; j < NPL; ++j) {
        low = low || energy_far(sc.em, q[j].E);
        slow = slow || sh.key[el][4] - fx_keys<D>(q[j]).v > (kCrossBits << 20);
      }
      if (__any_sync(0xffffffffu, sc.ok && (low || slow))) {
        unsigned* sk = reinterpret_cast<unsigned*>(elem);
#pragma unroll
        for (int j = 0; j < NPL; ++j) sk[lane + 32 * j] = fx_keys<D>(q[j]).v;
        __syncwarp();
#pragma unroll 1
        for (int j = 0; j < NPL; ++j)
          low = low || fx_slow_node<D, N>(sh.key[el], lane + 32 * j, [&](int n) { return sk[n]; });
        if (__any_sync(0xffffffffu, low)) sc.ok = 0;
      }
#pragma unroll
      for (int j = 0; j < NPL; ++j)
        fx_stage_node<D, N>(q[j], sc, g.gm1, elem, fx_place<D, N>(lane + 32 * j));
      __syncwarp();
      const int l = lane % T::LPW, t = lane / T::LPW;
#pragma unroll 1
      for (int dir = 0; dir < D; ++dir) {
#pragma unroll 1
        for (int r = 0; r < T::ROUNDS; ++r) {
          int a, b;
          tourney_pair<N>(r, t, a, b);
          fx_pair<D, N>(elem, sc, sh.Ds[dir], tb.Ds[dir], dir, l, a, b);
          __syncwarp();
        }
      }
      __syncwarp();
#pragma unroll 1
      for (int j = 0; j < NPL; ++j) {
        // N = 3: the nodes of the two z faces first, then those that have no
        // face in z, so that the second pass skips that direction's lifting
        const int node = D == 3 && N == 3 ? (lane & 15) + 16 * (lane < 16 ? j : 3 - j)
                                          : lane + 32 * j;
        double val[NV];
        fx_result<D, N>(elem, sc, ed, tb, fs, nelem, e, sh.left[el], node, val);
#pragma unroll
        for (int v = 0; v < NV; ++v)
          fx_store<D>(u, du, fz, ((long long)e * NV + v) * P + node, val[v]);
      }
    }
  } else {
    const unsigned bad = fx_load<D, N>(u, g, e0, count, smem, sh.key);
    if (bad) atomicOr(err, bad);
    __syncthreads();
    bool slow = false;
    if ((int)threadIdx.x < count) {
      sh.scale[threadIdx.x] = fx_scale(sh.key[threadIdx.x], cb, ed);
      slow = fx_slow(sh.key[threadIdx.x], sh.scale[threadIdx.x]);
    }
    if (__syncthreads_or(slow)) {
      fx_slow_elements<D, N>(count, smem, FxShape<D, N>::ELEM, 3, sh.key,
                             [&](int el) { sh.scale[el].ok = 0; });
      __syncthreads();
    }
    fx_stage<D, N>(g, count, smem, sh.scale);
    __syncthreads();
    const int lane = threadIdx.x & 31, t = lane / T::LPW;
#pragma unroll 1
    for (int dir = 0; dir < D; ++dir) {
      for (int w = threadIdx.x >> 5; w * T::LPW < count * LINES; w += blockDim.x >> 5) {
        const int ln = w * T::LPW + lane % T::LPW;
        const bool in = t < T::T && ln < count * LINES;
        const int el = ln / LINES, l = ln % LINES;
#pragma unroll 1
        for (int r = 0; r < T::ROUNDS; ++r) {
          if (in) {
            int a, b;
            tourney_pair<N>(r, t, a, b);
            fx_pair<D, N>(smem + el * ELEM, sh.scale[el], sh.Ds[dir], tb.Ds[dir], dir, l, a, b);
          }
          __syncwarp();
        }
      }
      __syncthreads();
    }
    for (int t2 = threadIdx.x; t2 < count * P; t2 += blockDim.x) {
      const int el = t2 / P, node = t2 % P, e = e0 + el;
      double val[NV];
      fx_result<D, N>(smem + el * ELEM, sh.scale[el], ed, tb, fs, nelem, e, sh.left[el], node,
                      val);
#pragma unroll
      for (int v = 0; v < NV; ++v)
        fx_store<D>(u, du, fz, ((long long)e * NV + v) * P + node, val[v]);
    }
  }
}

// CTA shape: elements per CTA and threads (whole warps, one pass over the
// lines where that is at most 256 threads)
template <int D, int N>
struct FxLaunch {
  static constexpr int LINES = Shape<D, N>::LINES;
  static constexpr int ELEM = FxShape<D, N>::ELEM;
  static constexpr int LPW = Tourney<N>::LPW;
  static constexpr int BY_THREADS = 8 * LPW / LINES > 0 ? 8 * LPW / LINES : 1;
  static constexpr int BY_SMEM = 65536 / ELEM > 0 ? 65536 / ELEM : 1;
  static constexpr int MOST = BY_THREADS < BY_SMEM ? BY_THREADS : BY_SMEM;
  static constexpr int EPB = MOST < 32 ? MOST : 32;
  static constexpr int threads(int epb) { return 32 * ((epb * LINES + LPW - 1) / LPW); }
};

template <int D, int N, int EPB>
__global__ void __launch_bounds__(FxLaunch<D, N>::threads(EPB), 768 / FxLaunch<D, N>::threads(EPB) > 0 ? 768 / FxLaunch<D, N>::threads(EPB) : 1)
    volume_fx_kernel(double* u, double* __restrict__ du, const double* __restrict__ fs, Geom g,
                     Tables<double> tb, unsigned* __restrict__ err, StageFuse fz) {
  extern __shared__ __align__(16) unsigned char dg_smem[];
  __shared__ Tables<double> s_tab;  // fx_batch's first barrier follows
  __shared__ FxShared<D, EPB> sh;
  stage_tables<D, N, double>(s_tab, tb, fz.k ? *fz.dt : 1.0);
  const int e0 = blockIdx.x * EPB;
  const int left = (int)g.nelem - e0;
  fx_batch<D, N, EPB>(u, du, fs, g, s_tab, err, fz, e0, left < EPB ? left : EPB, dg_smem,
                       sh);
}

// ---- tiny meshes: one thread per node pair ----
// The CTA's elements with a thread per (direction, line, pair), whose fluxes
// go to shared memory, then a thread per (variable, node) that sums its pairs
// (the fluxes of FP64-form elements in the order of the tournament's rounds),
// adds the lifting and stores. With FACES, warps of their own evaluate the
// elements' face fluxes beside the first phases, so that a whole rhs or stage
// is one launch. The results are bitwise those of fx_batch.
template <int D, int N, int EPB>
struct FxPairPar {
  static constexpr int P = Shape<D, N>::P, LINES = Shape<D, N>::LINES, NV = D + 2;
  static constexpr int NPAIRS = N * (N + 1) / 2;
  // directions per phase: all of them when an element's pair fluxes fit in 96 KB
  static constexpr int GROUP = D * LINES * NPAIRS * NV * 8 <= 98304 ? D : 1;
  static constexpr int WORK = GROUP * LINES * NPAIRS;
  static constexpr int THREADS = EPB * WORK < 512 ? ((EPB * WORK + 31) / 32) * 32 : 512;
  static constexpr int ELEM = FxShape<D, N>::ELEM + WORK * NV * 8;
  static constexpr int SMEM = EPB * ELEM;
  static constexpr int FITEMS = EPB * 2 * D * LINES;
  static constexpr int THREADS_F = THREADS + ((FITEMS + 31) / 32) * 32;
  static_assert(THREADS_F <= 1024, "face warps do not fit the CTA");
  static constexpr int SMEM_F = SMEM + EPB * 2 * D * NV * LINES * 8;
  static_assert(EPB * P <= THREADS, "a node per volume thread");
  // 32 warps per SM whatever the CTA's size: a mesh of a few hundred elements
  // then needs one wave of CTAs fewer than with the compiler's own choice of
  // up to 98 registers (8^3 N = 3: 35 us per rhs against 27)
  static constexpr int MIN_CTAS = 1024 / THREADS_F < 1 ? 1 : 1024 / THREADS_F;
};

// node i's partner in round r of the tournament; -1: none
template <int N>
__device__ __forceinline__ int tourney_partner(int r, int i) {
  constexpr int NP = N + 1, M = NP % 2 ? NP : (NP > 1 ? NP - 1 : 1);
  if (NP % 2 == 0 && i == NP - 1) return r;
  int j = 2 * r - i;
  if (j < 0) j += M;
  if (j >= M) j -= M;
  if (j != i) return j;
  return NP % 2 ? -1 : NP - 1;
}

template <int D, int N, bool FACES, int EPB>
__global__ void __launch_bounds__(FACES ? FxPairPar<D, N, EPB>::THREADS_F
                                        : FxPairPar<D, N, EPB>::THREADS,
                                  FxPairPar<D, N, EPB>::MIN_CTAS)
    volume_fx_pp_kernel(double* u, double* __restrict__ du, const double* __restrict__ fs, Geom g,
                        Tables<double> tbg, unsigned* __restrict__ err, StageFuse fz, int sfk) {
  using C = FxPairPar<D, N, EPB>;
  constexpr int NP = N + 1, P = C::P, NV = C::NV, LINES = C::LINES, NPAIRS = C::NPAIRS,
                GROUP = C::GROUP, WORK = C::WORK, SL = FxShape<D, N>::SLOTS;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ Tables<double> tb;
  __shared__ FxShared<D, EPB> sh;
  double* sfc = reinterpret_cast<double*>(smem + C::SMEM);  // [el][side][dir][c][l]
  const int e0 = blockIdx.x * EPB;
  const int count = (int)g.nelem - e0 < EPB ? (int)g.nelem - e0 : EPB;
  const int nelem = (int)g.nelem;
  const int wt = FACES ? C::THREADS : (int)blockDim.x;  // volume threads
  const bool vol = (int)threadIdx.x < wt;
  // the volume threads synchronise among themselves until the first sums
  auto vsync = [&]() {
    if (FACES) asm volatile("bar.sync 1, %0;" ::"r"(C::THREADS) : "memory");
    else __syncthreads();
  };
  if (FACES && !vol) {
    constexpr int PER = 2 * D * LINES;  // face nodes per element
    for (int t = (int)threadIdx.x - C::THREADS; t < count * PER;
         t += (int)blockDim.x - C::THREADS) {
      const int el = t / PER, r = t % PER;
      const int side = r / (D * LINES), dir = (r / LINES) % D, l = r % LINES;
      const int e = e0 + el;
      const int owner = side == 0 ? e : neighbour32(g, e, dir, -1);
      double f[NV];
      face_flux_nf_dir<D, N, double, D == 3>(dir, u, g, sfk, owner, l, f);
      double* dst = sfc + (el * PER * NV + (side * D + dir) * NV * LINES + l);
#pragma unroll
      for (int c = 0; c < NV; ++c) dst[c * LINES] = f[c];
    }
  } else {
    // one node per thread, its loads in flight while the tables are staged
    const int t = threadIdx.x;
    const bool in = t < count * P;
    const int el = in ? t / P : 0, node = in ? t % P : 0;
    double c[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) c[v] = in ? u[(long long)e0 * NV * P + (el * NV + v) * P + node] : 1.0;
    const double sc0 = fz.k ? *fz.dt : 1.0;
    unsigned m = 0;
#pragma unroll
    for (int k = 0; k < D; ++k) {
      const unsigned h = (unsigned)__double2hiint(sc0 * tbg.Ds[k][0][1]) & 0x7fffffffu;
      m = h > m ? h : m;
    }
    const int ed = fx::exp_above(m);
    for (int i = t; i < D * NP * NP; i += wt) {
      const int dir = i / (NP * NP), a = (i / NP) % NP, b = i % NP;
      const double ds = sc0 * tbg.Ds[dir][a][b];
      tb.Ds[dir][a][b] = ds;
      sh.Ds[dir][a][b] = fx::limbs(fx::half_fixed(ds, ed));
    }
    if (t < D) {
      tb.liftR[t] = sc0 * tbg.liftR[t];
      tb.liftL[t] = sc0 * tbg.liftL[t];
    }
    if (t < count) {
      fx_clear_key(sh.key[t]);
      for (int k = 0; k < D; ++k) sh.left[t][k] = neighbour32(g, e0 + t, k, -1);
    }
    if (t == 0) {
      sh.ed = ed;
      sh.far = 0;
    }
    int cb[2];
    fx::scale_bits(g.gm1, cb);
    FxPrim<D> q = {};
    if (in) {
      unsigned bad = 0;
      q = fx_prim<D>(c, g, bad);
      if (bad) atomicOr(err, bad);
    }
    vsync();
    const int first = (t & ~31) / P, lastt = (t | 31) < count * P ? (t | 31) : count * P - 1;
    const FxKeys kk = fx_keys<D>(q);
    for (int ek = first; ek <= lastt / P; ++ek)
      fx_merge_keys<false>(kk, in && el == ek, sh.key[ek]);
    vsync();
    if (in) {
      const fx::Scale sc = fx_scale(sh.key[el], cb, ed);
      if (node == 0) sh.scale[el] = sc;
      if (sc.ok && (energy_far(sc.em, q.E) || sh.key[el][4] - kk.v > (kCrossBits << 20)))
        sh.far = 1;
      fx_stage_node<D, N>(q, sc, g.gm1, smem + el * C::ELEM, fx_place<D, N>(node));
    }
    vsync();
    if (sh.far) {  // some node may lie too far below: staged again, maybe in FP64
      unsigned* sk = reinterpret_cast<unsigned*>(smem + el * C::ELEM);
      FxPrim<D> p = {};
      if (in) {
        double cc[NV];
        unsigned seen = 0;
#pragma unroll
        for (int v = 0; v < NV; ++v) cc[v] = u[(long long)e0 * NV * P + (el * NV + v) * P + node];
        p = fx_prim<D>(cc, g, seen);
        sk[node] = fx_keys<D>(p).v;
      }
      vsync();
      if (in && sh.scale[el].ok &&
          (energy_far(sh.scale[el].em, p.E) ||
           fx_slow_node<D, N>(sh.key[el], node, [&](int n) { return sk[n]; })))
        sh.scale[el].ok = 0;
      vsync();
      if (in)
        fx_stage_node<D, N>(p, sh.scale[el], g.gm1, smem + el * C::ELEM, fx_place<D, N>(node));
      vsync();
    }
  }
#pragma unroll 1
  for (int d0 = 0; d0 < D; d0 += GROUP) {
    for (int t = threadIdx.x; t < count * WORK && vol; t += wt) {
      const int el = t / WORK, w = t % WORK;
      unsigned char* elem = smem + el * C::ELEM;
      const int dir = d0 + w / (LINES * NPAIRS), rem = w % (LINES * NPAIRS), l = rem / NPAIRS;
      int a, b;
      pp_pair_of<N>(rem % NPAIRS, a, b);
      const int t1 = (dir + 1) % D, t2 = (dir + 2) % D;
      const int na = fx_place<D, N>(line_node_rt<D, N>(dir, l, a));
      const int nb = fx_place<D, N>(line_node_rt<D, N>(dir, l, b));
      fx::i64* sf = reinterpret_cast<fx::i64*>(elem + FxShape<D, N>::ELEM) + w * NV;
      if (sh.scale[el].ok) {
        const fx::i64* sx = reinterpret_cast<const fx::i64*>(elem);
        fx::i64 f[NV];
        fx::pair_flux<D>(fx_node<D, N>(sx, dir, t1, t2, na), fx_node<D, N>(sx, dir, t1, t2, nb),
                         sh.scale[el], f);
#pragma unroll
        for (int v = 0; v < NV; ++v) sf[v] = f[v];
      } else {
        const double* sp = reinterpret_cast<const double*>(elem);
        double f[NV], an;
        ranocha_nf<double, D>(fp64_node<D, N>(sp, dir, t1, t2, na),
                              fp64_node<D, N>(sp, dir, t1, t2, nb), f, an);
#pragma unroll
        for (int v = 0; v < NV; ++v) sf[v] = __double_as_longlong(f[v]);
      }
    }
    __syncthreads();
    for (int t = threadIdx.x; t < count * NV * P; t += blockDim.x) {
      const int el = t / (NV * P), v = (t / P) % NV, node = t % P, e = e0 + el;
      unsigned char* elem = smem + el * C::ELEM;
      const fx::Scale sc = sh.scale[el];
      const fx::i64* sf = reinterpret_cast<const fx::i64*>(elem + FxShape<D, N>::ELEM);
      fx::i64* sa = reinterpret_cast<fx::i64*>(elem) + (SL + v) * P + fx_place<D, N>(node);
      fx::i64 acc = *sa;
#pragma unroll 1
      for (int gd = 0; gd < GROUP; ++gd) {
        const int dir = d0 + gd, c = nf_component<D>(v, dir);
        int l, i;
        pp_line_of<D, N>(dir, node, l, i);
        const fx::i64* fl = sf + (gd * LINES + l) * NPAIRS * NV + c;
        if (sc.ok) {
#pragma unroll
          for (int r = 0; r < Tourney<N>::ROUNDS; ++r) {
            const int j = tourney_partner<N>(r, i);
            if (j >= 0)
              acc = fx::fma64(sh.Ds[dir][i][j],
                              fx::limbs(fl[pp_pair_index<N>(i < j ? i : j, i < j ? j : i) * NV]),
                              acc);
          }
        } else {
          double s = __longlong_as_double(acc);
          for (int r = 0; r < Tourney<N>::ROUNDS; ++r) {
            const int j = tourney_partner<N>(r, i);
            if (j >= 0)
              s = fma(tb.Ds[dir][i][j],
                      __longlong_as_double(
                          fl[pp_pair_index<N>(i < j ? i : j, i < j ? j : i) * NV]),
                      s);
          }
          acc = __double_as_longlong(s);
        }
      }
      if (d0 + GROUP < D) {
        *sa = acc;
        continue;
      }
      double val = fx_value<D, N>(acc, v, sc, sh.ed);
      const double* fce = sfc + el * 2 * D * LINES * NV;
#pragma unroll
      for (int dir = 0; dir < D; ++dir) {
        int l, i;
        pp_line_of<D, N>(dir, node, l, i);
        if (i == 0 || i == N) {
          const int c = nf_component<D>(v, dir);
          const double f =
              FACES ? fce[(((i == N ? 0 : D) + dir) * NV + c) * LINES + l]
                    : fs[(long long)(dir * NV + v) * nelem * LINES +
                         (long long)(i == N ? e : sh.left[el][dir]) * LINES + l];
          val = fma(i == N ? tb.liftR[dir] : tb.liftL[dir], f, val);
        }
      }
      fx_store<D>(u, du, fz, (long long)e0 * NV * P + t, val);
    }
    if (d0 + GROUP < D) __syncthreads();
  }
}

}  // namespace dg
