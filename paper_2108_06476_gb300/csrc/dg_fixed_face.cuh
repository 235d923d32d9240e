// The local Lax-Friedrichs and HLL face fluxes of FP64 Cartesian meshes on
// 64-bit integers (dg_fixed.cuh), one thread per face node.
//
// In FP64 a face node costs about 58 instructions (LLF), 64 cycles each of the
// SM sub-partition's FP64 unit. Both fluxes are sums of products of the two
// traces once 1/rho and the sound speeds are known: the reciprocals and the
// square roots stay in FP64 (15 instructions for LLF), the rest runs on
// integers with power-of-two exponents chosen per face node from its two
// traces, 61 to 63 bits below the larger one. Faces whose densities or energies
// differ by more than 2^6, or with non-finite or non-positive values, take the
// FP64 form (surface_nf): beyond that the weaker trace would keep fewer bits
// than FP64 has. Where HLL takes one trace's own flux, that is evaluated in
// FP64 from this trace, whatever the other one's size. Measured at 64^3 N = 3
// (12.6 M face nodes, LLF): 1.38 ms in FP64, 0.66 ms here (80 registers, 24
// warps per SM; 96 registers were an eighth slower).
#pragma once
#include "dg_fixed.cuh"

namespace dg {
namespace fx {

// x in format 63 - E (|x| < 2^E (1 - 2^-21))
__device__ __forceinline__ i64 full_fixed(double x, int E) { return half_fixed(x, E - 1); }

// d shifted up until its leading bit is at 61 or 60; n the shift
__device__ __forceinline__ i64 normalised(i64 d, int& n) {
  n = __clzll(d < 0 ? ~d : d) - 2;
  if (n < 0) n = 0;
  if (n > 60) n = 60;
  return d << n;
}

// sqrt(x 2^-62) in 2^-62 for 0 <= x < 2^62, within a few units of the shifted
// argument's 2^-60: a 23-bit reciprocal square root, then g += (x - g^2) r/2
// twice (each squares the relative error down to the residual's rounding)
__device__ __forceinline__ i64 sqrt_fixed(i64 x) {
  if (x <= 0) return 0;
  const int n = (__clzll(x) - 2) & ~1;
  const i64 xs = x << n;  // in [2^60, 2^62)
  const float f = __int2float_rn((int)(xs >> 32)) * 0x1p-30f;
  const Limbs r = limbs((i64)__float2int_rn(rsqrtf(f) * 0x1p29f) << 32);  // 61
  i64 g = mul(limbs(xs), r) << 3;                                         // 62
  i64 d = (xs >> 2) - sqr(limbs(g));                                      // 60, below 2^40
  g += mul(limbs(d << 20), r) >> 16;
  d = (xs >> 2) - sqr(limbs(g));                                          // below 2^20
  g += mul(limbs(d << 40), r) >> 36;
  return g >> (n / 2);
}

__device__ __forceinline__ i64 abs64(i64 a) { return a < 0 ? -a : a; }

// f = fr + w (fl - fr) + kappa (qR - qL) of the two traces, for LLF (w = 1/2,
// kappa = -lambda/2) and HLL (w = sR/(sR - sL), kappa = w sL)
struct FaceBlend {
  bool hll;
  int side;      // HLL: 1 or 2 where the flux is the left or the right one
  Limbs kap, w;  // kappa (62 - eL + kx), w (62)
  int eL, kx;

  // from the normal velocities (62 - ev) and sound speeds (62 - ec; LLF: the
  // larger one in both)
  __device__ __forceinline__ void speeds(bool is_hll, i64 vl, i64 vr, int ev, i64 cl, i64 cr,
                                         int ec) {
    hll = is_hll;
    side = 0;
    eL = (ev > ec ? ev : ec) + 1;
    const int dv = eL - ev < 63 ? eL - ev : 63, dc = eL - ec < 63 ? eL - ec : 63;
    vl >>= dv;
    vr >>= dv;
    cl >>= dc;
    cr >>= dc;
    i64 k, x = 0;
    kx = 0;
    if (!hll) {
      const i64 a = abs64(vl), b = abs64(vr);
      k = -((a > b ? a : b) + cl);  // -lambda
      kx = 1;                       // halved
    } else {
      const i64 sL = vl - cl < vr - cr ? vl - cl : vr - cr;
      const i64 sR = vl + cl > vr + cr ? vl + cl : vr + cr;
      k = 0;
      if (sL >= 0) {
        side = 1;
      } else if (sR <= 0) {
        side = 2;
      } else {
        // sR/(sR - sL), both speeds below 2^62: the quotient in FP64
        const double sr = to_double_int(sR, 0), sl = to_double_int(sL, 0);
        x = half_fixed(sr * rcp(sr - sl), 0);
        if (x > (1LL << 62)) x = 1LL << 62;
        k = mul(limbs(x), limbs(sL)) << 2;
      }
    }
    kap = limbs(k);
    w = limbs(x);
  }
  // one component: the fluxes in units 2^ea, the jump d in 2^ed
  __device__ __forceinline__ double operator()(i64 fl, i64 fr, int ea, i64 d, int ed) const {
    i64 a;
    if (!hll) {
      a = (fl >> 1) + (fr >> 1);
    } else {
      a = (fr >> 1) + (mul(w, limbs((fl >> 1) - (fr >> 1))) << 2);
    }
    ea += hll ? 1 : 0;
    int n;
    const i64 dn = normalised(d, n);
    const i64 b = mul(kap, limbs(dn));
    const int eb = ed - n + eL + 2 - kx;
    if (b == 0) return to_double_int(a, ea);
    if (a == 0) return to_double_int(b, eb);
    // both to the coarser unit, one bit of headroom
    const int base = (ea > eb ? ea : eb) + 1;
    const int sa = base - ea < 63 ? base - ea : 63, sb = base - eb < 63 ? base - eb : 63;
    return to_double_int((a >> sa) + (b >> sb), base);
  }
};

// one trace: v (62 - ev, normal first), p (62 - ee), c2 = p/rho (61 - ee - er1)
// and the physical flux: mass (62 - em), momenta (61 - em - ev, without p),
// energy (60 - ee - ev)
template <int D>
struct FaceSide {
  i64 m[D];  // 63 - em
  i64 E;     // 62 - ee
  i64 vn, p, c2, fm[D], fe;
};

// The physical flux of a 2D trace (normal component first) in FP64. Out of
// line, the compiler else issues its few FP64 instructions under predicates in
// every warp (HLL faces of 185 x 225 elements of degree 3 33 us, 27 so); in 3D
// it branches, and a call would cost registers (3%).
struct SideFlux2 {
  double f[4];
};
static __device__ __noinline__ SideFlux2 side_flux_2d(double rho, double mn, double mt, double E,
                                                      double gm1) {
  const double c[4] = {rho, mn, mt, E};
  double rr;
  const Prim<double, 2> q = prim_rcp<2>(c, gm1, rr);
  return {{mn, fma(mn, q.v[0], q.p), mn * q.v[1], (E + q.p) * q.v[0]}};
}

// LLF or HLL from the conserved traces, normal component first. Returns false
// (f not written) if the FP64 form is due.
template <int D>
__device__ __forceinline__ bool face_fixed(bool hll, const double* cl, const double* cr,
                                           double gamma, double gm1, double f[D + 2]) {
  auto hiword = [](double x) { return (unsigned)__double2hiint(x); };
  const unsigned rl = hiword(cl[0]), rr = hiword(cr[0]);
  const unsigned rmax = rl > rr ? rl : rr, rmin = rl > rr ? rr : rl;
  unsigned km = 0;
#pragma unroll
  for (int k = 0; k < D; ++k) {
    const unsigned a = hiword(cl[1 + k]) & 0x7fffffffu, b = hiword(cr[1 + k]) & 0x7fffffffu;
    km = a > km ? a : km;
    km = b > km ? b : km;
  }
  const unsigned el = hiword(cl[D + 1]), er_ = hiword(cr[D + 1]);
  const unsigned ke = el > er_ ? el : er_;  // above 0x7ff... if one is negative or NaN
  const unsigned kd = ke - (el > er_ ? er_ : el);
  const unsigned lo = (kBias - 150u) << 20, hi = (kBias + 150u) << 20;
  if (!(rmax < hi && rmin > lo && rmax - rmin < (6u << 20) && km < hi && ke < hi && ke > lo &&
        kd < (6u << 20)))
    return false;
  const int eg = exp_above(hiword(gm1));
  const int er = exp_above(rmax);
  int em = exp_above(km);
  if (em < -400) em = -400;  // nothing moves
  const double il = rcp(cl[0]), ir = rcp(cr[0]);
  const int e1 = exp_above(hiword(rl > rr ? ir : il));  // 1/rho < 2^e1
  const int ev = em + e1;
  int ee = exp_above(ke) + 1 + (eg > 0 ? eg : 0);
  if (ee < em + ev) ee = em + ev;
  const int sh = ee - em - ev;  // kinetic energy (61 - em - ev) to 62 - ee, halved
  const Limbs G = limbs(full_fixed(gm1, eg));
  FaceSide<D> S[2];
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    FaceSide<D>& q = S[s];
    const double* c = s ? cr : cl;
    const Limbs r1 = limbs(full_fixed(s ? ir : il, e1));
    i64 ke2 = 0;
    Limbs mn, vn;
    i64 v[D];
#pragma unroll
    for (int k = 0; k < D; ++k) {
      q.m[k] = full_fixed(c[1 + k], em);
      const Limbs mk = limbs(q.m[k]);
      v[k] = mul(mk, r1);  // 62 - ev
      const Limbs vk = limbs(v[k]);
      if (k == 0) {
        mn = mk;
        vn = vk;
      }
      ke2 = fma64(mk, vk, ke2);
    }
    q.E = half_fixed(c[D + 1], ee);
    const i64 I = q.E - (ke2 >> (sh < 63 ? sh : 63));
    if (I <= 0) return false;
    const i64 p = mul(limbs(I), G);  // 61 - ee - eg
    q.p = eg >= -1 ? p << (1 + eg) : p >> (-1 - eg);
    q.vn = v[0];
    q.c2 = mul(limbs(q.p), r1);
#pragma unroll
    for (int k = 0; k < D; ++k) q.fm[k] = mul(mn, limbs(v[k]));
    q.fe = mul(limbs(q.E + q.p), vn);
  }
  // pressures in the momentum fluxes' format: both to 61 - ef
  const int ef = ee > em + ev ? ee : em + ev;
#pragma unroll
  for (int s = 0; s < 2; ++s) {
#pragma unroll
    for (int k = 0; k < D; ++k) {
      const int d = ef - em - ev;
      S[s].fm[k] = S[s].fm[k] >> (d < 63 ? d : 63);
    }
    S[s].fm[0] += S[s].p >> (1 + ef - ee);
  }
  // wave speeds: the larger sound speed (LLF) or both (HLL)
  const i64 cm = S[0].c2 > S[1].c2 ? S[0].c2 : S[1].c2;
  const int ec = ee + e1 - 61;
  const double ca = sqrt_pos(gamma * to_double(hll ? S[0].c2 : cm, ec));
  const double cb = hll ? sqrt_pos(gamma * to_double(S[1].c2, ec)) : ca;
  const unsigned kc = hiword(ca) > hiword(cb) ? hiword(ca) : hiword(cb);
  if (kc >= hi) return false;
  const int es = exp_above(kc);
  FaceBlend blend;
  blend.speeds(hll, S[0].vn, S[1].vn, ev, half_fixed(ca, es), half_fixed(cb, es), es);
  if (blend.side) {
    const double* c = blend.side == 1 ? cl : cr;
    double cc[D + 2];
#pragma unroll
    for (int v = 0; v < D + 2; ++v) cc[v] = c[v];
    if constexpr (D == 2) {
      const SideFlux2 o = side_flux_2d(cc[0], cc[1], cc[2], cc[3], gm1);
#pragma unroll
      for (int v = 0; v < 4; ++v) f[v] = o.f[v];
    } else {
      double rr;
      const Prim<double, D> q = prim_rcp<D>(cc, gm1, rr);
      f[0] = cc[1];
#pragma unroll
      for (int k = 0; k < D; ++k) f[1 + k] = fma(cc[1], q.v[k], k == 0 ? q.p : 0.0);
      f[D + 1] = (cc[D + 1] + q.p) * q.v[0];
    }
    return true;
  }
  const i64 drho = full_fixed(cr[0], er) - full_fixed(cl[0], er);
  f[0] = blend(S[0].m[0], S[1].m[0], em - 63, drho, er - 63);
#pragma unroll
  for (int k = 0; k < D; ++k)
    f[1 + k] = blend(S[0].fm[k], S[1].fm[k], ef - 61, (S[1].m[k] >> 1) - (S[0].m[k] >> 1), em - 62);
  f[D + 1] = blend(S[0].fe, S[1].fe, ee + ev - 60, S[1].E - S[0].E, ee - 62);
  return true;
}

}  // namespace fx
}  // namespace dg
