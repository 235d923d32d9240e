// Ranocha's volume flux in 64-bit fixed point (FP64 meshes).
//
// The FP64 unit of this GPU issues one warp instruction per 64 cycles and SM
// sub-partition, so a flux-differencing kernel in FP64 spends nearly all its
// time there with the other pipes idle (88% of the cycles at N = 3). The same
// sub-partition multiplies two 64-bit integers to their high 64 bits and adds
// a third in about 18 cycles and adds two in 3, both measured. The pair
// fluxes are polynomials in values of bounded size apart from the two
// logarithmic means, so inside one element they run on integers scaled by
// per-element powers of two, with 62 to 63 bits below the element's largest
// value (FP64 has 53 below each value's own). An element is taken if its
// densities and its internal energies lie within a factor 2^6 of each other
// each (the latter less the bits by which the kinetic energies exceed them: at
// gamma = 1.4 an element of uniform energies is refused from a Mach number
// between 5.7 and 10.6, where its powers of two fall, and one of energies 6
// times apart between 3.0 and 5.1), its total energies within 2^10 of the units
// and the velocities on every node's lines within 2^6 of the largest
// (element_scale; energy_far and cross_far in dg_rhs_kernels.cuh): each node's
// sums then keep at least 45 bits of their own size, nearly all of them more
// than FP64's. Other elements, and any that hold a non-finite or non-positive
// value, take the FP64 form in the same kernel (fx_pair; measured beside
// volume_fx_kernel).
//
// The logarithmic means need no division: with L = ln(rho), D = L_b - L_a,
//   ln_mean(rho_a, rho_b) = (rho_a + rho_b)/2 tanh(D/2)/(D/2),
// and with e = p/((gamma-1) rho) the internal energy, D = ln(e_b) - ln(e_a),
//   p_a p_b/((gamma-1) ln_mean(rho_a p_b, rho_b p_a)) = (e_a + e_b)/2 D/sinh(D)
// (the left side is the energy term of Ranocha's flux). The logarithms are
// per-node values, each within 2^-53; an error d in D reaches the means only as
// D d/6, far below the rounding of the means.
//
// Numbers: a 64-bit integer X stands for x = X 2^-q 2^E with a format q known
// at compile time and a per-element exponent E (Scale). mul() returns the
// high 64 bits of a product: formats q1 and q2 give q1 + q2 - 64. Operands
// are split into balanced 32-bit limbs (the low one signed), which needs the
// value below 2^63 - 2^32 in magnitude.
//
// With DG_FX_HOST defined the file compiles as plain C++ (the host tests).
#pragma once
#ifdef DG_FX_HOST
#include <cmath>
#define __align__(n) alignas(n)
#else
#include "dg_device.cuh"  // which includes this file before its log means
#endif
#include "dg_fixed_tables.cuh"

namespace dg {
namespace fx {

typedef long long i64;
typedef unsigned long long u64;
#ifdef DG_FX_HOST
#define DG_FX_FN inline
inline int mulhi32(int a, int b) { return (int)(((i64)a * b) >> 32); }
inline u64 dbits(double x) { u64 b; __builtin_memcpy(&b, &x, 8); return b; }
inline double bitsd(u64 b) { double x; __builtin_memcpy(&x, &b, 8); return x; }
static const LogEntry kLog[128] = {DG_FX_LOG_ROWS};
static const i64 kTanhFar[] = DG_FX_TanhFar, kSinhFar[] = DG_FX_SinhFar;
inline LogEntry log_entry(int i) { return kLog[i]; }
inline int clz64(u64 a) { return a ? __builtin_clzll(a) : 64; }
#else
#define DG_FX_FN __device__ __forceinline__
__device__ __forceinline__ int mulhi32(int a, int b) { return __mulhi(a, b); }
__device__ __forceinline__ u64 dbits(double x) { return (u64)__double_as_longlong(x); }
__device__ __forceinline__ double bitsd(u64 b) { return __longlong_as_double((i64)b); }
static __device__ const LogEntry kLog[128] = {DG_FX_LOG_ROWS};
static __constant__ i64 kTanhFar[] = DG_FX_TanhFar, kSinhFar[] = DG_FX_SinhFar;
__device__ __forceinline__ int clz64(u64 a) { return __clzll((i64)a); }
__device__ __forceinline__ LogEntry log_entry(int i) {
  const int4 v = __ldg(reinterpret_cast<const int4*>(kLog) + i);
  LogEntry e;
  e.l = (i64)(((u64)(unsigned)v.y << 32) | (unsigned)v.x);
  e.r = v.z;
  e.pad = 0;
  return e;
}
#endif

// balanced limbs: a = h 2^32 + l, l signed
struct Limbs {
  int h, l;
};
DG_FX_FN Limbs limbs(i64 a) {
  Limbs r;
  r.l = (int)a;
  r.h = (int)(a >> 32) + (int)((unsigned)r.l >> 31);
  return r;
}
// the high 64 bits of a b, plus c. The product of the low limbs is left out
// (at most a quarter of a unit, of either sign) and the two middle products
// are truncated, so a product with zero is zero and any other loses one unit
// on average; sums of many products start from their number of terms to make
// up for it (fx_stage). (Rounding the middle products' 64-bit sum instead
// costs 20% of the volume kernel's time: two IMAD.WIDE with 64-bit addends in
// place of two IMAD.HI.)
DG_FX_FN i64 fma64(Limbs a, Limbs b, i64 c) {
  const int t = mulhi32(a.h, b.l) + mulhi32(a.l, b.h);
  return (i64)a.h * b.h + c + (i64)t;
}
DG_FX_FN i64 mul(Limbs a, Limbs b) {
  const int t = mulhi32(a.h, b.l) + mulhi32(a.l, b.h);
  return (i64)a.h * b.h + (i64)t;
}
DG_FX_FN i64 sqr(Limbs a) {
  const int t = mulhi32(a.h, a.l);
  return (i64)a.h * a.h + ((i64)t + (i64)t);
}
// the product of a and b shifted down by 64 - s bits (0 <= s < 32; within one
// unit), for factors whose element-wide bounds overstate the product
DG_FX_FN i64 mul_up(Limbs a, Limbs b, int s) {
  const i64 mid = (i64)a.h * b.l + ((i64)a.l * b.h + (i64)mulhi32(a.l, b.l)) +
                  (i64)(0x80000000u >> s);
  return (i64)((u64)((i64)a.h * b.h) << s) + (mid >> (32 - s));
}

// ---- per-element scales ----
// rho < 2^er, |v_k| < 2^ev, e < 2^(ee - 1), pressures and momentum fluxes by
// em, energy fluxes by em + ev (element_scale says how much below)
struct Scale {
  int er, ev, ee, em;
  int kv, km, s;  // alignments: v.v to e, mass flux to momentum flux, and
                  // the excess of the bound of rho e over em
  int ok;         // 0: the element takes the FP64 form
};

// Keys are the high words of the (non-negative) doubles; a negative or NaN
// value gives a key above every accepted one.
constexpr unsigned kBias = 1023;
DG_FX_FN int exp_above(unsigned hi) {  // E with x < 2^E (1 - 2^-21), x's high word hi
  return (int)((hi + 1u) >> 20) - (int)kBias + 1;
}
// keys: the largest and smallest density, the largest and smallest internal
// energy, the largest |v_k| and pressure. c[0], c[1]: bits by which em exceeds
// the pressures (scale_bits below).
// With q = rho_a/rho_b, rho_ln times the energies' mean is at most
// sinh(ln(q)/2)/(ln(q)/2) times the geometric mean of p_a/(gamma-1) and
// p_b/(gamma-1): 1.1 for densities within a factor 4, 2.2 within 2^6. So with
// p < 2^(em - c) and rho v^2 < 2^(em - 3) the energy flux stays below
// 1.2 2^(em + ev), whatever product of largest density and largest internal
// energy the element has (on an isobaric density wave that product exceeds
// the pressure by the density ratio).
DG_FX_FN Scale element_scale(const unsigned* key, const int* c) {
  const unsigned rmax = key[0], rmin = key[1], emax = key[2], emin = key[3], vmax = key[4],
                 pmax = key[5];
  Scale s;
  s.er = exp_above(rmax);
  s.ev = exp_above(vmax);
  const int ee = exp_above(emax);
  s.em = exp_above(pmax) + (rmax - rmin < (1u << 20) ? c[0] : c[1]);
  // velocities below 2^-28 of the sound speed keep the scale of that size
  const int floor_ev = (s.em - s.er - 60) >> 1;
  if (s.ev < floor_ev) s.ev = floor_ev;
  if (s.em < s.er + 2 * s.ev + 3) s.em = s.er + 2 * s.ev + 3;
  s.ee = ee + 1;
  if (s.ee < 2 * s.ev + 2) s.ee = 2 * s.ev + 2;
  if (s.ee < s.em - s.er) s.ee = s.em - s.er;
  s.kv = s.ee - 2 * s.ev - 2;
  s.km = s.em - s.er - 2 * s.ev - 2;
  s.s = s.er + s.ee - s.em;
  const unsigned lo = (kBias - 150u) << 20, hi = (kBias + 150u) << 20;
  s.ok = rmax < hi && rmin > lo && emax < hi && emin > lo && vmax < hi && pmax < hi &&
         rmax - rmin < (6u << 20) && emax - emin < (6u << 20) &&
         (int)((emax - emin) >> 20) + s.ee - ee <= 8 && s.s < 16 && s.kv < 63 && s.km < 63;
  return s;
}
// c with p (f/(gamma-1) + 1) < 2^c p, f = 1.1 and 2.2, in FP32 (an FP64
// division in every warp would cost as much as a node's primitives; f has 2%
// to spare)
DG_FX_FN void scale_bits(double gm1, int* c) {
#ifdef DG_FX_HOST
  const float g = (float)gm1;
#else
  const float g = d2f(gm1);
#endif
  const float x[2] = {1.1f / g + 1.0f, 2.2f / g + 1.0f};
  for (int i = 0; i < 2; ++i) {
#ifdef DG_FX_HOST
    unsigned b;
    __builtin_memcpy(&b, &x[i], 4);
#else
    const unsigned b = __float_as_uint(x[i]);
#endif
    c[i] = (int)(b >> 23) - 127 + 1;
  }
}

// x/2 in format 63 - E (|x| < 2^E): the 53-bit significand aligned to bit 62,
// shifted down (truncated) by the exponents' difference
DG_FX_FN i64 half_fixed(double x, int E) {
  const u64 b = dbits(x);
  const int e = (int)(b >> 52) & 0x7ff;
  const u64 m = ((b & 0xfffffffffffffULL) | 0x10000000000000ULL) << 10;
  const int n = E + (int)kBias - e;  // >= 1
  const i64 v = n > 62 ? 0 : (i64)(m >> n);
  return (i64)b < 0 ? -v : v;
}

// ln(x 2^-E) in units of 2^-60 for a positive normal x, within about 2^-53:
// x = m 2^j, m r/256 = 1 + z from the table's reciprocal r, ln(1 + z) = z +
// z^2 g, g = -1/2 + z/3 - ... (w = 2^7 z; the terms from z/3 on in 32 bits)
DG_FX_FN i64 ln_fixed(double x, int E) {
  const u64 b = dbits(x);
  const int j = (int)(b >> 52) - (int)kBias - E;
  const i64 m = (i64)((b & 0xfffffffffffffULL) | 0x10000000000000ULL);
  const LogEntry t = log_entry((int)(b >> 45) & 127);
  const i64 z = m * t.r - (1LL << 60);
  const Limbs w = limbs(z << 9);  // 2^-62 of w
  int y = -8;                     // -1/8 in 2^-6; five bits more in each step
  y = mulhi32(w.h, y) + 293;        // 1/7
  y = mulhi32(w.h, y) - 10923;      // -1/6
  y = mulhi32(w.h, y) + 419430;     // 1/5
  y = mulhi32(w.h, y) - 16777216;   // -1/4
  y = mulhi32(w.h, y) + 715827883;  // 1/3 in 2^-31
  const i64 zy = (i64)w.h * y + (i64)mulhi32(w.l, y);  // 2^-68
  const i64 g = (zy >> 6) - (1LL << 61);               // 2^-62
  const i64 q = mul(limbs(sqr(w)), limbs(g));          // z^2 g, 2^-72
  return z + (q >> 12) + t.l + (i64)j * kLn2;
}

// ---- the logarithmic means from D (units of 2^-60) ----
// |D| < 1/4: x = D^2 (2^-62) and a polynomial of degree 6 in x, its high
// terms in 32 bits; |D| < 1: degree 11 in 64 bits (both below 6e-19)
DG_FX_FN bool d_short(int dh) { return (unsigned)(dh + (1 << 26)) < (1u << 27); }
DG_FX_FN bool d_mid(int dh) { return (unsigned)(dh + (1 << 28) - 1) < (1u << 29) - 2; }

DG_FX_FN i64 short_poly(Limbs x, const i64* c, const int* c32) {
  int y = mulhi32(x.h, c32[2]) + c32[1];
  y = mulhi32(x.h, y) + c32[0];
  i64 r = (i64)x.h * y + c[2];
  r = fma64(x, limbs(r), c[1]);
  return fma64(x, limbs(r), c[0]);
}
template <int n>
DG_FX_FN i64 mid_poly(Limbs x, const i64* c) {
  i64 r = c[n - 1];
#ifndef DG_FX_HOST
#pragma unroll
#endif
  for (int k = n - 2; k >= 0; --k) r = fma64(x, limbs(r), c[k]);
  return r;
}

// |D| from 1 to 4.18 (the accepted ratio 2^6 is 4.16): 1 + c in powers of z =
// (x - 8.75)/16, x = D^2, as a loop over the coefficients (2^-61, within 3e-19);
// c in 2^-61
DG_FX_FN i64 far_poly(i64 D, const i64* c) {
  const i64 x = sqr(limbs(D)) - ((35LL << 56) / 4);  // 2^-56
  const Limbs z = limbs(x << 3);                     // 2^-63
  i64 r = c[kFarN - 1];
#ifndef DG_FX_HOST
#pragma unroll 1
#endif
  for (int k = kFarN - 2; k >= 0; --k) r = c[k] + (mul(z, limbs(r)) << 1);
  return r;
}

// c with mean factor 1 + c, tanh form (2^-64) and sinh form (2^-63), for a
// short D
DG_FX_FN i64 tanh_short(Limbs x) {
  const i64 c[] = DG_FX_TanhShort;
  const int c32[] = DG_FX_TanhShort32;
  return mul(x, limbs(short_poly(x, c, c32)));
}
DG_FX_FN i64 sinh_short(Limbs x) {
  const i64 c[] = DG_FX_SinhShort;
  const int c32[] = DG_FX_SinhShort32;
  return mul(x, limbs(short_poly(x, c, c32)));
}
DG_FX_FN Limbs square_of(i64 D) { return limbs(sqr(limbs(D << 3))); }

// (rho_a + rho_b)/2 tanh(D/2)/(D/2) from the mean s (format 63), any D
DG_FX_FN i64 ln_mean_fixed(i64 s, i64 D) {
  if (!d_mid((int)(D >> 32))) return s + (mul(limbs(s), limbs(far_poly(D, kTanhFar))) << 3);
  const i64 c[] = DG_FX_TanhMid;
  const Limbs x = square_of(D);
  return fma64(limbs(s), limbs(mul(x, limbs(mid_poly<kTanhMidN>(x, c)))), s);
}
// (e_a + e_b)/2 D/sinh(D) from the mean s (format 63), any D
DG_FX_FN i64 inv_ln_mean_fixed(i64 s, i64 D) {
  if (!d_mid((int)(D >> 32))) return s + (mul(limbs(s), limbs(far_poly(D, kSinhFar))) << 3);
  const i64 c[] = DG_FX_SinhMid;
  const Limbs x = square_of(D);
  return fma64(limbs(s), limbs(mul(x, limbs(mid_poly<kSinhMidN>(x, c))) << 1), s);
}
// both means of a pair: the short forms in one block, so that their two
// dependent chains overlap
DG_FX_FN void both_means(i64 sr, i64 dr, i64 se, i64 de, i64& rho, i64& e) {
  if (d_short((int)(dr >> 32)) && d_short((int)(de >> 32))) {
    const i64 cr = tanh_short(square_of(dr)), ce = sinh_short(square_of(de));
    rho = fma64(limbs(sr), limbs(cr), sr);
    e = fma64(limbs(se), limbs(ce << 1), se);
  } else {
    rho = ln_mean_fixed(sr, dr);
    e = inv_ln_mean_fixed(se, de);
  }
}

// ---- the two-point flux ----
// Node values: r = rho/2 (63 - er), e = e/2 (63 - ee), p = p/2 (63 - em),
// v = v/2 (63 - ev), normal component first, and the two logarithms.
template <int D>
struct Node {
  i64 r, lr, e, le, p, v[D];
};

// f[0] mass (62 - er - ev), f[1..D] momenta, normal first (63 - em),
// f[D + 1] energy (61 - em - ev); all below 2^62 in magnitude, but for the
// normal momentum where gamma > 3 (c = 1 in scale_bits): below 1.25 2^62
template <int D>
DG_FX_FN void pair_flux(const Node<D>& a, const Node<D>& b, const Scale& sc, i64 f[D + 2]) {
  i64 rho, ee;
  both_means(a.r + b.r, b.lr - a.lr, a.e + b.e, b.le - a.le, rho, ee);
  const Limbs van = limbs(a.v[0]), vbn = limbs(b.v[0]);
  i64 vv = mul(van, vbn);
#ifndef DG_FX_HOST
#pragma unroll
#endif
  for (int j = 1; j < D; ++j) vv = fma64(limbs(a.v[j]), limbs(b.v[j]), vv);
  ee += vv >> sc.kv;  // v_a.v_b/2 + p_a p_b/((gamma-1) ln_mean), 63 - ee
  const Limbs vn = limbs(a.v[0] + b.v[0]);
  const i64 f0 = mul(limbs(rho), vn);
  f[0] = f0;
  const Limbs g = limbs(f0 >> sc.km);
  f[1] = fma64(g, vn, a.p + b.p);
#ifndef DG_FX_HOST
#pragma unroll
#endif
  for (int j = 1; j < D; ++j) f[1 + j] = mul(g, limbs(a.v[j] + b.v[j]));
  const i64 pv = fma64(limbs(a.p), vbn, mul(limbs(b.p), van));
  f[D + 1] = pv + mul_up(limbs(f0), limbs(ee), sc.s);
}

// ---- results back to FP64 ----
// a 2^e, rounded once: the two halves of a as doubles of known exponents
// (exact), their sum, and the exponent shifted
DG_FX_FN double to_double(i64 a, int e) {
  if (a == 0) return 0.0;
  const unsigned lo = (unsigned)a, hi = (unsigned)((u64)a >> 32) ^ 0x80000000u;
  // 2^84 + hi 2^32, less 2^84 + 2^63 + 2^52, plus 2^52 + lo
  const double h = bitsd(((u64)0x45300000u << 32) | hi) - 19342822341709703277445120.0;
  const double r = h + bitsd(((u64)0x43300000u << 32) | lo);
  return bitsd(dbits(r) + ((u64)(i64)e << 52));
}

// a 2^e rounded to FP64 on the integer pipe (to_double's two FP64 additions
// would double the FP64 work of a face node); ties away from zero
DG_FX_FN double to_double_int(i64 a, int e) {
  if (a == 0) return 0.0;
  const u64 m0 = (u64)(a < 0 ? -a : a);
  const int n = clz64(m0);
  const u64 m = m0 << n;  // leading one at bit 63
  const u64 q = (m >> 11) + ((m >> 10) & 1);
  const u64 b = q + ((u64)(i64)((int)kBias + 62 - n + e) << 52);
  return bitsd(b | ((u64)a & 0x8000000000000000ULL));
}

// ln(y/x) in FP64 for normal x and y in (2^-1000, 2^1000), within 2^-52 and its
// own rounding: the log means' far range (|ln(y/x)| > 1.09) divides by it. On
// the integer pipe: log1p((y - x)/x) costs some 50 instructions of the FP64
// unit, and a warp runs them if only one of its lanes is in that range.
DG_FX_FN double ln_ratio(double x, double y) {
  const int ex = (int)(dbits(x) >> 52) - (int)kBias, ey = (int)(dbits(y) >> 52) - (int)kBias;
  const i64 m = ln_fixed(y, ey) - ln_fixed(x, ex);  // of the significands, 2^-60
  const i64 j = ey - ex;
  if (j > -10 && j < 10) return to_double_int(m + j * kLn2, -60);
  return to_double_int((m >> 8) + j * (kLn2 >> 8) + ((j * (kLn2 & 255)) >> 8), -52);
}
DG_FX_FN bool ln_ratio_in_range(double x, double y) {
  const u64 lo = (u64)(kBias - 1000u) << 52, n = (u64)2000u << 52;
  return dbits(x) - lo < n && dbits(y) - lo < n;
}

}  // namespace fx
}  // namespace dg
