// fixed_pair.cuh -- FP64-accurate pair sums with most of the arithmetic on the
// integer pipes.
//
// GB300 issues one FP64 instruction per warp and SM sub-partition in 64
// cycles (measured 68 at the nominal clock), a 32 x 32 -> 64 bit multiply-add
// in 5, other integer instructions in 1 or 2, and the pipes run side by side.
// A single + double layer pair in FP64 takes 27 FP64 instructions besides the
// reciprocal square root; here the differences, the four dot products, 1/r and
// 1/r^2 are fixed point, and the FP64 pipe keeps 9 instructions: the products
// of the dots and the sums into the targets (8 for one layer).
//
// Fixed point: positions are 64-bit integers on one grid for all points
// (quantum 2^(E - 62), 2^E above every coordinate), so d = x - y is exact; d,
// q, n and psi are block fixed point: three 61-bit components on a common
// exponent, their largest at least half of full scale, split into a high part
// (31 bits, signed) and a low part (30 bits, non-negative).  A dot product is
// then 9 multiply-adds into two 64-bit sums and is low by up to 2^-56 (4 units of
// 2^-60 of the vectors' scales) of |a|_max |b|_max, with the operands' rounding 2^-55,
// against the 2^-53 of |a| |b| that FP64 sums carry; 1/r carries up to 2^-55
// before it is rounded to FP64.  The conversions to FP64 truncate (2^-52).  Measured over
// 2 million differences: dots within 3.9 units, 1/r within 1.7 2^-58.
//
// What fixed point cannot hold takes the FP64 pair (fx_slow): a coordinate
// below 2^(E - 10) in magnitude may have bits under the quantum ("inexact"),
// which matters for a pair closer than 2^(E - 8) and for one whose difference is
// nearly perpendicular to n or psi component by component (fx_faint_dot: a flat
// wall seen from just beside it; with exact coordinates its dot products are summed
// exactly instead); pairs closer than 2^(E - 26) (coincident ones among them)
// always take it.
#pragma once

#include <cmath>
#include <cstdint>

#if defined(__CUDACC__)
#include "common.cuh"
#define FX_HD __host__ __device__ __forceinline__
#define FX_RARE static __host__ __device__ __noinline__
#else  // a host build checks the arithmetic (tests/fixed_pair)
namespace stk {
enum Kind : int { K_SL = 1, K_DL = 2, K_SLDL = 3 };
}
#define FX_HD inline
#define FX_RARE static
#endif
#ifndef FX_HOST_ERR  // relative error a host build adds to the estimate of 1/sqrt
#define FX_HOST_ERR 0.f
#endif

namespace stk {

// ------------------------------------------------------------ integer helpers
FX_HD int fx_clz(uint32_t x) {
#if defined(__CUDA_ARCH__)
  return __clz((int)x);
#else
  return x ? __builtin_clz(x) : 32;
#endif
}
// high word of (hi:lo) << s, low word of (hi:lo) >> s, 0 <= s <= 31
FX_HD uint32_t fx_shl(uint32_t lo, uint32_t hi, int s) {
#if defined(__CUDA_ARCH__)
  return __funnelshift_l(lo, hi, s);
#else
  return s ? (hi << s) | (lo >> (32 - s)) : hi;
#endif
}
FX_HD uint32_t fx_shr(uint32_t lo, uint32_t hi, int s) {
#if defined(__CUDA_ARCH__)
  return __funnelshift_r(lo, hi, s);
#else
  return s ? (lo >> s) | (hi << (32 - s)) : lo;
#endif
}
FX_HD int64_t fx_mad(int32_t a, int32_t b, int64_t c) { return (int64_t)a * (int64_t)b + c; }
FX_HD uint64_t fx_mulhi(uint64_t a, uint64_t b) {
#if defined(__CUDA_ARCH__)
  return __umul64hi(a, b);
#else
  return (uint64_t)(((unsigned __int128)a * b) >> 64);
#endif
}
FX_HD int32_t fx_mulhi32(int32_t a, int32_t b) {
#if defined(__CUDA_ARCH__)
  return __mulhi(a, b);
#else
  return (int32_t)(((int64_t)a * b) >> 32);
#endif
}
FX_HD double fx_bits(uint32_t hi, uint32_t lo) {
#if defined(__CUDA_ARCH__)
  return __hiloint2double((int)hi, (int)lo);
#else
  const uint64_t u = ((uint64_t)hi << 32) | lo;
  double d;
  __builtin_memcpy(&d, &u, 8);
  return d;
#endif
}
FX_HD uint64_t fx_to_bits(double d) {
#if defined(__CUDA_ARCH__)
  return (uint64_t)__double_as_longlong(d);
#else
  uint64_t u;
  __builtin_memcpy(&u, &d, 8);
  return u;
#endif
}
FX_HD double fx_fma(double a, double b, double c) {
#if defined(__CUDA_ARCH__)
  return __fma_rn(a, b, c);
#else
  return std::fma(a, b, c);
#endif
}

// ------------------------------------------------------------------- storage
constexpr uint32_t kFxLow = 0x3fffffffu;  // the low part: 30 bits

// A pair whose largest |d_k| has a high word below both points' thresholds
// takes the FP64 form.
constexpr uint32_t kFxExact = 1u;          // exact coordinates: |d| < 2^32 quanta (2^36 with
constexpr uint32_t kFxRoundQ = 2u, kFxRoundN = 4u, kFxRoundP = 8u;  //   these): q, n, psi lost bits
constexpr uint32_t kFxInexact = 1u << 22;  // an inexact coordinate: |d| < 2^54 quanta
constexpr uint32_t kFxNever = ~0u;         // nothing of the point fits

// Positions on the grid, and block fixed point vectors (value = (h 2^30 + l) 2^(e - 60)).
struct alignas(16) SrcFx {
  int64_t y[3];
  uint32_t thr;      // threshold (above)
  int16_t eq, epn;   // exponent of q; of psi and n together
  double q[3];
  int32_t qh[3], ql[3], nh[3], nl[3], ph[3], pl[3];
};
static_assert(sizeof(SrcFx) == 128, "SrcFx layout");

// Exponents the fixed form accepts, of the largest coordinate and of each
// vector's largest component: the FP64 exponent fields below stay in (0, 2047).
constexpr int kFxMaxExp = 300;

// State of the fixed form for one call, in device memory: the largest FP64
// exponent field of a coordinate, whether something does not fit, and the
// sources with an inexact coordinate.
struct FxState {
  int32_t field, bad, inexact, trg_inexact;
};
// What the FP64 engines need besides EngineParams.
struct FxParams {
  const SrcFx *rec;
  const FxState *state;          // NULL: the plain engine alone
  int64_t ns, nt;                // sources, targets
  const double *nrm, *phi, *w;   // the caller's (may be NULL where the kind has no use for it)
  double cdl;                    // double-layer factor
};
FX_HD int fx_exp(const FxState &s) { return s.field - 1022; }
// Points with bits below the grid (coordinates small against the largest one)
// send their close and faint pairs to the FP64 form; with more than one source or
// target in 16 like that the plain FP64 engine takes the call.
FX_HD bool fx_use(const FxState &s, int64_t ns, int64_t nt = 0) {
  const int E = fx_exp(s);
  return !s.bad && E <= kFxMaxExp && E >= -kFxMaxExp && (int64_t)s.inexact * 16 <= ns &&
         (int64_t)s.trg_inexact * 16 <= nt;
}

// A coordinate on the grid of exponent E (|v| < 2^E, kFxMaxExp >= |E|),
// rounded to nearest; thr is raised when bits are dropped.
FX_HD int64_t fx_coord(double v, int E, uint32_t &thr) {
  const uint64_t u = fx_to_bits(v);
  const int ef = (int)((u >> 52) & 0x7ff);
  if (ef == 0) {  // zero or far below the quantum
    if ((u << 1) && thr < kFxInexact) thr = kFxInexact;
    return 0;
  }
  const uint64_t m = (u & 0xfffffffffffffull) | (1ull << 52);
  const int s = ef - 1013 - E;  // m 2^(ef - 1075) = m 2^s quanta
  uint64_t a;
  if (s > 9) {  // outside the grid (the engine's never are)
    thr = kFxNever;
    return 0;
  }
  bool inexact = false;
  if (s >= 0) {
    a = m << s;
  } else if (s < -54) {
    inexact = true;
    a = 0;
  } else {
    const int r = -s;
    inexact = (m & ((1ull << r) - 1)) != 0;
    a = (m + (1ull << (r - 1))) >> r;
  }
  if (inexact && thr < kFxInexact) thr = kFxInexact;
  return (u >> 63) ? -(int64_t)a : (int64_t)a;
}

// FP64 exponent field: |v| < 2^(field - 1022).
FX_HD int fx_field(double v) { return (int)((fx_to_bits(v) >> 52) & 0x7ff); }

// Block fixed point of a vector; returns its exponent e (|v_k| < 2^e; 0 for a
// zero vector, -1022, which fits no form, for one of subnormals).  `flag` is
// added to thr where a component loses bits.
FX_HD int fx_block(const double (&v)[3], int32_t (&h)[3], int32_t (&l)[3], uint32_t &thr,
                   uint32_t flag) {
  int ef = 0;
  uint64_t any = 0;
  for (int k = 0; k < 3; ++k) {
    ef = ef > fx_field(v[k]) ? ef : fx_field(v[k]);
    any |= fx_to_bits(v[k]) << 1;
  }
  const int e = ef || any ? ef - 1022 : 0;
  for (int k = 0; k < 3; ++k) {
    const uint64_t u = fx_to_bits(v[k]);
    const int f = (int)((u >> 52) & 0x7ff);
    int64_t V = 0;
    if (f) {  // (a subnormal or zero component is dropped)
      const uint64_t m = (u & 0xfffffffffffffull) | (1ull << 52);  // m 2^(f - 1075)
      const int s = f - 1015 - e;                                  // to quanta of 2^(e - 60): <= 7
      if (s < 0 && (s <= -54 || (m & ((1ull << -s) - 1)))) thr |= flag;
      if (s >= 0) V = (int64_t)(m << s);
      else if (s > -54) V = (int64_t)((m + (1ull << (-s - 1))) >> -s);
      if (u >> 63) V = -V;
    }
    if (!f && (u << 1)) thr |= flag;
    h[k] = (int32_t)(V >> 30);
    l[k] = (int32_t)((uint32_t)V & kFxLow);
  }
  return e;
}
FX_HD int fx_block(const double (&v)[3], int32_t (&h)[3], int32_t (&l)[3]) {
  uint32_t thr = 0u;
  return fx_block(v, h, l, thr, 0u);
}

// ---------------------------------------------------------------- conversions
// (hi:lo) 2^(eb - 1086) as FP64, truncated, for a magnitude of at least 2^32;
// smaller ones take fx_small, which rounds.  (1023 + 63 = 1086: eb is the exponent field of
// the result for a magnitude in [2^63, 2^64).)
FX_RARE double fx_small(int32_t hi, uint32_t lo, int eb) {
  const int64_t v = (int64_t)(((uint64_t)(uint32_t)hi << 32) | lo);
  if (v == 0) return 0.0;
  const uint64_t u = fx_to_bits((double)v);  // |v| <= 2^32: exact
  const int e = (int)((u >> 52) & 0x7ff) + eb - 1086;
  if (e < 1) return 0.0;
  return fx_bits((uint32_t)(u >> 63 << 31) | ((uint32_t)e << 20) | (uint32_t)((u >> 32) & 0xfffffu),
                 (uint32_t)u);
}
FX_HD double fx_to_double(int64_t v, int eb) {
  const int32_t hi = (int32_t)(v >> 32);
  const uint32_t lo = (uint32_t)v;
  const uint32_t sg = (uint32_t)(hi >> 31);
  const uint32_t h = (uint32_t)hi ^ sg, l = lo ^ sg;  // |v|, or one less
  if (h == 0u) return fx_small(hi, lo, eb);
  const int z = fx_clz(h);
  const uint32_t h2 = fx_shl(l, h, z), l2 = l << z;
  const uint32_t top = (h2 >> 11) + ((uint32_t)(eb - z - 1) << 20);  // the leading one adds 1
  return fx_bits(top | (sg & 0x80000000u), fx_shr(l2, h2, 11));
}

// A block fixed point vector's limbs from its left-justified components.
FX_HD void fx_limbs(int64_t D, int32_t &h, int32_t &l) {
  const uint32_t hi = (uint32_t)((uint64_t)D >> 32), lo = (uint32_t)D;
  h = (int32_t)hi >> 1;
  l = (int32_t)(fx_shr(lo, hi, 3) & kFxLow);
}

// Dot product of two limb vectors in units of 2^(ea + eb - 60).
FX_HD int64_t fx_dot(const int32_t (&ah)[3], const int32_t (&al)[3], const int32_t (&bh)[3],
                     const int32_t (&bl)[3]) {
  int64_t hh = fx_mad(ah[0], bh[0], 0), cr = fx_mad(ah[0], bl[0], 0);
  hh = fx_mad(ah[1], bh[1], hh);
  cr = fx_mad(al[0], bh[0], cr);
  hh = fx_mad(ah[2], bh[2], hh);
  cr = fx_mad(ah[1], bl[1], cr);
  cr = fx_mad(al[1], bh[1], cr);
  cr = fx_mad(ah[2], bl[2], cr);
  cr = fx_mad(al[2], bh[2], cr);
  return hh + (cr >> 30);
}
FX_HD int64_t fx_norm2(const int32_t (&h)[3], const int32_t (&l)[3]) {
  int64_t hh = fx_mad(h[0], h[0], 0), cr = fx_mad(h[0], l[0], 0);
  hh = fx_mad(h[1], h[1], hh);
  cr = fx_mad(h[1], l[1], cr);
  hh = fx_mad(h[2], h[2], hh);
  cr = fx_mad(h[2], l[2], cr);
  return hh + (cr >> 29);
}

// A dot product's error is absolute, some units of 2^-60 of the vectors' scales, where
// FP64's is relative to its products.  So a dot product V far below full scale (2^58 to
// 2^60) is looked at again: where larger products cancel FP64 loses as much and V stands;
// where each of them is small (a plane seen from just beside it) the products are summed
// exactly, if the coordinates and the vector b are exact, and the pair takes the FP64 form
// otherwise (false).  eb: V's exponent as for fx_to_double; exact: see above.
constexpr uint32_t kFxFaint = 1u << 18;  // 2^50 in the units of a dot product
FX_HD bool fx_faint(int64_t V) {
  const int32_t hi = (int32_t)(V >> 32);
  return (uint32_t)(hi ^ (hi >> 31)) < kFxFaint;
}
FX_HD bool fx_faint_dot(int64_t V, const int64_t (&J)[3], const int32_t (&dh)[3],
                        const int32_t (&bh)[3], const int32_t (&bl)[3], bool exact, int eb,
                        double &dot) {
  uint64_t size = 0;
  for (int k = 0; k < 3; ++k)
    size += (uint64_t)(uint32_t)(dh[k] < 0 ? -dh[k] : dh[k]) *
            (uint32_t)(bh[k] < 0 ? -bh[k] : bh[k]);
  if ((uint32_t)(size >> 32) >= kFxFaint) {
    dot = fx_to_double(V, eb);
    return true;
  }
  if (!exact) return false;
  __int128 sum = 0;  // units of 2^-63 of V's
  for (int k = 0; k < 3; ++k) sum += (__int128)J[k] * (((int64_t)bh[k] << 30) + bl[k]);
  const uint64_t sign = (uint64_t)(sum >> 127), hi = (uint64_t)(sum >> 64) ^ sign,
                 lo = (uint64_t)sum ^ sign;
  const int s = hi >> 32 ? 66 - fx_clz((uint32_t)(hi >> 32))  // sum 2^-s has at most 62 bits
                : hi     ? 34 - fx_clz((uint32_t)hi)
                         : (lo >> 62 ? 2 : 0);
  const int64_t v = (int64_t)(sum >> s);
  dot = s ? fx_to_double(v, eb - 63 + s)
          : fx_small((int32_t)(v >> 32), (uint32_t)v, eb - 63);  // rounded, not truncated
  return true;
}
// Whether the coordinates of both points and the vectors flagged are exact.
FX_HD bool fx_is_exact(uint32_t xthr, uint32_t ythr, uint32_t flag) {
  return (xthr | ythr) < kFxInexact && !((xthr | ythr) & flag);
}

// 1/sqrt of W 2^-60, W in [2^58, 2^62): Y 2^(b - 62) with Y in [2^61, 2^62].
// y0 = m 2^-24 is the FP32 estimate of 1/sqrt(w), w = W 2^(2b - 60) in [1, 4);
// with e = 1 - w y0^2, |e| < 2^-20, 1/sqrt(w) = y0 (1 + e/2 + 3 e^2/8 + ...),
// the next term below 2^-61.
FX_HD uint64_t fx_rsqrt(int64_t W, int &b) {
  const uint32_t hi = (uint32_t)((uint64_t)W >> 32), lo = (uint32_t)W;
  b = hi < (1u << 28) ? 1 : 0;
  const uint32_t wh = fx_shl(lo, hi, 2 * b), wl = lo << (2 * b);
#if defined(__CUDA_ARCH__)
  float y = rsqrt_ftz(__uint2float_rz(wh)) * 16384.f;  // wh ~ w 2^28
  y = fminf(fmaxf(y, 0.5f), 0.99999994f);
  const uint32_t m = (__float_as_uint(y) & 0x7fffffu) | 0x800000u;
#else
  float y = (float)(1.0 / std::sqrt((double)(float)wh)) * 16384.f;
  y = y * (1.f + FX_HOST_ERR);
  y = y < 0.5f ? 0.5f : y > 0.99999994f ? 0.99999994f : y;
  uint32_t m;
  __builtin_memcpy(&m, &y, 4);
  m = (m & 0x7fffffu) | 0x800000u;
#endif
  const uint64_t m2 = (uint64_t)m * m;  // y0^2 2^48
  // w y0^2 in units of 2^-60
  const uint64_t t = fx_mulhi(((uint64_t)wh << 32) | wl, m2 << 16);
  const int64_t e = (int64_t)((1ull << 60) - t);
  const int32_t es = (int32_t)(e >> 9);
  const int32_t e2 = fx_mulhi32(es, es);  // e^2 2^70
  const int64_t c = (e >> 1) + (int64_t)((3 * (uint32_t)e2) >> 13);
  // m c < 2^63 in units of 2^-84
  const int64_t mc = (int64_t)((uint64_t)(uint32_t)c * m) +
                     (int64_t)((uint64_t)((uint32_t)(c >> 32) * m) << 32);
  return ((uint64_t)m << 38) + (uint64_t)(mc >> 22);
}

// V 2^-62 in [1/2, 1] as FP64 with exponent field f for [1/2, 1).
FX_HD double fx_round(uint64_t V, int f) {
  const uint64_t M = (V + 256) >> 9;
  return fx_bits((uint32_t)(M >> 32) - 0x100000u + ((uint32_t)f << 20), (uint32_t)M);
}
// a b 2^-62 for a, b in [2^61, 2^62], doubled when below 2^61 (z: whether it was).
FX_HD uint64_t fx_mul62(uint64_t a, uint64_t b, int &z) {
  const uint64_t p = fx_mulhi(a << 1, b << 1);
  z = (uint32_t)(p >> 32) < (1u << 29) ? 1 : 0;
  return p << z;
}

// Difference of two positions, left-justified: d = J 2^(a - 63), |d| 2^-a in
// [1/2, 2) and the limbs of J; false when it is below the points' threshold.
FX_HD bool fx_diff(const int64_t (&x)[3], const int64_t (&y)[3], uint32_t xthr, uint32_t ythr,
                   int E, int64_t (&J)[3], int32_t (&dh)[3], int32_t (&dl)[3], int &a) {
  int64_t d[3];
  uint32_t any = 0u;
  for (int k = 0; k < 3; ++k) {
    d[k] = x[k] - y[k];
    const int32_t hi = (int32_t)(d[k] >> 32);
    any |= (uint32_t)(hi ^ (hi >> 31));
  }
  if (any < xthr || any < ythr) return false;
  const int s = fx_clz(any) - 1;  // left-justified: |J| in [2^62, 2^63)
  for (int k = 0; k < 3; ++k) {
    const uint32_t hi = (uint32_t)((uint64_t)d[k] >> 32), lo = (uint32_t)d[k];
    J[k] = (int64_t)(((uint64_t)fx_shl(lo, hi, s) << 32) | (lo << s));
    fx_limbs(J[k], dh[k], dl[k]);
  }
  a = E + 1 - s;  // d = J 2^-s quanta of 2^(E - 62)
  return true;
}

// ----------------------------------------------------------------------- pair
// Returns false when the pair has to take the FP64 form, else adds it to acc.
//   SL: q/r + d (d.q)/r^3,  DL: d (d.psi)(d.n)/r^5,  K_EQ: SL + s d/r^3 (an
//   equivalent density's force and point source)
// With d = 2^a D, R = |D|: the sums are 2^-a [q + D ((D.q) + 2^-a (D.psi)(D.n)
// /R^2) /R^2] /R for both layers (q = 0 and the first dot left out for DL).
constexpr int K_EQ = 4 | K_SL;
template <int KIND>
FX_HD bool fx_pair(const int64_t (&x)[3], uint32_t xthr, int E, const SrcFx &S, double (&acc)[3],
                   double s0 = 0.0) {
  int64_t J[3];
  int32_t dh[3], dl[3];
  int a, b, z;
  if (!fx_diff(x, S.y, xthr, S.thr, E, J, dh, dl, a)) return false;
  double dp = 0.0, dn = 0.0;
  if (KIND & K_DL) {
    // dots in units of 2^(e - 60): field 1086 + e - 60
    const int64_t vp = fx_dot(dh, dl, S.ph, S.pl), vn = fx_dot(dh, dl, S.nh, S.nl);
    if (!fx_faint(vp)) dp = fx_to_double(vp, 1026 + S.epn - a);
    else if (!fx_faint_dot(vp, J, dh, S.ph, S.pl, fx_is_exact(xthr, S.thr, kFxRoundP),
                           1026 + S.epn - a, dp))
      return false;
    if (!fx_faint(vn)) dn = fx_to_double(vn, 1026);
    else if (!fx_faint_dot(vn, J, dh, S.nh, S.nl, fx_is_exact(xthr, S.thr, kFxRoundN), 1026, dn))
      return false;
  }
  double D[3];
  for (int k = 0; k < 3; ++k) D[k] = fx_to_double(J[k], 1023);  // J 2^-63
  const uint64_t Y = fx_rsqrt(fx_norm2(dh, dl), b);             // 1/R = Y 2^(b - 62)
  const double ria = fx_round(Y, 1022 + b - a);                 // 2^-a / R
  const uint64_t Z = fx_mul62(Y, Y, z);                         // 1/R^2 = Z 2^(2b - z - 62)
  const double ri2 = fx_round(Z, 1022 + 2 * b - z);
  double c;
  if (KIND & K_DL) {
    if (KIND & K_SL) {
      const double dq = fx_to_double(fx_dot(dh, dl, S.qh, S.ql), 1026 + S.eq);
      c = fx_fma(dp * dn, ri2, dq) * ri2;
    } else {
      c = (dp * dn) * (ri2 * ri2);
    }
  } else {
    c = fx_to_double(fx_dot(dh, dl, S.qh, S.ql), 1026 + S.eq);
    if (KIND == K_EQ) c = fx_fma(s0, fx_bits((uint32_t)(1023 - a) << 20, 0u), c);
    c *= ri2;
  }
  if (KIND & K_SL) {
    for (int k = 0; k < 3; ++k) acc[k] = fx_fma(fx_fma(D[k], c, S.q[k]), ria, acc[k]);
  } else {
    c *= ria;
    for (int k = 0; k < 3; ++k) acc[k] = fx_fma(D[k], c, acc[k]);
  }
  return true;
}

// The adjoint's pairs (adjoint.cu) use the same parts for n points of both sets;
// the coordinates' exponent is within kFxAdjExp so that 1/r^3 stays in range.
constexpr int kFxAdjExp = 100;
FX_HD bool fx_adj_use(const FxState &s, int64_t n) {
  const int E = fx_exp(s);
  return fx_use(s, n) && E <= kFxAdjExp && E >= -kFxAdjExp;
}

}  // namespace stk
