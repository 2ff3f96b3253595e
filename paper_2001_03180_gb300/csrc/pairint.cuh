// Pair interactions in integer arithmetic: the separations, 1/r, 1/r^3, the two forces and the
// potential of a pair, accumulated in 64-bit fixed point, with no FP64 instruction per pair.
//
// Why: this part issues one FP64 warp instruction per 16 cycles per SM, so the nine of the
// mixed loop (three separations, six accumulations) take 144 cycles of an SM per warp step
// however little else the step does. The interaction below takes 175 integer and FP32
// instructions, 46 of them 32 x 32 + 64 bit multiply-adds, which bind it: 78 cycles per warp
// step and SM in a loop of its own, 65 with equal masses.
//
// Positions of the two tiles are fixed-point integers X = round(x 2^-u) (mod 2^64) with one u
// for the tile pair, chosen so that no difference reaches 2^62. A coordinate of at least 2^-10
// of the tile pair's extent is represented exactly, and its differences are exact too, where
// FP64 rounds them; the others are rounded at 2^-63 of the extent. Only pairs at least 2^-10 of
// the extent apart are taken here (fix_window), so a separation is wrong by at most 2^-53 of r.
//
// Per pair: D = X_j - X_i is shifted so that its largest component lies in [2^61, 2^62)
// (normalisation by s bits), split into signed 32-bit halves, and
//   r^2 = M 2^(64 + 2 (u - s)),        M in (2^58, 3 2^60], truncated to an integer;
//   1/r = Rn 2^(s - u - 124)           from a float seed y and the series 1 + e/2 + 3 e^2/8 with
//                                      e = 1 - r^2 y^2 formed in units of 2^-72;
//   1/r^3 normalised to [2^62, 2^63),  S = m / r^3 in [2^60, 2^62);
//   force component = (S D) >> 64, rounded to nearest, S shifted first to the accumulator's unit.
// Errors: below 2^-55 relative on S (truncations), half a unit on each product. The unit 2^L of a
// body's accumulators is 2^-58 of a power of two at least 1.3 times the largest force of these 32
// partners on that body, so a sum of up to 32 terms stays below 2^63 and a term is off by at most
// a unit: a binary64 accumulation loses 2^-54 of the running sum per term.
// Where all masses are equal the products are formed once, in the finer of the two bodies' units, and
// shifted down for the other without rounding: half a unit per term too low on average there, at most
// 2^-52 of the largest force of the 32 partners in all. Against long double sums (n = 64, 600, 2047 Plummer
// spheres, in units of 2^-53 of a body's force) the mean error of a component is 0.00 to 0.08,
// within its statistical error, and the rms error 0.4, 0.6 and 0.83; FP64 sums had 0.6, 0.8 and
// 1.2, and rounded shifts 0.4, 0.6 and 0.65 for 9 % more time (N = 10002 attempts 32.0 against 29.5 ms).
// The potential m_j / r is truncated to a unit of its own, 2^-58 of a power of two at least 1.3 and at
// most 4 times the largest m_j / r among the body's partners that are not masked, whatever the body's
// own mass and those of the other bodies: half a unit is given back for every term, so 32 terms err
// by at most 2^-52 of the sum together, 2^-55 typically, for any ratio of the masses.
#pragma once

#include "device.cuh"

namespace mstar {

// round(x 2^-u) mod 2^64 (two's complement).
__device__ __forceinline__ long long fix_of(double x, int u) {
  const int hi = __double2hiint(x);
  const int e = (hi >> 20) & 0x7ff;
  const unsigned long long sig =
      ((unsigned long long)(((unsigned)hi & 0xfffffu) | 0x100000u) << 32) | (unsigned)__double2loint(x);
  const int s = e - 1075 - u;  // x = sig 2^s in units of 2^u
  unsigned long long v;
  if (s >= 0) {
    v = s < 64 ? sig << s : 0ull;
  } else {
    v = s > -55 ? ((sig >> (-s - 1)) + 1ull) >> 1 : 0ull;
  }
  return (long long)(hi < 0 ? 0ull - v : v);
}

// x to the nearest float (halfway cases away from zero; 0 below 2^-126; |x| < 2^127), in integer
// instructions: a conversion holds the FP64 pipe like any other FP64 instruction. The twenty of a pair
// of 32-body tiles (and eight FP64 comparisons) cost 560 of the 5300 cycles that the mixed
// arithmetic then needs for the pairs: attempts on a thin disc of 5003 bodies took 17.9 ms with them,
// 16.7 without.
__device__ __forceinline__ float float_of(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x) + 0x10000000ull;
  const unsigned hi = (unsigned)(b >> 32), lo = (unsigned)b;
  // exponent (9 low bits) and significand; 896 = 1023 - 127
  const unsigned f = __funnelshift_l(lo, hi, 3) - (896u << 23);
  return __uint_as_float((hi & 0x7fffffffu) < (897u << 20) ? 0u : (f & 0x7fffffffu) | (hi & 0x80000000u));
}

// x >> q for 0 <= q (0 from 64 on), x a 64-bit unsigned value.
__device__ __forceinline__ unsigned long long shr_clamp(unsigned long long x, int q) {
  unsigned long long r;
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(q));
  return r;
}

__device__ __forceinline__ float rsqrt_seed(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

__device__ __forceinline__ float rcp_approx(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// 2^e for a normal result.
__device__ __forceinline__ double exp2_int(int e) { return __hiloint2double((e + 1023) << 20, 0); }

// 32 x 32 + 64 bit multiply-adds. Written out: from the equivalent 64-bit expressions the compiler
// builds 1.4 times the instructions (335 against 246 per warp step of the whole kernel).
__device__ __forceinline__ unsigned long long madu(unsigned a, unsigned b, unsigned long long c) {
  unsigned long long r;
  asm("mad.wide.u32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
}
__device__ __forceinline__ unsigned long long mulu(unsigned a, unsigned b) {
  unsigned long long r;
  asm("mul.wide.u32 %0, %1, %2;" : "=l"(r) : "r"(a), "r"(b));
  return r;
}
__device__ __forceinline__ long long mads(int a, int b, long long c) {
  long long r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
}
__device__ __forceinline__ long long muls(int a, int b) {
  long long r;
  asm("mul.wide.s32 %0, %1, %2;" : "=l"(r) : "r"(a), "r"(b));
  return r;
}

// Accumulators of one body's force components in units of 2^L. Every fix_add leaves 2^30 too much
// in each (kFixBias; the products' middle parts are kept non-negative, which saves their sign
// extension), taken off when the sums are read.
struct FixAcc {
  long long x, y, z;
};
constexpr long long kFixBias = 1ll << 30;

// The three products (S D_c) >> 64, rounded to nearest, added to a. S < 2^62; D_c = h 2^32 + l
// with signed halves, |h| <= 2^30.
__device__ __forceinline__ void fix_add(FixAcc& a, unsigned long long S, int hx, int lx, int hy, int ly, int hz,
                                        int lz) {
  const int sl = (int)(unsigned)S;
  const int sh = (int)(unsigned)((S + 0x80000000ull) >> 32);  // S = sh 2^32 + sl
  const long long k = (1ll << 62) + 0x80000000ll;             // bias (2^30 after the shift), rounding
  a.x = mads(sh, hx, a.x) + (long long)((unsigned long long)mads(sl, hx, mads(sh, lx, k)) >> 32);
  a.y = mads(sh, hy, a.y) + (long long)((unsigned long long)mads(sl, hy, mads(sh, ly, k)) >> 32);
  a.z = mads(sh, hz, a.z) + (long long)((unsigned long long)mads(sl, hz, mads(sh, lz, k)) >> 32);
}

// (a b) >> 64 less the carry of the low halves' product (a, b < 2^63; error < 2 units).
__device__ __forceinline__ unsigned long long mul_top(unsigned long long a, unsigned long long b) {
  const unsigned ah = (unsigned)(a >> 32), al = (unsigned)a, bh = (unsigned)(b >> 32), bl = (unsigned)b;
  return madu(ah, bh, madu(al, bh, mulu(ah, bl)) >> 32);
}

// A pair's geometry in integers: the separation's components d = h 2^32 + l normalised by s bits,
// 1/r = Rn 2^(s - u - 124), and 1/r^3 = R3 2^(3 (s - u - 124) + 128 - s3) (both 0 when masked).
//
// The scales are chosen so that most shifts are by 32 (a choice of register): a 64-bit shift
// costs as much as two of the multiply-adds.
struct FixGeom {
  int hx, lx, hy, ly, hz, lz, s, s3;
  unsigned long long Rn, R3;
};

__device__ __forceinline__ FixGeom fix_geom(long long Xi, long long Yi, long long Zi, long long Xj, long long Yj,
                                            long long Zj, bool masked) {
  FixGeom g;
  long long dx = Xj - Xi, dy = Yj - Yi, dz = Zj - Zi;
  const int n = max(abs((int)(dx >> 32)), max(abs((int)(dy >> 32)), abs((int)(dz >> 32))));
  const int s = __clz(n) - 2;  // n < 2^30: s >= 0
  dx <<= s;
  dy <<= s;
  dz <<= s;
  // signed halves: d = h 2^32 + l
  g.lx = (int)dx;
  g.ly = (int)dy;
  g.lz = (int)dz;
  g.hx = (int)((dx + 0x80000000ll) >> 32);
  g.hy = (int)((dy + 0x80000000ll) >> 32);
  g.hz = (int)((dz + 0x80000000ll) >> 32);
  g.s = s;
  // M = d^2 2^-64, in (2^58, 3 2^60] (the 1 keeps Rn below 2^63; the low halves' squares are below 1)
  const unsigned long long M =
      (unsigned long long)(mads(g.hz, g.hz, mads(g.hy, g.hy, mads(g.hx, g.hx, 1))) +
                           (mads(g.hz, g.lz, mads(g.hy, g.ly, muls(g.hx, g.lx))) >> 31));
  const unsigned mh = (unsigned)(M >> 32), ml = (unsigned)M;
  // y = yb 2^-36 ~ (M 2^-32)^(-1/2) in (2^-14.8, 2^-13]: adding 2^-13 leaves it in the low bits
  unsigned yb = __float_as_uint(rsqrt_seed(__uint2float_rn(mh)) + 0x1p-13f) - 0x39000000u;
  yb = masked ? 0u : yb;
  const unsigned long long Y2 = mulu(yb, yb);
  const unsigned yh = (unsigned)(Y2 >> 32), yl = (unsigned)Y2;
  // e = 1 - M y^2 in units of 2^-72 (|e| < 2^-20.5), from M Y2 >> 32 modulo 2^64
  const unsigned long long w = madu(mh, yl, madu(ml, yh, mulu(ml, yl) >> 32));
  const long long e = -(long long)(((unsigned long long)((unsigned)(w >> 32) + mh * yh) << 32) | (unsigned)w);
  // c = e/2 + 3 e^2/8 in units of 2^-73, and Rn = yb (1 + c) 2^40 in (2^61.2, 2^63)
  const int et = (int)(e >> 32);  // units of 2^-40
  const long long c = e + (long long)(unsigned)(muls(et, et + et + et) >> 10);
  const long long rc = mads((int)yb, (int)(c >> 32), (long long)(mulu(yb, (unsigned)c) >> 32));
  g.Rn = ((unsigned long long)rc + ((unsigned long long)(yb << 9) << 32)) >> 1;
  const unsigned a = (unsigned)(g.Rn >> 32), b = (unsigned)g.Rn;
  const unsigned long long R2 = madu(a, a, mulu(a + a, b) >> 32);
  const unsigned a2 = (unsigned)(R2 >> 32), b2 = (unsigned)R2;
  const unsigned long long R3 = madu(a2, a, madu(b2, a, mulu(a2, b)) >> 32);
  g.s3 = __clz((int)(R3 >> 32)) - 1;  // R3 in (2^55.6, 2^61) when not masked (0 stays 0)
  g.R3 = R3 << g.s3;
  return g;
}

// One pair. Xi, Xj: fixed-point positions; mmi 2^mei, mmj 2^mej the masses (mm in [2^62, 2^63));
// ci = L_i + 116 + 2u and cj likewise (L the exponent of the accumulators' unit); cu = L_U + 60 +
// u for the potential. Adds m_j d / r^3 to ai, m_i d / r^3 to aj (the partner's sums keep the
// opposite sign) and m_j / r to ui; only the biases when masked.
__device__ __forceinline__ void fix_pair(long long Xi, long long Yi, long long Zi, long long Xj, long long Yj,
                                         long long Zj, unsigned long long mmi, int mei, unsigned long long mmj, int mej,
                                         int ci, int cj, int cu, bool masked, FixAcc& ai, FixAcc& aj,
                                         unsigned long long& ui) {
  const FixGeom g = fix_geom(Xi, Yi, Zi, Xj, Yj, Zj, masked);
  const int qs = g.s3 - 2 * g.s;
  fix_add(ai, shr_clamp(mul_top(mmj, g.R3), ci - mej + qs), g.hx, g.lx, g.hy, g.ly, g.hz, g.lz);
  fix_add(aj, shr_clamp(mul_top(mmi, g.R3), cj - mei + qs), g.hx, g.lx, g.hy, g.ly, g.hz, g.lz);
  ui += shr_clamp(mul_top(mmj, g.Rn), cu - mej - g.s);
}

// The same for two tiles whose bodies all have one mass, which the sums leave out: m = 1, with 64
// (its exponent beside a significand of 2^64) added to ci, cj and cu. The products are formed once,
// in the finer of the two bodies' units, and shifted to each. 65 cycles per warp step and SM in a
// loop of its own, against 78 with the masses. No bias is left in the sums.
__device__ __forceinline__ void fix_pair_eq(long long Xi, long long Yi, long long Zi, long long Xj, long long Yj,
                                            long long Zj, int ci, int cj, int cu, bool masked, FixAcc& ai,
                                            FixAcc& aj, unsigned long long& ui) {
  const FixGeom g = fix_geom(Xi, Yi, Zi, Xj, Yj, Zj, masked);
  const int cm = min(ci, cj);
  const unsigned long long S = shr_clamp(g.R3, cm + g.s3 - 2 * g.s);
  FixAcc p{-kFixBias, -kFixBias, -kFixBias};
  fix_add(p, S, g.hx, g.lx, g.hy, g.ly, g.hz, g.lz);
  const int qi = ci - cm, qj = cj - cm;
  ai.x += p.x >> qi;
  ai.y += p.y >> qi;
  ai.z += p.z >> qi;
  aj.x += p.x >> qj;
  aj.y += p.y >> qj;
  aj.z += p.z >> qj;
  ui += shr_clamp(g.Rn, cu - g.s);
}

}  // namespace mstar
