// One pair of 32-body sub-tiles of the pair loops: the arithmetic is chosen (integer fixed point,
// pairint.cuh, or a fallback in FP64), the pairs of a range of rotation steps evaluated, and the
// sums of both sides added to FP64 accumulators.
#pragma once

#include "pairint.cuh"

namespace mstar {

// The near and invalid pairs of a sub-tile pair as one bit per step: bit k of lane l's word is
// set when body i must not meet j-slot (l + k) mod 32 of the sub-tile. near_row: the tree's near
// partners of body i among those 32 (k_near_words; null: none are masked); cnt: bodies of the
// sub-tile below n; self: the sub-tile is the warp's own (each pair once: step 16 for half the
// lanes).
__device__ __forceinline__ unsigned mask_word(const unsigned* near_row, bool i_pad, int cnt, bool self, int lane) {
  unsigned w = near_row ? *near_row : 0u;
  if (cnt < 32) w |= cnt > 0 ? ~0u << cnt : ~0u;
  w = __funnelshift_r(w, w, lane);
  if (self && lane >= 16) w |= 1u << 16;
  return i_pad ? ~0u : w;
}

// Floats ordered as signed integers, for the warp-wide minima and maxima.
__device__ __forceinline__ int float_key(float f) {
  const int b = __float_as_int(f);
  return b ^ ((b >> 31) & 0x7fffffff);
}
__device__ __forceinline__ float key_float(int k) { return __int_as_float(k ^ ((k >> 31) & 0x7fffffff)); }

// Common scale of a tile pair for the integer pair arithmetic (pairint.cuh).
struct FixWindow {
  bool ok;        // the tile pair can be taken in integers
  int u;          // unit 2^u of the positions
  float inv_max;  // 1 / r^2 limit: pairs closer than 2^-10 of the extent are not taken
};

// From the extents lo[3], hi[3] of the two tiles' bodies and, unless all masses are equal (which the
// float bounds leave out), the exponent of the smallest mass (at least 2^em): every m / r^2 is at
// least 2^(em - 2E - 2), and its float must not vanish or lose bits. The float copies of the
// positions err by 2^-24 of the largest coordinate, which must not exceed 2^8 extents, so a float
// r^2 of a pair at the limit is within 12 % (the limit allows for 30 %).
__device__ __forceinline__ FixWindow fix_window(const float* lo, const float* hi, int em, bool eq, bool ok) {
  FixWindow w;
  const float ext = fmaxf(hi[0] - lo[0], fmaxf(hi[1] - lo[1], hi[2] - lo[2])) * (1.0f + 0x1p-14f);
  float big = 0.0f;
#pragma unroll
  for (int c = 0; c < 3; ++c) big = fmaxf(big, fmaxf(fabsf(lo[c]), fabsf(hi[c])));
  w.ok = ok && ext >= 0x1p-30f && big <= 256.0f * ext;
  const int E = (int)((__float_as_uint(ext) >> 23) & 255u) - 126;  // ext < 2^E
  w.u = E - 62;
  w.ok &= eq || em - 2 * E > -118;
  const float r = ext * 0x1p-10f;
  w.inv_max = 1.0f / (1.3f * r * r);
  return w;
}

// |x| < 2^50 (false for NaN) and equality of bits, off the FP64 pipe.
__device__ __forceinline__ bool below_2_50(double x) {
  return ((unsigned)__double2hiint(x) & 0x7fffffffu) < (1073u << 20);
}
__device__ __forceinline__ bool same_bits(double a, double b) {
  return __double_as_longlong(a) == __double_as_longlong(b);
}

// Extent, mass range and equal masses of a tile pair, for fix_window: every warp of the CTA gives
// its lanes' bodies (those of the i-tile and of the j-tile a lane holds; pads are left out), all get
// the result. sbox: NW x 8 ints of shared memory; every thread of the CTA calls it (it holds a
// barrier when NW > 1). m0: a mass to compare with.
template <int NW>
__device__ __forceinline__ FixWindow tile_window(const double (&pi3)[3], const double (&pj3)[3], double mi, double mj,
                                                 bool i_pad, bool j_pad, double m0, int (*sbox)[8], bool* eq_out) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const float kInf = __int_as_float(0x7f800000);
  float lo[3], hi[3];
  bool ok = true;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const float gi = float_of(pi3[c]), gj = float_of(pj3[c]);
    lo[c] = fminf(i_pad ? kInf : gi, j_pad ? kInf : gj);
    hi[c] = fmaxf(i_pad ? -kInf : gi, j_pad ? -kInf : gj);
    ok &= (i_pad || below_2_50(pi3[c])) && (j_pad || below_2_50(pj3[c]));
  }
  // masses within 2^-41 ... 2^40, so that the float bounds of m / r^2 do not overflow
  const int ei = mass_split(mi).e + 64, ej = mass_split(mj).e + 64;
  ok &= (i_pad || (ei > -40 && ei < 40)) && (j_pad || (ej > -40 && ej < 40));
  const int em = min(i_pad ? 4096 : ei - 1, j_pad ? 4096 : ej - 1);
  bool eq = __all_sync(0xffffffffu, (i_pad || same_bits(mi, m0)) && (j_pad || same_bits(mj, m0)));
  ok = __all_sync(0xffffffffu, ok);
  int key[7];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    key[c] = __reduce_min_sync(0xffffffffu, float_key(lo[c]));
    key[3 + c] = __reduce_max_sync(0xffffffffu, float_key(hi[c]));
  }
  key[6] = __reduce_min_sync(0xffffffffu, em);
  if constexpr (NW > 1) {
    if (lane == 0) {
#pragma unroll
      for (int c = 0; c < 7; ++c) sbox[warp][c] = key[c];
      sbox[warp][7] = (ok ? 1 : 0) | (eq ? 2 : 0);
    }
    __syncthreads();
#pragma unroll
    for (int w = 0; w < NW; ++w) {
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        key[c] = min(key[c], sbox[w][c]);
        key[3 + c] = max(key[3 + c], sbox[w][3 + c]);
      }
      key[6] = min(key[6], sbox[w][6]);
      ok &= (sbox[w][7] & 1) != 0;
      eq &= (sbox[w][7] & 2) != 0;
    }
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    lo[c] = key_float(key[c]);
    hi[c] = key_float(key[3 + c]);
  }
  FixWindow fw = fix_window(lo, hi, key[6], eq, ok);
  // The three components of a force share one unit. Where this warp's bodies lie flat (the mean
  // distance from the middle of the extent along one axis below an eighth of that along
  // another), the small component would keep fewer bits than binary64 sums do: not taken.
  const float sc = exp2f((float)(-(fw.u + 62))) * 0x1p16f;  // extent -> at most 2^16
  unsigned dev[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const float mid = 0.5f * (lo[c] + hi[c]);
    const float di = i_pad ? 0.0f : fabsf(float_of(pi3[c]) - mid) * sc;
    const float dj = j_pad ? 0.0f : fabsf(float_of(pj3[c]) - mid) * sc;
    dev[c] = __reduce_add_sync(0xffffffffu, (unsigned)fminf(di + dj, 0x1p20f));
  }
  fw.ok &= 8u * min(dev[0], min(dev[1], dev[2])) >= max(dev[0], max(dev[1], dev[2]));
  *eq_out = eq;
  return fw;
}

// mass = m 2^e with m in [2^62, 2^63), for fix_pair.
__device__ __forceinline__ MassSplit fix_mass(double m) {
  MassSplit s = mass_split(m);
  s.m >>= 1;
  s.e += 1;
  return s;
}

// The lane's body of the i side. Its binary64 position and mass stay in memory: only the fallback
// reads them, and registers bound the warps in flight.
struct TilePos {
  long long fx, fy, fz;  // fixed point
  float gx, gy, gz, gm;  // float copies (gm: the mass's root)
  MassSplit ms;          // fix_mass
  __device__ __forceinline__ void set(double x, double y, double z, double m, const FixWindow& w) {
    fx = fix_of(x, w.u);
    fy = fix_of(y, w.u);
    fz = fix_of(z, w.u);
    ms = fix_mass(m);
    gx = float_of(x);
    gy = float_of(y);
    gz = float_of(z);
    gm = sqrtf(float_of(m));
  }
};

// Its binary64 position and mass, for the fallback.
struct BodyPos {
  double x, y, z, m;
};

// A load that the compiler does not replace by a value it has loaded before (and would have to keep
// in registers until then).
__device__ __forceinline__ double load_again(const double* p) {
  double x;
  asm volatile("ld.global.f64 %0, [%1];" : "=d"(x) : "l"(p));
  return x;
}

// TilePos with its sums over the partners met so far.
struct TileBody : TilePos {
  double ax = 0.0, ay = 0.0, az = 0.0, u = 0.0;
  UAcc uacc;             // sum of m_j / r_ij of the pairs taken in the mixed arithmetic
  bool bad = false;      // a coincident pair: the force is undefined
  __device__ __forceinline__ double u_sum() const {
    return bad ? __longlong_as_double(0x7ff8000000000000LL) : u + uacc.value();
  }
};

// A sub-tile of partners in shared memory (32 entries each), the warp's own accumulators for it
// (jx, jy, jz, with the opposite sign) and its scratch.
struct SubTile {
  const double *x, *y, *z;
  const long long *fx, *fy, *fz;
  const unsigned long long* mm;  // fix_mass
  const int* me;
  const float4* f;               // float copies: x, y, z and the mass's root
  const double* m;               // masses (read by the plain fallback only)
  double *jx, *jy, *jz;
  long long *bx, *by, *bz;       // integer sums of the partners
  int* cj;                       // the c of their units (fix_pair)
};

// The float pass over kPre steps from k on: inv_hi, 1 / r^2 of the closest pair; the largest force on
// body i and, handed from lane to lane with the partners, on each j, as fi and fj: m_j / r^2, with
// the square root taken of it where masses differ (t.f and b.gm then hold the masses' roots);
// and the largest m_j / r of body i. With equal masses the bounds leave the mass out.
template <int kPre, bool kEq>
__device__ __forceinline__ void bound_steps(const TilePos& b, const SubTile& t, unsigned mw, int k, int lane,
                                            float& inv_hi, float& fi, float& fj, float& pu) {
#pragma unroll
  for (int q = 0; q < kPre; ++q, ++k) {
    const float4 c = t.f[(lane + k) & 31];
    const float dx = c.x - b.gx, dy = c.y - b.gy, dz = c.z - b.gz;
    const float r2 = fmaf(dz, dz, fmaf(dy, dy, dx * dx));
    if (kEq) {
      float inv = rcp_approx(r2);
      inv = (mw >> k) & 1u ? 0.0f : inv;
      fi = fmaxf(fi, inv);
      fj = fmaxf(fj, inv);
    } else {
      float rinv = rsqrt_seed(r2);
      rinv = (mw >> k) & 1u ? 0.0f : rinv;
      const float a = c.w * rinv;
      inv_hi = fmaxf(inv_hi, rinv);
      fi = fmaxf(fi, a);
      fj = fmaxf(fj, b.gm * rinv);
      pu = fmaxf(pu, c.w * a);
    }
    fj = __shfl_sync(0xffffffffu, fj, (lane + 1) & 31);  // now of partner (lane + k + 1) mod 32
  }
}

// Steps [k0, k1) of the warp's rotation (a multiple of kPre of them): at step k lane l meets partner
// (l + k) mod 32, unless bit k of its mask mw is set. m0: the common mass when eq. The fallback for
// pairs that integers do not serve is the mixed FP64 / integer arithmetic, FP64 throughout, which
// takes masses of any value and leaves NaN where bodies coincide, or the caller's; pos() reads body
// i's binary64 position and mass for it. True if integers served. kUnroll: steps of the integer
// loops written out in a row (two where code size does not count).
enum class Fallback { mixed, plain, none };
template <Fallback kFallback, int kPre, int kUnroll, typename Pos>
__device__ __forceinline__ bool subtile_pairs(TileBody& b, const SubTile& t, const FixWindow& fw, bool eq, double m0,
                                              unsigned mw, int k0, int k1, int lane, Pos pos) {
  // The closest pair decides whether integers serve. It is looked at every kPre steps: where it
  // rules them out, it mostly does so at once (attempts at N = 10002 with 5 % of the bodies 10^3
  // core radii out: 69.3 ms with the pass run to its end, 64.5 with this and float_of).
  float fi = 0.0f, fj = 0.0f, pu = 0.0f, inv_hi = 0.0f;
  if (fw.ok) {
    if (eq) {
      for (int k = k0; k < k1; k += kPre) {
        bound_steps<kPre, true>(b, t, mw, k, lane, inv_hi, fi, fj, pu);
        if (__any_sync(0xffffffffu, fi > fw.inv_max)) break;
      }
      inv_hi = fi;
      pu = sqrtf(fi);
    } else {
      const float rinv_max = sqrtf(fw.inv_max);
      for (int k = k0; k < k1; k += kPre) {
        bound_steps<kPre, false>(b, t, mw, k, lane, inv_hi, fi, fj, pu);
        if (__any_sync(0xffffffffu, inv_hi > rinv_max)) break;
      }
      inv_hi *= inv_hi;
      fi *= fi;
      fj *= fj;
    }
    fj = __shfl_sync(0xffffffffu, fj, (lane - k1) & 31);  // held for partner lane + k1: to its own lane
  }
  const bool ints = __all_sync(0xffffffffu, fw.ok && inv_hi <= fw.inv_max);
  if (ints) {
    // accumulator units 2^L: forces and potentials below 2^58 units (the bounds hold within 1.5)
    const int Li = (int)(__float_as_uint(1.5f * fi) >> 23) - 184, Lj = (int)(__float_as_uint(1.5f * fj) >> 23) - 184,
              LU = (int)(__float_as_uint(1.5f * pu) >> 23) - 184;
    const int cx = 116 + 2 * fw.u + (eq ? 64 : 0), ci = Li + cx, cu = LU + 60 + fw.u + (eq ? 64 : 0);
    t.cj[lane] = Lj + cx;
    t.bx[lane] = 0;
    t.by[lane] = 0;
    t.bz[lane] = 0;
    __syncwarp();
    FixAcc ai{0, 0, 0};
    // the sum's shifts truncate: half a unit back for every term
    unsigned long long ui = __popc(~mw & (0xffffffffu >> (32 - k1) & 0xffffffffu << k0)) / 2;
    double si = exp2_int(Li), sj = exp2_int(Lj), su = exp2_int(LU);
    if (eq) {
#pragma unroll kUnroll
      for (int k = k0; k < k1; ++k) {
        const int r = (lane + k) & 31;
        FixAcc aj{t.bx[r], t.by[r], t.bz[r]};
        fix_pair_eq(b.fx, b.fy, b.fz, t.fx[r], t.fy[r], t.fz[r], ci, t.cj[r], cu, (mw >> k) & 1u, ai, aj, ui);
        t.bx[r] = aj.x;
        t.by[r] = aj.y;
        t.bz[r] = aj.z;
        __syncwarp();
      }
      si *= m0;
      sj *= m0;
      su *= m0;
    } else {
#pragma unroll kUnroll
      for (int k = k0; k < k1; ++k) {
        const int r = (lane + k) & 31;
        FixAcc aj{t.bx[r], t.by[r], t.bz[r]};
        fix_pair(b.fx, b.fy, b.fz, t.fx[r], t.fy[r], t.fz[r], b.ms.m, b.ms.e, t.mm[r], t.me[r], ci, t.cj[r], cu,
                 (mw >> k) & 1u, ai, aj, ui);
        t.bx[r] = aj.x;
        t.by[r] = aj.y;
        t.bz[r] = aj.z;
        __syncwarp();
      }
    }
    const long long bias = eq ? 0 : (k1 - k0) * kFixBias;
    b.ax = fma((double)(ai.x - bias), si, b.ax);
    b.ay = fma((double)(ai.y - bias), si, b.ay);
    b.az = fma((double)(ai.z - bias), si, b.az);
    b.u = fma((double)ui, su, b.u);
    t.jx[lane] = fma((double)(t.bx[lane] - bias), sj, t.jx[lane]);
    t.jy[lane] = fma((double)(t.by[lane] - bias), sj, t.jy[lane]);
    t.jz[lane] = fma((double)(t.bz[lane] - bias), sj, t.jz[lane]);
    __syncwarp();
  } else if constexpr (kFallback == Fallback::plain) {
    const BodyPos bi = pos();
#pragma unroll 1
    for (int k = k0; k < k1; ++k) {
      const int r = (lane + k) & 31;
      const double dx = t.x[r] - bi.x, dy = t.y[r] - bi.y, dz = t.z[r] - bi.z, mj = t.m[r];
      double rinv = rsqrt_fp64(fma(dz, dz, fma(dy, dy, dx * dx)));
      rinv = (mw >> k) & 1u ? 0.0 : rinv;
      const double rinv3 = (rinv * rinv) * rinv;
      const double sj = mj * rinv3, si = bi.m * rinv3;
      b.ax = fma(sj, dx, b.ax);
      b.ay = fma(sj, dy, b.ay);
      b.az = fma(sj, dz, b.az);
      b.u = fma(mj, rinv, b.u);
      t.jx[r] = fma(si, dx, t.jx[r]);
      t.jy[r] = fma(si, dy, t.jy[r]);
      t.jz[r] = fma(si, dz, t.jz[r]);
      __syncwarp();
    }
  } else if constexpr (kFallback == Fallback::mixed) {
    const BodyPos bi = pos();
#pragma unroll 2
    for (int k = k0; k < k1; ++k) {
      const int r = (lane + k) & 31;
      const bool masked = (mw >> k) & 1u;
      double dx = t.x[r] - bi.x, dy = t.y[r] - bi.y, dz = t.z[r] - bi.z;
      // keep the separations in registers: recomputing them for the accumulations would
      // cost three more FP64 instructions per pair
      asm volatile("" : "+d"(dx), "+d"(dy), "+d"(dz));
      unsigned long long Rn;
      int eR;
      double sj, si;
      const unsigned long long mjm = t.mm[r] << 1;
      const int mje = t.me[r] - 1;
      pair_scalars_core(dx, dy, dz, MassSplit{mjm, mje}, MassSplit{b.ms.m << 1, b.ms.e - 1}, Rn, eR, sj, si);
      // masked pairs contribute nothing (integer selects on the bit patterns)
      sj = __longlong_as_double(masked ? 0ll : __double_as_longlong(sj));
      si = __longlong_as_double(masked ? 0ll : __double_as_longlong(si));
      b.bad |= !masked && Rn == 0ull;
      // m_j / r = mjm Rn 2^(mje + eR) ~ hi64(mjm Rn) 2^(mje + eR + 64)
      b.uacc.add(masked ? 0ull : __umul64hi(mjm, Rn), masked ? b.uacc.L : mje + eR + 64);
      b.ax = fma(sj, dx, b.ax);
      b.ay = fma(sj, dy, b.ay);
      b.az = fma(sj, dz, b.az);
      // j-side sums are kept with the opposite sign and negated once when written
      t.jx[r] = fma(si, dx, t.jx[r]);
      t.jy[r] = fma(si, dy, t.jy[r]);
      t.jz[r] = fma(si, dz, t.jz[r]);
      __syncwarp();
    }
  }
  return ints;
}

}  // namespace mstar
