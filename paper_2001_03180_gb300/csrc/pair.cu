// The O(N^2) pair loop (Eq. 2) with the near/far separation rule of Sec. 3.4.
//
// Far pairs use Cartesian separations r_j - r_i; near pairs (within N_d tree edges,
// Eq. LCA) use sums of MST edge vectors. The tiled kernel evaluates every unordered far
// pair exactly once and applies the result to both bodies (a_i += m_j d/r^3,
// a_j -= m_i d/r^3), which halves the work. Near pairs are masked out of the tiles (by words that
// the tree gives) and summed in a sparse pass with the edge-vector separations.
//
// Two arithmetics, chosen per pair of 32-body sub-tiles:
//  - integer (pairint.cuh): the whole interaction on the integer and FP32 pipes, accumulated in
//    64-bit fixed point over the sub-tile and added to the FP64 sums once per sub-tile. The FP64
//    pipe bound the mixed loop (9 instructions of 16 cycles per SM per warp step, 165 cycles
//    measured); this one is bound by the integer multiply-adds, 78 cycles a warp step in a loop of
//    its own, 65 where all masses of the tile pair are equal. Attempts at N = 10002 61.1 -> 29.6 ms
//    (one force evaluation in them 0.84 -> 0.41 ms), at N = 2050 3.22 -> 1.88 ms.
//  - mixed, for the sub-tile pairs the integer window does not cover: a flat or very wide tile
//    pair, masses or coordinates outside its exponent range, or an unmasked pair closer than
//    2^-10 of the tile pair's extent (about 1 % of random sub-tile pairs of a Plummer sphere).
//    There the FP64 pipe issues the separation (3 DADD) and the two force accumulations (6
//    DFMA); r^2, 1/r, 1/r^3 and the mass products run on the integer pipe (pair_scalars_core), and
//    so does the force-function sum: m_j / r is a 64-bit product of significands added exactly
//    into a 128-bit fixed-point accumulator (UAcc). A system that is taken here throughout (a thin
//    disc, or 5 % of the bodies 10^3 core radii out) gains nothing: attempts 62.1 -> 63.6 ms at
//    N = 10002, 16.2 -> 16.8 at 5003, against the loop that knew only this arithmetic.
// A float pass over the sub-tile's pairs finds the closest pair, which decides, and bounds of the
// largest force on each body and the largest m_j / r, which set its accumulators' units. All are
// functions of the positions and masses alone, so results do not depend on timing.
//
// Tiles: the N bodies form NT tiles of T = 32*W. CTA (I, J), I <= J, owns the I-tile as
// "i" bodies (one per thread, accumulators in registers) and stages the J-tile ("j"
// bodies) in shared memory together with their accumulators, a copy per warp (added in warp
// order at the end: the warps, whose sub-tiles may take different arithmetics, need no barrier
// between sub-tiles). Each warp sweeps the W 32-wide sub-tiles in a rotated order; within a
// sub-tile, lane l pairs with j-slot (l + k) mod 32 at step k, so the 32 lanes update 32 distinct
// j accumulators at every step and no atomics are needed. On a diagonal tile only pairs i < j
// are visited. Near and padding pairs are masked by one bit per step (mask_word), from the
// near-pair words of the current tree.
//
// Determinism: CTA (I, J) writes its i-side sums into partial slot J of the i bodies and
// its j-side sums into slot I of the j bodies (a diagonal tile writes both into slot I).
// Every body thus receives exactly one write per slot, and the NT slots are added in a
// fixed order.
//
// Reduction on chip: every tile receives exactly NT contributions (CTAs (t, J >= t) and
// (I < t, t)). After writing its partials, a CTA counts itself in for its tiles; the CTA
// that brings a tile's count to NT adds that tile's NT slots (ascending) while they are
// still in L2, writes the 4 sums per body, resets the count and discards the partials'
// L2 lines, so that they are never written back to DRAM. Nothing waits: the last CTA to
// arrive finds everything it needs already written. The division slots of a launch run one
// after another (blockIdx.y), so a slot's last tiles are summed while later slots' CTAs
// compute. The trailing slots - those whose CTAs can still be resident together at the end
// of the launch, or all whose partials fit in L2 anyway - are left to the finishing pass,
// which reads their partials from L2 right after, so that no reduction trails the launch.
#include "device.cuh"
#include "internal.h"
#include "pairtile.cuh"

namespace mstar {
namespace {

// Sum of tile t's NT partial slots (ascending s, four at a time by pairs: a chain a quarter as long,
// in time and in roundings) for its T bodies, one per thread of the
// first T of the CTA's NTH threads, into Pt (4 planes); then its count is reset and the
// partials' lines dropped from L2. Every thread of the CTA calls it (it holds a barrier).
template <int T, int NTH = T>
__device__ __forceinline__ void finish_tile(int t, int npad, int NT, const double* Ps, double* Pt, int* cnt) {
  const int tid = threadIdx.x;
  if (NTH == T || tid < T) {
    const double* q = Ps + (size_t)t * T + tid;
    double ax = 0.0, ay = 0.0, az = 0.0, u = 0.0;
    // L2 loads (the slots were written by other CTAs after this SM's L1 could have seen
    // them), four slots at a time ahead of their additions
    int s = 0;
    for (; s + 4 <= NT; s += 4) {
      double b[4][4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const double* qs = q + (size_t)(s + k) * 4 * npad;
        b[k][0] = __ldcg(qs);
        b[k][1] = __ldcg(qs + npad);
        b[k][2] = __ldcg(qs + 2 * (size_t)npad);
        b[k][3] = __ldcg(qs + 3 * (size_t)npad);
      }
      ax += (b[0][0] + b[1][0]) + (b[2][0] + b[3][0]);
      ay += (b[0][1] + b[1][1]) + (b[2][1] + b[3][1]);
      az += (b[0][2] + b[1][2]) + (b[2][2] + b[3][2]);
      u += (b[0][3] + b[1][3]) + (b[2][3] + b[3][3]);
    }
    for (; s < NT; ++s) {
      const double* qs = q + (size_t)s * 4 * npad;
      ax += __ldcg(qs);
      ay += __ldcg(qs + npad);
      az += __ldcg(qs + 2 * (size_t)npad);
      u += __ldcg(qs + 3 * (size_t)npad);
    }
    double* o = Pt + (size_t)t * T + tid;
    o[0] = ax;
    o[(size_t)npad] = ay;
    o[2 * (size_t)npad] = az;
    o[3 * (size_t)npad] = u;
  }
  __syncthreads();  // every thread has read the tile's slots
  // the slots of tile t: NT x 4 runs of T doubles, each starting on a 256-byte boundary
  // (npad and t T are multiples of T >= 32); T / 16 lines of 128 bytes per run
  constexpr int kLinesPerRun = T / 16;
  for (int l = tid; l < NT * 4 * kLinesPerRun; l += NTH) {
    const int run = l / kLinesPerRun, line = l - run * kLinesPerRun;
    const double* a = Ps + (size_t)run * npad + (size_t)t * T + 16 * line;
    asm volatile("discard.global.L2 [%0], 128;" ::"l"(a) : "memory");
  }
  if (tid == 0) cnt[t] = 0;
}

// The near pairs of Sec. 3.4 (N_d <= 2) of the CTA's bodies, into Nb (4 planes: ax, ay, az and the
// sum of m/r over partners of higher index). They depend on the slot's edge vectors alone, so the
// pair launches take them in CTAs of their own ahead of the tile pairs, and the finishing pass adds
// them to the tile sums instead of walking the near partners itself.
//
// L lanes share a body's partners: a walk by one lane is a chain of up to some 25 partners (the
// largest counts in its warp), each an L2 access and a dependent 1/r^3, and bound the launches of
// small systems (N = 256: 14.8 us a launch, 8.2 with eight lanes and k_pair_tiles_ks' integers). Where
// the tile pairs fill the GPU the idle lanes' FP64 slots count instead: eight lanes cost 1 % of an
// attempt at N = 5003.
template <int S>
constexpr int kNearLanes = S > 1 ? 8 : 1;
template <int L>
__device__ __forceinline__ void near_block(int n, int npad, int slot, int n_d, const double* __restrict__ m,
                                           const int* __restrict__ parent, const int* __restrict__ gp,
                                           const int* __restrict__ child_off, const int* __restrict__ child_idx,
                                           const double* __restrict__ sX, double* __restrict__ Nb) {
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  const int l = threadIdx.x & (L - 1);
  const unsigned group = ((1u << L) - 1) << (threadIdx.x & 31 & ~(L - 1));
  const int p = idx / L;
  if (p >= n) return;  // whole groups
  const double *Xx = sX + (size_t)slot * 3 * npad, *Xy = Xx + npad, *Xz = Xy + npad;
  const bool nd2 = n_d >= 2;
  const int pp = parent[p], g = nd2 ? gp[p] : -1, c0 = child_off[p], c1 = child_off[p + 1];
  const int b0 = nd2 && pp >= 0 ? child_off[pp] : 0, b1 = nd2 && pp >= 0 ? child_off[pp + 1] : 0;
  const double xp = Xx[p], yp = Xy[p], zp = Xz[p];
  NearAcc acc;
  // +x, -x or 0 (sign and keep masks): off the FP64 pipe
  auto pick = [](double x, unsigned long long sign, unsigned long long keep) {
    return __longlong_as_double((long long)(((unsigned long long)__double_as_longlong(x) ^ sign) & keep));
  };
  // parent, grandparent, children, siblings: the separation is the picked X_k plus -X_p or 0
  for (int t = l; t < 2 + (c1 - c0) + (b1 - b0); t += L) {
    int q, k;
    constexpr unsigned long long kSign = 1ull << 63;
    unsigned long long sign = 0ull, keep = ~0ull, keep_p = ~0ull;
    if (t < 2) {
      q = t == 0 ? pp : g;
      k = pp;
      sign = kSign;
      keep = t == 0 ? 0ull : ~0ull;
    } else if (t < 2 + (c1 - c0)) {
      q = k = child_idx[c0 + t - 2];
      keep_p = 0ull;
    } else {
      q = k = child_idx[b0 + t - 2 - (c1 - c0)];
      if (q == p) q = -1;
    }
    if (q >= 0)
      acc.add(p, q, pick(Xx[k], sign, keep) + pick(xp, kSign, keep_p), pick(Xy[k], sign, keep) + pick(yp, kSign, keep_p),
              pick(Xz[k], sign, keep) + pick(zp, kSign, keep_p), m[q]);
  }
  if (nd2) {
    // grandchildren, in the children's order: L children at a time
    for (int a = c0; a < c1; a += L) {
      const int c = a + l < c1 ? child_idx[a + l] : -1;
      const int o = c >= 0 ? child_off[c] : 0, cnt = c >= 0 ? child_off[c + 1] - o : 0;
      int inc = cnt;
#pragma unroll
      for (int d = 1; d < L; d <<= 1) {
        const int v = __shfl_up_sync(group, inc, d, L);
        inc += l >= d ? v : 0;
      }
      const int tot = __shfl_sync(group, inc, L - 1, L);
      for (int t0 = 0; t0 < tot; t0 += L) {
        const int t = t0 + l;
        int k = 0;  // the child holding grandchild t
#pragma unroll
        for (int d = 0; d < L - 1; ++d) k += __shfl_sync(group, inc, d, L) <= t;
        const int ck = __shfl_sync(group, c, k, L);
        const int at = __shfl_sync(group, o - (inc - cnt), k, L) + t;
        if (t < tot) {
          const int q = child_idx[at];
          acc.add(p, q, Xx[q] + Xx[ck], Xy[q] + Xy[ck], Xz[q] + Xz[ck], m[q]);
        }
      }
    }
  }
#pragma unroll
  for (int d = L / 2; d > 0; d >>= 1) {
    acc.ax += __shfl_xor_sync(group, acc.ax, d);
    acc.ay += __shfl_xor_sync(group, acc.ay, d);
    acc.az += __shfl_xor_sync(group, acc.az, d);
    acc.u += __shfl_xor_sync(group, acc.u, d);
  }
  double* o = Nb + (size_t)slot * 4 * npad + p;
  if constexpr (L >= 4) {
    if (l < 4) o[(size_t)l * npad] = l == 0 ? acc.ax : (l == 1 ? acc.ay : (l == 2 ? acc.az : acc.u));
  } else if (l == 0) {
    o[0] = acc.ax;
    o[(size_t)npad] = acc.ay;
    o[2 * (size_t)npad] = acc.az;
    o[3 * (size_t)npad] = acc.u;
  }
}

// 24 warps per SM (80 registers; with W > 1 some 100 bytes spilt outside the pair loops). With 16, 20,
// 24 and 28, attempts at N = 10002 (W = 4) took 30.8, 29.6, 29.8 and 29.2 ms, at N = 5003 (W = 1)
// 8.40, 7.89, 7.75 and 7.80.
template <int W>
__global__ void __launch_bounds__(32 * W, 24 / W)
k_pair_tiles(int n, int npad, int NT, int slot_lo, int n_d, const double* __restrict__ m,
             const unsigned* __restrict__ near_words, const int* __restrict__ parent, const int* __restrict__ gp,
             const double* __restrict__ sr,
             double* __restrict__ P, double* __restrict__ Pt, int* __restrict__ tcnt, int keep_from,
             const int* __restrict__ child_off, const int* __restrict__ child_idx, const double* __restrict__ sX,
             double* __restrict__ Nb, int nnear) {
  constexpr int T = 32 * W;
  // tile J: positions, masses, fixed-point and float copies; the partner sums, a copy per warp;
  // the integer sums and units of the sub-tile a warp is at
  __shared__ double sx[T], sy[T], sz[T], sax[W][T], say[W][T], saz[W][T];
  __shared__ long long sfx[T], sfy[T], sfz[T], sbx[T], sby[T], sbz[T];
  __shared__ unsigned long long smm[T];
  __shared__ int sme[T], scj[T];
  __shared__ float4 sf[T];
  __shared__ int sbox[W][8];

  const int slot = slot_lo + blockIdx.y;
  if ((int)blockIdx.x < nnear) {
    near_block<kNearLanes<1>>(n, npad, slot, n_d, m, parent, gp, child_off, child_idx, sX, Nb);
    return;
  }
  int I, J;
  tile_pair((int)blockIdx.x - nnear, NT, I, J);
  const double* rx = sr + (size_t)slot * 3 * npad;
  const double* ry = rx + npad;
  const double* rz = ry + npad;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int j0 = J * T;
  const int i = I * T + tid;
  const double pi3[3] = {rx[i], ry[i], rz[i]};
  const double pj3[3] = {rx[j0 + tid], ry[j0 + tid], rz[j0 + tid]};
  const double mi = m[i], mj = m[j0 + tid], m0 = m[I * T];
  const bool i_pad = i >= n;
  const bool diag = (I == J);
  bool eq;  // all masses of the tile pair are equal
  const FixWindow fw = tile_window<W>(pi3, pj3, mi, mj, i_pad, j0 + tid >= n, m0, sbox, &eq);
  sx[tid] = pj3[0];
  sy[tid] = pj3[1];
  sz[tid] = pj3[2];
  sfx[tid] = fix_of(pj3[0], fw.u);
  sfy[tid] = fix_of(pj3[1], fw.u);
  sfz[tid] = fix_of(pj3[2], fw.u);
  sf[tid] = make_float4(float_of(pj3[0]), float_of(pj3[1]), float_of(pj3[2]), sqrtf(float_of(mj)));
  const MassSplit msj = fix_mass(mj);
  smm[tid] = msj.m;
  sme[tid] = msj.e;
#pragma unroll
  for (int w = 0; w < W; ++w) {
    sax[w][tid] = 0.0;
    say[w][tid] = 0.0;
    saz[w][tid] = 0.0;
  }
  TileBody body;
  body.set(pi3[0], pi3[1], pi3[2], mi, fw);
  __syncthreads();

#pragma unroll 1
  for (int s = 0; s < W; ++s) {
    const int sub = (warp + s) & (W - 1);
    const bool self = diag && sub == warp;
    if (diag && sub < warp) continue;
    const int js = sub * 32, wo = warp * 32;
    const unsigned mw = mask_word(near_words ? near_words + (size_t)(J * W + sub) * npad + i : nullptr, i_pad,
                                  n - j0 - js, self, lane);
    const SubTile t{sx + js,  sy + js,  sz + js,       sfx + js,      sfy + js,      sfz + js, smm + js, sme + js,
                    sf + js,  nullptr, &sax[warp][js], &say[warp][js], &saz[warp][js], sbx + wo,      sby + wo, sbz + wo, scj + wo};
    subtile_pairs<Fallback::mixed, 8, 2>(body, t, fw, eq, m0, mw, self ? 1 : 0, self ? 17 : 32, lane,
                                         [&] { return BodyPos{load_again(rx + i), load_again(ry + i), load_again(rz + i), 0.0}; });
  }
  __syncthreads();
  // the warps' partner sums, in warp order
  double jx = sax[0][tid], jy = say[0][tid], jz = saz[0][tid];
#pragma unroll
  for (int w = 1; w < W; ++w) {
    jx += sax[w][tid];
    jy += say[w][tid];
    jz += saz[w][tid];
  }

  const double axi = body.ax, ayi = body.ay, azi = body.az, ui = body.u_sum();
  double* Ps = P + (size_t)slot * NT * 4 * npad;
  if (diag) {
    double* q = Ps + (size_t)I * 4 * npad + i;
    q[0] = axi - jx;
    q[(size_t)npad] = ayi - jy;
    q[2 * (size_t)npad] = azi - jz;
    q[3 * (size_t)npad] = ui;
  } else {
    double* q = Ps + (size_t)J * 4 * npad + i;
    q[0] = axi;
    q[(size_t)npad] = ayi;
    q[2 * (size_t)npad] = azi;
    q[3 * (size_t)npad] = ui;
    double* qj = Ps + (size_t)I * 4 * npad + j0 + tid;
    qj[0] = -jx;
    qj[(size_t)npad] = -jy;
    qj[2 * (size_t)npad] = -jz;
    qj[3 * (size_t)npad] = 0.0;
  }

  // count this CTA in for tiles I and J; the last of a tile's NT contributors sums it (the
  // trailing slots from keep_from on are summed by the finishing pass)
  if ((int)blockIdx.y >= keep_from) return;
  __shared__ int s_last[2];
  __threadfence();  // this CTA's partials are visible device-wide before it is counted
  __syncthreads();
  if (tid == 0) {
    int* cnt = tcnt + (size_t)slot * NT;
    s_last[0] = atomicAdd(&cnt[I], 1) == NT - 1;
    s_last[1] = diag ? 0 : atomicAdd(&cnt[J], 1) == NT - 1;
    __threadfence();  // the counts seen before the other contributors' partials are read
  }
  __syncthreads();
  if (s_last[0] | s_last[1]) {
    int* cnt = tcnt + (size_t)slot * NT;
    double* Pts = Pt + (size_t)slot * 4 * npad;
    if (s_last[0]) finish_tile<T>(I, npad, NT, Ps, Pts, cnt);
    if (s_last[1]) {
      __syncthreads();
      finish_tile<T>(J, npad, NT, Ps, Pts, cnt);
    }
  }
}

// The pair loop of small systems: the 32-body tiles and the arithmetic of k_pair_tiles<1>, with the
// 32 partner steps of a tile pair split over S warps (S divides 16). Warp w takes steps
// [32 w / S, 32 (w + 1) / S) of an off-diagonal pair and [1 + 16 w / S, 1 + 16 (w + 1) / S) of a
// diagonal one, keeping its own i-side and partner sums; the S copies are added in warp order at the
// end. At N ~ 10^2 to 10^3 a tile pair's 32 dependent steps in one warp bind the launch; S warps
// shorten them S-fold. What does not shrink is done once, by warp 0 (conversions and window), or
// binds larger S (a warp's flush to FP64: 14 FP64 instructions). Attempts with S = 1, 2, 4, 8:
// 0.67, 0.58, 0.54, 0.56 ms at N = 256, 0.78, 0.71, 0.68, 0.74 at 512.
template <int S>
__global__ void __launch_bounds__(32 * S, 24 / S)
k_pair_tiles_ks(int n, int npad, int NT, int slot_lo, int n_d, const double* __restrict__ m,
                const int* __restrict__ parent, const int* __restrict__ gp, const double* __restrict__ sr,
                double* __restrict__ P, double* __restrict__ Pt, int* __restrict__ tcnt, int keep_from,
                const int* __restrict__ child_off, const int* __restrict__ child_idx,
                const double* __restrict__ sX, double* __restrict__ Nb, int nnear) {
  constexpr int T = 32;
  __shared__ double sx[T], sy[T], sz[T];
  __shared__ long long sfx[T], sfy[T], sfz[T];
  __shared__ unsigned long long smm[T];
  __shared__ int sme[T], scj[S][T], sp[T], sg[T];
  __shared__ float4 sf[T];
  __shared__ TilePos sbody[T];
  __shared__ FixWindow sfw;
  __shared__ bool seq;
  __shared__ double sj3[S][3][T];  // partner sums per warp
  __shared__ double si4[S][4][T];  // integer sums of the partners, then the i-side sums per warp
  const int slot = slot_lo + blockIdx.y;
  if ((int)blockIdx.x < nnear) {
    near_block<kNearLanes<S>>(n, npad, slot, n_d, m, parent, gp, child_off, child_idx, sX, Nb);
    return;
  }
  int I, J;
  tile_pair((int)blockIdx.x - nnear, NT, I, J);
  const double* rx = sr + (size_t)slot * 3 * npad;
  const double* ry = rx + npad;
  const double* rz = ry + npad;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int j0 = J * T, i = I * T + lane, j = j0 + lane;
  const bool i_pad = i >= n, diag = I == J;
  const int pi = parent[i], gpi = gp[i];
  const double m0 = m[I * T];
  if (warp == 0) {  // the conversions once: FP64 pipe
    const double pi3[3] = {rx[i], ry[i], rz[i]};
    const double pj3[3] = {rx[j], ry[j], rz[j]};
    const double mi = m[i], mj = m[j];
    bool eq;
    const FixWindow fw = tile_window<1>(pi3, pj3, mi, mj, i_pad, j >= n, m0, nullptr, &eq);
    sx[lane] = pj3[0];
    sy[lane] = pj3[1];
    sz[lane] = pj3[2];
    sfx[lane] = fix_of(pj3[0], fw.u);
    sfy[lane] = fix_of(pj3[1], fw.u);
    sfz[lane] = fix_of(pj3[2], fw.u);
    sf[lane] = make_float4(float_of(pj3[0]), float_of(pj3[1]), float_of(pj3[2]), sqrtf(float_of(mj)));
    const MassSplit ms = fix_mass(mj);
    smm[lane] = ms.m;
    sme[lane] = ms.e;
    sp[lane] = parent[j];
    sg[lane] = gp[j];
    TilePos b;
    b.set(pi3[0], pi3[1], pi3[2], mi, fw);
    sbody[lane] = b;
    if (lane == 0) {
      sfw = fw;
      seq = eq;
    }
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) sj3[warp][c][lane] = 0.0;
  __syncthreads();
  TileBody body;
  static_cast<TilePos&>(body) = sbody[lane];
  const FixWindow fw = sfw;
  const bool eq = seq;
  {
    long long* sb = reinterpret_cast<long long*>(&si4[warp][0][0]);
    const SubTile t{sx,           sy,           sz,           sfx, sfy,    sfz,    smm,      sme, sf, nullptr,
                    sj3[warp][0], sj3[warp][1], sj3[warp][2], sb,  sb + 32, sb + 64, scj[warp]};
    const int k0 = diag ? 1 + 16 * warp / S : 32 * warp / S, k1 = k0 + (diag ? 16 : 32) / S;
    // the near pairs of the warp's few steps, here (a pass of its own over the tree would cost
    // small systems a launch)
    unsigned mw = mask_word(nullptr, i_pad, n - j0, diag, lane);
    if (n_d >= 1)
      for (int k = k0; k < k1; ++k) {
        const int q = (lane + k) & 31, jq = j0 + q, pj = sp[q];
        bool near = (pi == jq) | (pj == i);
        near |= (n_d >= 2) & ((gpi == jq) | (sg[q] == i) | (pi == pj));
        mw |= near ? 1u << k : 0u;
      }
    subtile_pairs<Fallback::mixed, S == 2 ? 8 : 16 / S, 2>(body, t, fw, eq, m0, mw, k0, k1, lane, [&] {
      return BodyPos{load_again(rx + i), load_again(ry + i), load_again(rz + i), 0.0};
    });
  }
  __syncwarp();
  si4[warp][0][lane] = body.ax;
  si4[warp][1][lane] = body.ay;
  si4[warp][2][lane] = body.az;
  si4[warp][3][lane] = body.u_sum();
  __syncthreads();
  // warp c (round robin) adds component c of the S copies
  double* Ps = P + (size_t)slot * NT * 4 * npad;
  for (int c = warp; c < 4; c += S) {
    double a = si4[0][c][lane], jv = c < 3 ? sj3[0][c][lane] : 0.0;
#pragma unroll
    for (int w = 1; w < S; ++w) {
      a += si4[w][c][lane];
      if (c < 3) jv += sj3[w][c][lane];
    }
    if (diag) {
      Ps[(size_t)I * 4 * npad + (size_t)c * npad + i] = a - jv;
    } else {
      Ps[(size_t)J * 4 * npad + (size_t)c * npad + i] = a;
      Ps[(size_t)I * 4 * npad + (size_t)c * npad + j] = -jv;
    }
  }
  // the on-chip reduction of k_pair_tiles (the first 32 threads sum a tile)
  if ((int)blockIdx.y >= keep_from) return;
  __shared__ int s_last[2];
  __threadfence();
  __syncthreads();
  if (tid == 0) {
    int* cnt = tcnt + (size_t)slot * NT;
    s_last[0] = atomicAdd(&cnt[I], 1) == NT - 1;
    s_last[1] = diag ? 0 : atomicAdd(&cnt[J], 1) == NT - 1;
    __threadfence();
  }
  __syncthreads();
  if (s_last[0] | s_last[1]) {
    int* cnt = tcnt + (size_t)slot * NT;
    double* Pts = Pt + (size_t)slot * 4 * npad;
    if (s_last[0]) finish_tile<T, 32 * S>(I, npad, NT, Ps, Pts, cnt);
    if (s_last[1]) {
      __syncthreads();
      finish_tile<T, 32 * S>(J, npad, NT, Ps, Pts, cnt);
    }
  }
}

// The tile sums plus the near pairs of Sec. 3.4 (N_d <= 2: parent, child, grandparent,
// grandchild, sibling), times G. Writes a (3 planes) and per-block sums of m_p * u_p, where
// u_p sums m_q / r_pq over partners q > p (each unordered pair once). The trailing slots
// (blockIdx.y >= keep_from) sum their NT partial slots here (ascending, as the tile kernel does
// for the other slots).
//
// A CTA takes kBlock bodies with kFinishPlanes threads each: thread (c, b) sums plane c (ax, ay,
// az, u) of body b over the slots, so the four sums run side by side (each in the same order
// as one thread summing all four), and the first kBlock threads finish the bodies. Where the
// pass runs beside pair launches of other divisions, which keep the FP64 pipe busy, its share
// of the pipe grows with its warps.
constexpr int kFinishPlanes = 4;
__global__ void __launch_bounds__(kBlock * kFinishPlanes)
k_pair_finish(int n, int npad, int NT, int slot_lo, int n_d, double G, const double* __restrict__ m,
              const double* __restrict__ Nb, const double* __restrict__ P, const double* __restrict__ Pt,
              double* __restrict__ sa, double* __restrict__ Ublk, int nblk, int keep_from) {
  __shared__ double scratch[32];
  __shared__ double splane[kFinishPlanes][kBlock];
  const int slot = slot_lo + blockIdx.y;
  const int plane = threadIdx.x / kBlock, b = threadIdx.x - plane * kBlock;
  const int p = blockIdx.x * kBlock + b;
  const bool deferred = (int)blockIdx.y >= keep_from;
  if (deferred) {
    double acc = 0.0;
    if (p < n) {
      const double* q = P + (size_t)slot * NT * 4 * npad + (size_t)plane * npad + p;
      int s = 0;
      for (; s + 4 <= NT; s += 4) {
        double t[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) t[k] = q[(size_t)(s + k) * 4 * npad];
        acc += (t[0] + t[1]) + (t[2] + t[3]);
      }
      for (; s < NT; ++s) acc += q[(size_t)s * 4 * npad];
    }
    splane[plane][b] = acc;
    // the block's bodies' partials are read: drop their L2 lines, so that they are not
    // written back to DRAM when later launches' partials evict them (every slot is written
    // again before it is next read). NT x 4 runs of kBlock doubles, each starting on a
    // 512-byte boundary; a line is dropped only where it lies below npad.
    __syncthreads();
    constexpr int kLinesPerRun = kBlock / 16;
    const int b0 = blockIdx.x * kBlock;
    const double* base = P + (size_t)slot * NT * 4 * npad + b0;
    for (int l = threadIdx.x; l < NT * 4 * kLinesPerRun; l += blockDim.x) {
      const int run = l / kLinesPerRun, line = l - run * kLinesPerRun;
      if (b0 + 16 * line < npad) {
        const double* a = base + (size_t)run * npad + 16 * line;
        asm volatile("discard.global.L2 [%0], 128;" ::"l"(a) : "memory");
      }
    }
  }
  double um = 0.0;
  if (plane == 0 && p < n) {
    NearAcc acc;
    if (deferred) {
      acc.ax = splane[0][b];
      acc.ay = splane[1][b];
      acc.az = splane[2][b];
      acc.u = splane[3][b];
    } else {
      const double* q = Pt + (size_t)slot * 4 * npad + p;
      acc.ax = q[0];
      acc.ay = q[(size_t)npad];
      acc.az = q[2 * (size_t)npad];
      acc.u = q[3 * (size_t)npad];
    }
    if (n_d >= 1) {  // the near pairs, from the pair launch's near CTAs
      const double* nb = Nb + (size_t)slot * 4 * npad + p;
      acc.ax += nb[0];
      acc.ay += nb[(size_t)npad];
      acc.az += nb[2 * (size_t)npad];
      acc.u += nb[3 * (size_t)npad];
    }
    double* a = sa + (size_t)slot * 3 * npad + p;
    a[0] = G * acc.ax;
    a[(size_t)npad] = G * acc.ay;
    a[2 * (size_t)npad] = G * acc.az;
    um = m[p] * acc.u;
  }
  // the other planes' threads add zeros after the first kBlock threads' sum, so the block sum
  // is that of the kBlock bodies alone
  const double s = block_sum(um, scratch);
  if (threadIdx.x == 0) Ublk[(size_t)slot * nblk + blockIdx.x] = G * s;
}

// Partial bytes that the trailing slots of a launch may leave in L2 for the finishing pass.
constexpr double kDeferL2Bytes = 48.0 * 1024 * 1024;

// Trailing slots of a launch left to the finishing pass: the slots whose CTAs can be resident
// together at the end of the launch (plus one), and at least as many as fit in the L2 budget.
template <typename K>
int defer_slots(const mstar_ctx* c, K kernel, int threads) {
  int per_sm = 0, sms = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, 0) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device) != cudaSuccess) {
    cudaGetLastError();
    return 1 << 20;  // unknown: every slot is summed by the finishing pass
  }
  const long long resident = (long long)per_sm * sms;
  const int d_wave = (int)((resident + c->ntp - 1) / c->ntp) + 1;
  const double slot_bytes = (double)c->NT * 4.0 * c->npad * sizeof(double);
  const int d_l2 = (int)(kDeferL2Bytes / slot_bytes);
  return d_wave > d_l2 ? d_wave : d_l2;
}

template <int W, int S>
cudaError_t run_tiles(mstar_ctx* c, int slot_lo, int nsl, int n_d, int keep_from) {
  constexpr int threads = S == 1 ? 32 * W : 32 * S;
  const int nnear = n_d >= 1 ? (c->n * kNearLanes<S> + threads - 1) / threads : 0;  // the near CTAs come first
  dim3 grid(nnear + c->ntp, nsl);
  if (c->prof) prof_begin(c);
  if constexpr (S == 1)
    k_pair_tiles<W><<<grid, 32 * W, 0, c->stream>>>(c->n, c->npad, c->NT, slot_lo, n_d, c->d.m,
                                                    n_d >= 1 ? c->d.near_words : nullptr, c->d.parent, c->d.gp,
                                                    c->d.sr, c->d.P, c->d.Pt, c->d.tcnt, keep_from, c->d.child_off,
                                                    c->d.child_idx, c->d.sX, c->d.Nb, nnear);
  else
    k_pair_tiles_ks<S><<<grid, 32 * S, 0, c->stream>>>(c->n, c->npad, c->NT, slot_lo, n_d, c->d.m, c->d.parent,
                                                       c->d.gp, c->d.sr, c->d.P, c->d.Pt, c->d.tcnt, keep_from,
                                                       c->d.child_off, c->d.child_idx, c->d.sX, c->d.Nb, nnear);
  MSTAR_LAUNCHED(c);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  if (c->prof) prof_end(c, nsl);
  return cudaSuccess;
}

}  // namespace

// The pair launches run beside the small kernels of other divisions (a stream per division),
// several of which take tens of KB of shared memory (the staged rebuild). An SM runs CTAs of
// kernels together only under one split of its on-chip memory between L1 and shared memory, so
// every kernel of an attempt asks for the largest shared-memory share: the small kernels' CTAs
// can then start on SMs that hold pair CTAs (GBS steps at N = 2050 2.4 % faster). A hint: a
// device that ignores it loses nothing else.
void prefer_shared_pair_kernels() {
  cudaFuncSetAttribute(k_pair_tiles<1>, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
  cudaFuncSetAttribute(k_pair_tiles<2>, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
  cudaFuncSetAttribute(k_pair_tiles<4>, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
  cudaFuncSetAttribute(k_pair_tiles_ks<2>, cudaFuncAttributePreferredSharedMemoryCarveout,
                       cudaSharedmemCarveoutMaxShared);
  cudaFuncSetAttribute(k_pair_tiles_ks<4>, cudaFuncAttributePreferredSharedMemoryCarveout,
                       cudaSharedmemCarveoutMaxShared);
  cudaFuncSetAttribute(k_pair_tiles_ks<8>, cudaFuncAttributePreferredSharedMemoryCarveout,
                       cudaSharedmemCarveoutMaxShared);
  cudaFuncSetAttribute(k_pair_finish, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
  cudaGetLastError();
}

// Bit s & 31 of word (s >> 5, p): bodies p and s are near (at most n_d tree edges apart), for the
// tiled pair loop's masks. One thread per body walks its own near partners; the words were cleared.
// (atomicOr, although no two threads meet in a word: without a result to wait for, 10 -> 6 us.)
__global__ void __launch_bounds__(kBlock)
k_near_words(int n, int npad, int n_d, const int* __restrict__ parent, const int* __restrict__ gp,
             const int* __restrict__ child_off, const int* __restrict__ child_idx, unsigned* __restrict__ words) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n) return;
  auto put = [&](int q) { atomicOr(&words[(size_t)(q >> 5) * npad + p], 1u << (q & 31)); };
  const int pp = parent[p];
  if (pp >= 0) put(pp);
  const int c0 = child_off[p], c1 = child_off[p + 1];
  for (int a = c0; a < c1; ++a) put(child_idx[a]);
  if (n_d < 2) return;
  if (gp[p] >= 0) put(gp[p]);
  for (int a = c0; a < c1; ++a) {
    const int ch = child_idx[a];
    for (int b = child_off[ch]; b < child_off[ch + 1]; ++b) put(child_idx[b]);
  }
  if (pp >= 0)
    for (int b = child_off[pp]; b < child_off[pp + 1]; ++b)
      if (child_idx[b] != p) put(child_idx[b]);
}

cudaError_t launch_near_words(mstar_ctx* c) {
  if (!c->d.near_words || c->p.n_d < 1) return cudaSuccess;
  cudaError_t e = cudaMemsetAsync(c->d.near_words, 0, sizeof(unsigned) * (size_t)(c->npad / 32) * c->npad, c->stream);
  if (e != cudaSuccess) return e;
  k_near_words<<<(c->n + kBlock - 1) / kBlock, kBlock, 0, c->stream>>>(c->n, c->npad, c->p.n_d, c->d.parent, c->d.gp,
                                                                       c->d.child_off, c->d.child_idx,
                                                                       c->d.near_words);
  MSTAR_LAUNCHED(c);
  return cudaGetLastError();
}

cudaError_t launch_forces(mstar_ctx* c, int slot_lo, int slot_hi, int n_d) {
  const int nsl = slot_hi - slot_lo;
  if (nsl <= 0) return cudaSuccess;
  if (c->pair_defer < 0) {
    if (c->W == 1) {
      switch (c->S) {
        case 2: c->pair_defer = defer_slots(c, k_pair_tiles_ks<2>, 64); break;
        case 4: c->pair_defer = defer_slots(c, k_pair_tiles_ks<4>, 128); break;
        case 8: c->pair_defer = defer_slots(c, k_pair_tiles_ks<8>, 256); break;
        default: c->pair_defer = defer_slots(c, k_pair_tiles<1>, 32); break;
      }
    } else {
      c->pair_defer = c->W == 2 ? defer_slots(c, k_pair_tiles<2>, 64) : defer_slots(c, k_pair_tiles<4>, 128);
    }
  }
  const int keep_from = nsl - c->pair_defer;  // slots below this index are summed on chip
  cudaError_t e;
  if (c->W == 1) {
    switch (c->S) {
      case 2: e = run_tiles<1, 2>(c, slot_lo, nsl, n_d, keep_from); break;
      case 4: e = run_tiles<1, 4>(c, slot_lo, nsl, n_d, keep_from); break;
      case 8: e = run_tiles<1, 8>(c, slot_lo, nsl, n_d, keep_from); break;
      default: e = run_tiles<1, 1>(c, slot_lo, nsl, n_d, keep_from); break;
    }
  } else {
    e = c->W == 2 ? run_tiles<2, 1>(c, slot_lo, nsl, n_d, keep_from) : run_tiles<4, 1>(c, slot_lo, nsl, n_d, keep_from);
  }
  if (e != cudaSuccess) return e;
  dim3 grid(c->nblk, nsl);
  k_pair_finish<<<grid, kBlock * kFinishPlanes, 0, c->stream>>>(c->n, c->npad, c->NT, slot_lo, n_d, c->p.G,
                                                                c->d.m, c->d.Nb, c->d.P, c->d.Pt, c->d.sa,
                                                                c->d.Ublk, c->nblk, keep_from);
  MSTAR_LAUNCHED(c);
  c->force_evals += nsl;
  return cudaGetLastError();
}

}  // namespace mstar
