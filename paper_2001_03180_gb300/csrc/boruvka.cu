// Exact MST for the GBS step by Boruvka rounds over the whole GPU.
//
// Sec. 3.2 builds the MST with Prim's algorithm; its N sequential iterations keep a GPU on
// one SM. When all squared distances that decide the tree are distinct, the MST is unique
// (Sec. 3.1), so any exact MST algorithm yields Prim's tree. Boruvka's rounds are
// parallel: every vertex finds its nearest vertex outside its component (exact FP64
// comparisons, filtered by rigorous float lower bounds), every component takes its
// cheapest outgoing edge, and components merge along those edges. If two different
// candidates ever compare exactly equal in FP64, the tree could depend on tie-breaking
// rules, and the caller falls back to the Prim kernel, which applies the paper's rule.
// The tree is then oriented from Prim's root (the body closest to the centre of mass), which gives
// the same parent and level as Prim's indexing.
//
// Distances are computed exactly as the CPU definition does: ((dx*dx)+(dy*dy))+(dz*dz)
// with dx = x_u - x_v, each operation rounded separately.
#include <climits>
#include <cstring>

#include "device.cuh"
#include "internal.h"
#include "nearest.cuh"

namespace mstar {
namespace {

constexpr int kBT = 128;  // vertices per CTA in the nearest-foreign-neighbour search

__device__ __forceinline__ double d2_exact(const double* X, const double* Y, const double* Z, int u, int v) {
  const double dx = __dsub_rn(X[u], X[v]), dy = __dsub_rn(Y[u], Y[v]), dz = __dsub_rn(Z[u], Z[v]);
  return __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
}

// Nearest foreign neighbour (smallest exact squared distance to a vertex of another
// component) of every vertex whose cached neighbour is missing or has become internal;
// CTA (tile, part) scans the part-th slice of the candidates. Writes per (vertex, part)
// the exact distance bits and the neighbour; exact equal distances to two different
// candidates at the minimum set *tie. One float pass and one exact distance per vertex
// (NearestScan), where two float passes with upper and lower bounds of 22 instructions a candidate
// each took 17, 17, 52 and 193 us per round at N = 601, 2050, 5003 and 10002; 6, 7, 20 and 70 now.
__global__ void __launch_bounds__(kBT)
k_nfn(int n, int npad, int nparts, const double* __restrict__ X, const double* __restrict__ Y,
      const double* __restrict__ Z, const float* __restrict__ f4, const int* __restrict__ comp,
      const int* __restrict__ nbr, unsigned long long* __restrict__ partD, int* __restrict__ partJ,
      int* __restrict__ flags) {
  // The round's gate: flags[4] = 1 once the tree is complete (flags[1] = n - 1 edges) or a tie has
  // been seen (flags[0]), decided by the last kernel of the previous round; the round's kernels then
  // return at once, and flags[3] counts the rounds that ran. Rounds can thus be issued ahead of
  // the host's check: a round after the last one needed changes nothing (without the gate it
  // would find no foreign neighbour and report a tie). No kernel of the round writes flags[4]
  // before k_relabel, so every CTA of the search decides alike: a tie found while it runs ends the
  // build after this round, whose other kernels still get a neighbour for every vertex. The search's
  // first CTA copies the gate to flags[2] for them.
  const bool stop = flags[4] != 0;
  if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) {
    flags[2] = stop;
    if (!stop) flags[3] += 1;
  }
  if (stop) return;
  int* tie = flags;
  __shared__ float4 sq[kBT];  // x, y, z and the component's bits
  __shared__ int any, s_emax;
  const int i = blockIdx.x * kBT + threadIdx.x;
  const int part = blockIdx.y;
  bool need = false;
  int ci = -1;
  if (i < n) {
    ci = comp[i];
    const int b = nbr[i];
    need = (b < 0) || (comp[b] == ci);
  }
  if (threadIdx.x == 0) {
    any = 0;
    s_emax = 0;
  }
  __syncthreads();
  if (need) any = 1;
  __syncthreads();
  if (!any) return;
  const float4* f = reinterpret_cast<const float4*>(f4);
  const float4 fi = i < n ? f[i] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  const int per = (n + nparts - 1) / nparts;
  const int j_lo = part * per, j_hi = min(n, j_lo + per);
  NearestScan ns;
  ns.clear();
  for (int t0 = j_lo; t0 < j_hi; t0 += kBT) {
    __syncthreads();
    const int j = t0 + threadIdx.x;
    float4 q = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if (j < j_hi) {
      q = f[j];
      sq[threadIdx.x] = make_float4(q.x, q.y, q.z, __int_as_float(comp[j]));
    }
    const int e = __reduce_max_sync(0xffffffffu, __float_as_int(q.w));  // non-negative floats
    if ((threadIdx.x & 31) == 0) atomicMax(&s_emax, e);
    __syncthreads();
    if (!need) continue;
    const int cnt = min(kBT, j_hi - t0);
#pragma unroll 4
    for (int k = 0; k < cnt; ++k) {
      const float4 c = sq[k];
      ns.add(fi.x - c.x, fi.y - c.y, fi.z - c.z, __float_as_int(c.w) != ci, t0 + k);
    }
  }
  __syncthreads();
  const float emax = fi.w + __int_as_float(s_emax);
  unsigned long long bD = ~0ull;
  int bj = -1;
  int mytie = 0;
  const bool found = need && !ns.none();  // (a slice may hold no vertex of another component)
  const bool sure = !found || ns.certain(emax);
  if (found && sure) {
    bj = ns.j1;
    bD = key_bits(d2_exact(X, Y, Z, i, bj));
  }
  // the undecided vertices of the warp, one at a time over its 32 lanes
  const int lane = threadIdx.x & 31;
  for (unsigned todo = __ballot_sync(0xffffffffu, !sure); todo; todo &= todo - 1) {
    const int l = __ffs(todo) - 1;
    const int vi = __shfl_sync(0xffffffffu, i, l), vc = __shfl_sync(0xffffffffu, ci, l);
    const float lim = __shfl_sync(0xffffffffu, ns.limit(emax), l);
    const float vx = __shfl_sync(0xffffffffu, fi.x, l), vy = __shfl_sync(0xffffffffu, fi.y, l),
                vz = __shfl_sync(0xffffffffu, fi.z, l);
    unsigned long long d = ~0ull;
    int dj = -1, tied = 0;
    for (int jj = j_lo + lane; jj < j_hi; jj += 32) {
      if (comp[jj] == vc) continue;
      const float4 c = f[jj];
      const float dx = vx - c.x, dy = vy - c.y, dz = vz - c.z;
      if (fmaf(dz, dz, fmaf(dy, dy, dx * dx)) > lim) continue;
      const unsigned long long db = key_bits(d2_exact(X, Y, Z, vi, jj));
      if (db < d) {
        d = db;
        dj = jj;
        tied = 0;
      } else if (db == d) {
        tied = 1;
      }
    }
    const unsigned mh = __reduce_min_sync(0xffffffffu, (unsigned)(d >> 32));
    const unsigned ml = __reduce_min_sync(0xffffffffu, (unsigned)(d >> 32) == mh ? (unsigned)d : ~0u);
    const unsigned long long dm = ((unsigned long long)mh << 32) | ml;
    const unsigned at = __ballot_sync(0xffffffffu, d == dm && dj >= 0);
    const unsigned tb = __ballot_sync(0xffffffffu, d == dm && tied != 0);
    const int j0 = __shfl_sync(0xffffffffu, dj, at ? __ffs(at) - 1 : 0);
    if (lane == l && at) {
      bD = dm;
      bj = j0;
      mytie = tb != 0 || (at & (at - 1)) != 0;
    }
  }
  if (!need) return;
  partD[(size_t)part * npad + i] = bD;
  partJ[(size_t)part * npad + i] = bj;
  if (mytie) atomicOr(tie, 1);
}

// Merge the parts: exact minimum, ties flagged; cache the neighbour.
__global__ void k_nfn_merge(int n, int npad, int nparts, const int* __restrict__ comp, int* __restrict__ nbr,
                            unsigned long long* __restrict__ nbrD, const unsigned long long* __restrict__ partD,
                            const int* __restrict__ partJ, int* __restrict__ tie, const int* __restrict__ stop) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n || *stop) return;
  const int b = nbr[i];
  if (b >= 0 && comp[b] != comp[i]) return;
  unsigned long long bD = ~0ull;
  int bj = -1;
  // the parts in ascending order, their values loaded four at a time ahead of the comparisons
  for (int p0 = 0; p0 < nparts; p0 += 4) {
    unsigned long long d[4];
    int j[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const bool in = p0 + k < nparts;
      d[k] = in ? partD[(size_t)(p0 + k) * npad + i] : ~0ull;
      j[k] = in ? partJ[(size_t)(p0 + k) * npad + i] : -1;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (j[k] < 0) continue;
      if (d[k] < bD) {
        bD = d[k];
        bj = j[k];
      } else if (d[k] == bD && j[k] != bj) {
        atomicOr(tie, 1);
      }
    }
  }
  nbr[i] = bj;
  nbrD[i] = bD;
}

__global__ void k_comp_min(int n, const int* __restrict__ comp, const unsigned long long* __restrict__ nbrD,
                           unsigned long long* __restrict__ cmin, const int* __restrict__ stop) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n && !*stop) atomicMin(&cmin[comp[i]], nbrD[i]);
}

__global__ void k_comp_edge(int n, const int* __restrict__ comp, const unsigned long long* __restrict__ nbrD,
                            const unsigned long long* __restrict__ cmin, int* __restrict__ cidx,
                            int* __restrict__ ccnt, int* __restrict__ tie, const int* __restrict__ stop) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n || *stop) return;
  const int c = comp[i];
  if (nbrD[i] == cmin[c]) {
    if (atomicAdd(&ccnt[c], 1) > 0) atomicOr(tie, 1);  // two cheapest edges of equal weight
    cidx[c] = i;
  }
}

// Hook every component onto the component at the far end of its cheapest edge. Two
// components that chose each other chose the same edge (weights distinct); the smaller
// label becomes the root and records the edge once.
__global__ void k_hook(int n, const int* __restrict__ comp, const int* __restrict__ nbr, const int* __restrict__ cidx,
                       int* __restrict__ nxt, int* __restrict__ eu, int* __restrict__ ev, int* __restrict__ ecount,
                       const int* __restrict__ stop) {
  const int C = blockIdx.x * blockDim.x + threadIdx.x;
  if (C >= n || *stop || comp[C] != C) return;
  const int i = cidx[C];
  const int j = nbr[i];
  const int T = comp[j];
  const int jT = nbr[cidx[T]];
  const bool mutual = comp[jT] == C;
  if (mutual && C < T) {
    nxt[C] = C;
  } else {
    nxt[C] = T;
  }
  if (!mutual || C < T) {
    const int e = atomicAdd(ecount, 1);
    if (e < n - 1) {
      eu[e] = i;
      ev[e] = j;
    }
  }
}

// The new labels, and the next round's gate.
__global__ void k_relabel(int n, int* __restrict__ comp, const int* __restrict__ nxt,
                          unsigned long long* __restrict__ cmin, int* __restrict__ ccnt, int* __restrict__ flags) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n || flags[2]) return;
  if (i == 0) flags[4] = flags[0] != 0 || flags[1] >= n - 1;
  int c = comp[i];
  for (int guard = 0; guard < n && nxt[c] != c; ++guard) c = nxt[c];
  comp[i] = c;
  cmin[i] = ~0ull;
  ccnt[i] = 0;
}

__global__ void k_boruvka_init(int n, const double* __restrict__ X, const double* __restrict__ Y,
                               const double* __restrict__ Z, float* __restrict__ f4, int* __restrict__ comp,
                               int* __restrict__ nbr, unsigned long long* __restrict__ cmin, int* __restrict__ ccnt) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float x = __double2float_rn(X[i]), y = __double2float_rn(Y[i]), z = __double2float_rn(Z[i]);
  f4[4 * i] = x;
  f4[4 * i + 1] = y;
  f4[4 * i + 2] = z;
  f4[4 * i + 3] = fmaxf(fabsf(x), fmaxf(fabsf(y), fabsf(z))) * 0x1p-23f + 1e-37f;
  comp[i] = i;
  nbr[i] = -1;
  cmin[i] = ~0ull;
  ccnt[i] = 0;
}

// |x| within [lo, hi] as floats, from the bits of a double (integer operations: a conversion costs
// an FP64 issue slot). hi is +inf from 2^127 on (and for NaN), lo is 0 below 2^-126.
__device__ __forceinline__ void abs_bounds(double x, float& lo, float& hi) {
  const int h = __double2hiint(x) & 0x7fffffff;
  const int e = (h >> 20) - 1023;
  const float f = __int_as_float(((e + 127) << 23) | ((h & 0xfffff) << 3));  // truncated: f <= |x| < f (1 + 2^-19)
  lo = e < -126 ? 0.0f : (e > 126 ? 0x1p126f : f);
  hi = e < -126 ? 0x1p-125f : (e > 126 ? __int_as_float(0x7f800000) : f * (1.0f + 0x1p-18f));
}

// Orient the tree from Prim's root (the body closest to the origin, lowest index on ties): parent
// and level of every vertex from the edge list, in one CTA.
//
// Euler tour and list ranking, because a walk level by level is a chain as long as the tree is
// deep (59 levels at N = 2050, 150 at N = 10002: 57 and 220 us in one warp, which measured faster
// than block barriers between levels). Edge e gives the arcs 2e (eu -> ev) and 2e + 1 (ev -> eu);
// the arc after u -> v in the tour is the one after v -> u in v's circular adjacency list. Up to
// blockDim arcs are splitters: each thread walks from its splitter to the next one (about 20 arcs
// at N = 10002, in shared memory), the splitters are ranked by pointer doubling, and a second walk
// gives every arc its rank. An arc that precedes its twin leads away from the root, and the
// running sum of +1 (away) and -1 (back) along the tour is the level it reaches. Parent and level
// do not depend on the order of the adjacency lists, which the atomic fill leaves open. An edge list
// that is no spanning tree gives the star around the root: whatever the list holds, every vertex gets
// a parent and every walk up the tree ends.
// 20 n bytes of shared memory hold the arcs as 16-bit numbers (2 (n - 1) < 2^16).
// N = 601, 2050, 5003, 10002: 28, 57, 122 and 220 us before, 11, 18, 30 and 51 us now.
constexpr int kNoSplitter = 0xffff;
static_assert(2 * MSTAR_MAX_N < kNoSplitter, "arcs and splitters must fit 16 bits");

__global__ void __launch_bounds__(1024, 1)
k_orient(int n, const double* __restrict__ X, const double* __restrict__ Y, const double* __restrict__ Z,
         const int* __restrict__ eu, const int* __restrict__ ev, int* __restrict__ parent, int* __restrict__ level,
         int* __restrict__ root_out) {
  extern __shared__ int smi[];
  typedef unsigned short u16;
  const int na = 2 * (n - 1);
  int* off = smi;                                    // n: end of each vertex's list (after the fill)
  u16* src = reinterpret_cast<u16*>(off + n);        // 2 n: source vertex of each arc
  u16* adj = src + 2 * n;                            // 2 n: arcs by source; then the ranks
  u16* pos = adj + 2 * n;                            // 2 n: place of each arc in adj; then its splitter; then the arc at each rank
  u16* succ = pos + 2 * n;                           // 2 n
  __shared__ unsigned long long rk[32];
  __shared__ int ri[32], part[32], s_root, s_bare;
  __shared__ float s_hi;
  __shared__ int s_len[2][1024], s_nxt[2][1024];
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
  for (int v = tid; v < n; v += nt) off[v] = 0;
  // root: float bounds of |r|^2 first, FP64 for the bodies whose lower bound does not exceed the
  // least upper bound (5 FP64 instructions per body on one SM would take 12 us at N = 10002)
  float uhi = __int_as_float(0x7f800000);
  for (int w = tid; w < n; w += nt) {
    float lx, hx, ly, hy, lz, hz;
    abs_bounds(X[w], lx, hx);
    abs_bounds(Y[w], ly, hy);
    abs_bounds(Z[w], lz, hz);
    uhi = fminf(uhi, (hx * hx + hy * hy + hz * hz) * (1.0f + 0x1p-20f) + 0x1p-126f);
  }
  uhi = __uint_as_float(__reduce_min_sync(0xffffffffu, __float_as_uint(uhi)));
  if (lane == 0) rk[warp] = __float_as_uint(uhi);
  __syncthreads();
  if (warp == 0) {
    const unsigned u = __reduce_min_sync(0xffffffffu, lane < nw ? (unsigned)rk[lane] : 0x7f800000u);
    if (lane == 0) s_hi = __uint_as_float(u);
  }
  // (endpoints outside [0, n) cannot come from the tree builders; they are made 0 so that no
  // shared-memory index leaves its array, and the list is then no tree)
  for (int e = tid; e < n - 1; e += nt) {
    int a = eu[e], b = ev[e];
    if ((unsigned)a >= (unsigned)n || (unsigned)b >= (unsigned)n) a = b = 0;
    src[2 * e] = (u16)a;
    src[2 * e + 1] = (u16)b;
    atomicAdd(&off[a], 1);
    atomicAdd(&off[b], 1);
  }
  __syncthreads();
  uhi = s_hi;
  unsigned long long bk = ~0ull;
  int bi = INT_MAX;
  for (int w = tid; w < n; w += nt) {
    float lx, hx, ly, hy, lz, hz;
    abs_bounds(X[w], lx, hx);
    abs_bounds(Y[w], ly, hy);
    abs_bounds(Z[w], lz, hz);
    if ((lx * lx + ly * ly + lz * lz) * (1.0f - 0x1p-20f) <= uhi) {
      const double x = X[w], y = Y[w], z = Z[w];
      const unsigned long long k =
          key_bits(__dadd_rn(__dadd_rn(__dmul_rn(x, x), __dmul_rn(y, y)), __dmul_rn(z, z)));
      if (k < bk || (k == bk && w < bi)) {
        bk = k;
        bi = w;
      }
    }
  }
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long k2 = __shfl_xor_sync(0xffffffffu, bk, o);
    const int i2 = __shfl_xor_sync(0xffffffffu, bi, o);
    if (k2 < bk || (k2 == bk && i2 < bi)) {
      bk = k2;
      bi = i2;
    }
  }
  if (lane == 0) {
    rk[warp] = bk;
    ri[warp] = bi;
  }
  __syncthreads();
  if (tid == 0) {
    s_bare = 0;
    for (int w = 1; w < nw; ++w)
      if (rk[w] < rk[0] || (rk[w] == rk[0] && ri[w] < ri[0])) {
        rk[0] = rk[w];
        ri[0] = ri[w];
      }
    s_root = min(ri[0], n - 1);
    root_out[0] = s_root;
  }
  // exclusive scan of the degrees: contiguous chunks per thread, then the chunk sums
  const int chunk = (n + nt - 1) / nt;
  const int b0 = min(n, tid * chunk), b1 = min(n, b0 + chunk);
  {
    int sum = 0, total;
    bool bare = false;
    for (int v = b0; v < b1; ++v) {
      sum += off[v];
      bare |= off[v] == 0;
    }
    sum = block_exclusive_scan(sum, part, &total);
    if (bare) s_bare = 1;
    for (int v = b0; v < b1; ++v) {
      const int d = off[v];
      off[v] = sum;
      sum += d;
    }
  }
  __syncthreads();
  const int root = s_root;
  auto star = [&] {
    for (int v = tid; v < n; v += nt) {
      parent[v] = v == root ? -1 : root;
      level[v] = v != root;
    }
  };
  if (s_bare) return star();  // a vertex without an edge
  for (int a = tid; a < na; a += nt) {
    const int p = atomicAdd(&off[src[a]], 1);
    adj[p] = (u16)a;
    pos[a] = (u16)p;
  }
  __syncthreads();
  const int head = adj[root > 0 ? off[root - 1] : 0];
  for (int a = tid; a < na; a += nt) {  // the arc after a: the one after its twin around v
    const int t = a ^ 1, v = src[t], q = pos[t] + 1;
    succ[a] = adj[q < off[v] ? q : (v > 0 ? off[v - 1] : 0)];
  }
  __syncthreads();
  // splitters: the head, and arcs at equal distances by number
  const int ns = min(nt, na);
  for (int a = tid; a < na; a += nt) pos[a] = (u16)kNoSplitter;
  __syncthreads();
  int mine = -1;
  if (tid < ns) mine = tid == 0 ? head : (int)((long long)tid * na / ns);
  if (tid > 0 && mine == head) mine = -1;
  if (mine >= 0) pos[mine] = (u16)tid;
  __syncthreads();
  int len = 0, nxt = 0;
  if (mine >= 0) {
    int a = mine;
    do {
      a = succ[a];
      ++len;
    } while (pos[a] == kNoSplitter && len < na);
    nxt = pos[a] == kNoSplitter ? 0 : pos[a];
  }
  // arcs from each splitter to the end of the tour, by pointer doubling (the segment that returns
  // to the head is the last one)
  s_len[0][tid] = len;
  s_nxt[0][tid] = mine >= 0 ? nxt : 0;  // 0: the end
  __syncthreads();
  int h = 0;
  for (int d = 1; d < ns; d <<= 1, h ^= 1) {
    const int q = s_nxt[h][tid];
    s_len[h ^ 1][tid] = s_len[h][tid] + (q ? s_len[h][q] : 0);
    s_nxt[h ^ 1][tid] = q ? s_nxt[h][q] : 0;
    __syncthreads();
  }
  if (s_len[h][0] != na) return star();  // not connected
  if (mine >= 0) {
    int k = na - s_len[h][tid], a = mine;  // rank of the splitter
    for (int j = 0; j < len; ++j, ++k) {
      adj[a] = (u16)min(max(k, 0), na - 1);
      a = succ[a];
    }
  }
  __syncthreads();
  for (int a = tid; a < na; a += nt) pos[adj[a]] = (u16)a;
  __syncthreads();
  const int ca = (na + nt - 1) / nt;
  const int r0 = min(na, tid * ca), r1 = min(na, r0 + ca);
  int depth = 0, total;
  for (int k = r0; k < r1; ++k) {
    const int a = min((int)pos[k], na - 1);
    depth += adj[a] < adj[a ^ 1] ? 1 : -1;
  }
  depth = block_exclusive_scan(depth, part, &total);
  for (int k = r0; k < r1; ++k) {
    const int a = min((int)pos[k], na - 1);
    const bool away = adj[a] < adj[a ^ 1];
    depth += away ? 1 : -1;
    if (away) {
      parent[src[a ^ 1]] = src[a];
      level[src[a ^ 1]] = depth;
    }
  }
  if (tid == 0) {
    parent[root] = -1;
    level[root] = 0;
  }
}

}  // namespace

// Orientation of an undirected spanning tree (edges eu[e]-ev[e], e < n-1) from Prim's root
// into d.parent, d.level, d.root.
cudaError_t launch_orient(mstar_ctx* c, const int* eu, const int* ev) {
  const int n = c->n;
  const double* X = c->d.r;
  const size_t smem = 20 * (size_t)n;
  cudaError_t e = cudaFuncSetAttribute(k_orient, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  k_orient<<<1, 1024, smem, c->stream>>>(n, X, X + c->npad, X + 2 * (size_t)c->npad, eu, ev, c->d.parent,
                                         c->d.level, c->d.root);
  MSTAR_LAUNCHED(c);
  return cudaGetLastError();
}

// Boruvka MST of d.r into parent/level/root; returns cudaSuccess and sets *tied when a
// tie was seen (the caller then runs the Prim kernel). Scratch lives in the pair partial
// buffer, which is free while the tree is being built.
cudaError_t launch_mst_boruvka(mstar_ctx* c, bool* tied) {
  const int n = c->n, npad = c->npad;
  // the candidates are split into parts, one CTA row each, until the search has about four
  // CTAs per SM (a CTA scanning alone is bound by its latency) or a part would hold fewer than
  // kBT candidates; at most 16
  int sms = 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device) != cudaSuccess) {
    cudaGetLastError();
    sms = 1;
  }
  const int nbt = (n + kBT - 1) / kBT;
  int nparts = 1;
  while (nparts < 16 && nbt * nparts < 4 * sms && n / (2 * nparts) >= kBT) nparts *= 2;
  char* base = reinterpret_cast<char*>(c->d.P);
  auto take = [&](size_t bytes) {
    char* p = base;
    base += (bytes + 255) & ~size_t(255);
    return p;
  };
  float* f4 = reinterpret_cast<float*>(take(sizeof(float) * 4 * npad));
  int* comp = reinterpret_cast<int*>(take(sizeof(int) * npad));
  int* nbr = reinterpret_cast<int*>(take(sizeof(int) * npad));
  unsigned long long* nbrD = reinterpret_cast<unsigned long long*>(take(8 * (size_t)npad));
  unsigned long long* cmin = reinterpret_cast<unsigned long long*>(take(8 * (size_t)npad));
  int* cidx = reinterpret_cast<int*>(take(sizeof(int) * npad));
  int* ccnt = reinterpret_cast<int*>(take(sizeof(int) * npad));
  int* nxt = reinterpret_cast<int*>(take(sizeof(int) * npad));
  int* eu = reinterpret_cast<int*>(take(sizeof(int) * npad));
  int* ev = reinterpret_cast<int*>(take(sizeof(int) * npad));
  unsigned long long* partD = reinterpret_cast<unsigned long long*>(take(8 * (size_t)npad * nparts));
  int* partJ = reinterpret_cast<int*>(take(sizeof(int) * (size_t)npad * nparts));
  int* flags = reinterpret_cast<int*>(take(sizeof(int) * 5));  // [0] tie, [1] edge count, [2] gate of the round,
                                                               // [3] rounds run, [4] gate of the next
  const size_t p_bytes = (size_t)c->nslots * c->NT * 4 * npad * sizeof(double);
  if ((size_t)(base - reinterpret_cast<char*>(c->d.P)) > p_bytes) {  // scratch does not fit: use Prim
    *tied = true;
    return cudaSuccess;
  }
  const double* X = c->d.r;
  const double* Y = X + npad;
  const double* Z = Y + npad;
  const int nb = (n + 255) / 256;
  cudaError_t e = cudaMemsetAsync(flags, 0, sizeof(int) * 5, c->stream);
  if (e != cudaSuccess) return e;
  k_boruvka_init<<<nb, 256, 0, c->stream>>>(n, X, Y, Z, f4, comp, nbr, cmin, ccnt);
  MSTAR_LAUNCHED(c);
  int edges = 0;
  *tied = false;
  // The first check comes after as many rounds as the context's last build ran (consecutive
  // steps build trees of nearly the same point set), then after every further round.
  int round = 0;
  while (round < 64 && edges < n - 1) {
    const int batch = round == 0 ? (c->mst_rounds > 0 ? c->mst_rounds : 1) : 1;
    for (int b = 0; b < batch && round < 64; ++b, ++round) {
      k_nfn<<<dim3((n + kBT - 1) / kBT, nparts), kBT, 0, c->stream>>>(n, npad, nparts, X, Y, Z, f4, comp, nbr,
                                                                       partD, partJ, flags);
      k_nfn_merge<<<(n + 63) / 64, 64, 0, c->stream>>>(n, npad, nparts, comp, nbr, nbrD, partD, partJ, flags,
                                                       flags + 2);
      k_comp_min<<<nb, 256, 0, c->stream>>>(n, comp, nbrD, cmin, flags + 2);
      k_comp_edge<<<nb, 256, 0, c->stream>>>(n, comp, nbrD, cmin, cidx, ccnt, flags, flags + 2);
      k_hook<<<nb, 256, 0, c->stream>>>(n, comp, nbr, cidx, nxt, eu, ev, flags + 1, flags + 2);
      k_relabel<<<nb, 256, 0, c->stream>>>(n, comp, nxt, cmin, ccnt, flags);
      c->launches += 6;
      if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    if ((e = cudaMemcpyAsync(c->host_buf, flags, sizeof(int) * 4, cudaMemcpyDeviceToHost, c->stream)) != cudaSuccess)
      return e;
    if ((e = cudaStreamSynchronize(c->stream)) != cudaSuccess) return e;
    int fl[4];
    std::memcpy(fl, c->host_buf, sizeof(fl));
    if (fl[0]) {
      *tied = true;
      return cudaSuccess;
    }
    edges = fl[1];
    c->mst_rounds = fl[3];
  }
  if (edges != n - 1) {  // cannot happen without ties; be safe
    *tied = true;
    return cudaSuccess;
  }
  return launch_orient(c, eu, ev);
}

}  // namespace mstar
