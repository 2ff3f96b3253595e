// Divide-and-conquer spanning tree of Sec. 3.3 on the GPU.
//
// The paper's large-N alternative to Prim's MST: split the bodies into about sqrt(N)
// subgraphs with an octree, build the MST of every subgraph and of the meta-graph whose
// vertices are the contracted subgraphs and whose edge weights are the cheapest edges
// between them (the cut property), and order the union of these edges by a walk from the
// root. The result is a spanning tree a few per cent longer than the MST that is locally
// the MST of every subgraph.
//
// Rules (each also the CPU definition's):
// - bounding cube: the centre of each coordinate's extent, half-size the largest half-extent;
//   at each of 16 depths a body goes to the child whose centre it is not below (x >= c);
//   the Morton key concatenates the x, y, z choices, most significant first;
// - partition: starting from the cube, the cell with the most bodies (the first in Morton
//   order on ties) is replaced by its non-empty children until there are at least
//   `nsub` cells or the most populous cell cannot split (one body or depth 16);
// - subgraph MSTs: Prim from the subgraph's lowest body index; a key is replaced only by a
//   strictly smaller squared distance; the next vertex is the lowest (key, index);
// - meta weights: for subgraphs a < b, the lexicographic minimum of (d^2, i, j) over
//   i in a, j in b; the meta-graph's Prim starts at subgraph 0 and compares these triples;
// - the walk: breadth first from the body closest to the centre of mass (lowest index on
//   ties); parent and level are unique for a tree whatever the visiting order.
// Squared distances are ((dx*dx)+(dy*dy))+(dz*dz) with dx = x_u - x_v, each operation rounded
// separately, as in the Prim kernel.
#include <algorithm>
#include <climits>
#include <cmath>
#include <cstring>

#include "device.cuh"
#include "internal.h"
#include "nearest.cuh"

namespace mstar {
namespace {

constexpr int kDepth = 16;
constexpr int kDcParts = 8;       // slices of the counting sort and of the neighbour search
constexpr int kMetaZ = 2;         // CTAs that share a pair of subgraphs' cheapest edge
constexpr int kDcBoundCtas = 32;  // CTAs of the bounding cube's reduction
constexpr int kIdxBits = 14;
constexpr unsigned long long kIdxMask = (1ull << kIdxBits) - 1;
constexpr unsigned long long kInfBits = 0x7ff0000000000000ull;
static_assert(MSTAR_MAX_N <= (1 << kIdxBits), "a body index must fit below the Morton key");

struct DcEdge {
  unsigned long long d;  // bits of the non-negative squared distance (ordered like the value)
  int i, j;              // i in the lower-numbered subgraph
};

__device__ __forceinline__ bool dc_less(const DcEdge& a, const DcEdge& b) {
  if (a.d != b.d) return a.d < b.d;
  if (a.i != b.i) return a.i < b.i;
  return a.j < b.j;
}

struct Cell {
  int depth, lo, hi;
};

// Device scratch of the builder (carved from the context workspace).
struct DcLayout {
  int mc;                        // cell capacity
  unsigned long long* keys;      // (Morton key << 14 | body) by body
  unsigned long long* sorted;    // the same, sorted
  int* rank;                     // kDcParts x n partial ranks of the sort
  double* bounds;                // kDcBoundCtas x 6 partial extrema
  float4* f4;                    // per body: float x, y, z and their conversion error bound
  int* ncell;                    // [1]
  int* leafid;                   // subgraph of each sorted position
  int* leaf_start;               // mc + 1
  unsigned long long* key;       // Prim keys by sorted position
  float* keyf;                   // the keys rounded up to float
  int* kp;                       // Prim parent candidates by sorted position
  DcEdge* W;                     // mc x mc meta weights (a < b entries)
  double* sx;                    // positions in sorted order (3 planes) ...
  float4* sf4;                   // ... and their float copies
  int *comp, *nbr, *nxt, *cidx;  // local Boruvka rounds, by sorted position
  unsigned long long* nbrD;
  unsigned long long* partD;     // kDcParts x n nearest foreign neighbours per slice
  int* partJ;
  int* lcount;                   // edges found per subgraph
  int* flags;                    // [0] tie, [1] edges, [3] rounds run
  int *eu, *ev;                  // the n - 1 tree edges
  size_t bytes;
};

int target_of(int n, int nsub) { return nsub > 0 ? nsub : (int)ceil(sqrt((double)n)); }

DcLayout dc_layout(int n, int nsub, char* base) {
  DcLayout L{};
  const int target = target_of(n, nsub);
  L.mc = target + 8 < n ? target + 8 : n;
  size_t off = 0;
  auto take = [&](size_t bytes) {
    off = (off + 255) & ~size_t(255);
    char* p = base ? base + off : nullptr;
    off += bytes;
    return p;
  };
  L.keys = reinterpret_cast<unsigned long long*>(take(8 * (size_t)n));
  L.sorted = reinterpret_cast<unsigned long long*>(take(8 * (size_t)n));
  L.rank = reinterpret_cast<int*>(take(sizeof(int) * (size_t)n * kDcParts));
  L.bounds = reinterpret_cast<double*>(take(sizeof(double) * 6 * kDcBoundCtas));
  L.f4 = reinterpret_cast<float4*>(take(sizeof(float4) * (size_t)n));
  L.ncell = reinterpret_cast<int*>(take(sizeof(int)));
  L.leafid = reinterpret_cast<int*>(take(sizeof(int) * (size_t)n));
  L.leaf_start = reinterpret_cast<int*>(take(sizeof(int) * (size_t)(L.mc + 1)));
  L.key = reinterpret_cast<unsigned long long*>(take(8 * (size_t)n));
  L.keyf = reinterpret_cast<float*>(take(sizeof(float) * (size_t)n));
  L.kp = reinterpret_cast<int*>(take(sizeof(int) * (size_t)n));
  L.W = reinterpret_cast<DcEdge*>(take(sizeof(DcEdge) * (size_t)L.mc * L.mc * kMetaZ));
  L.eu = reinterpret_cast<int*>(take(sizeof(int) * (size_t)n));
  L.ev = reinterpret_cast<int*>(take(sizeof(int) * (size_t)n));
  L.sx = reinterpret_cast<double*>(take(sizeof(double) * 3 * (size_t)n));
  L.sf4 = reinterpret_cast<float4*>(take(sizeof(float4) * (size_t)n));
  L.comp = reinterpret_cast<int*>(take(sizeof(int) * (size_t)n));
  L.nbr = reinterpret_cast<int*>(take(sizeof(int) * (size_t)n));
  L.nxt = reinterpret_cast<int*>(take(sizeof(int) * (size_t)n));
  L.cidx = reinterpret_cast<int*>(take(sizeof(int) * (size_t)n));
  L.nbrD = reinterpret_cast<unsigned long long*>(take(8 * (size_t)n));
  L.partD = reinterpret_cast<unsigned long long*>(take(8 * (size_t)n * kDcParts));
  L.partJ = reinterpret_cast<int*>(take(sizeof(int) * (size_t)n * kDcParts));
  L.lcount = reinterpret_cast<int*>(take(sizeof(int) * (size_t)L.mc));
  L.flags = reinterpret_cast<int*>(take(sizeof(int) * 4));
  L.bytes = (off + 255) & ~size_t(255);
  return L;
}

// Extrema of the coordinates, per CTA (k_dc_keys combines them): one CTA took 39 us at N = 10002 for
// 60000 FP64 comparisons.
__global__ void __launch_bounds__(256)
k_dc_bounds(int n, const double* __restrict__ X, const double* __restrict__ Y, const double* __restrict__ Z,
            double* __restrict__ bounds) {
  __shared__ double red[8][6];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  double v[6] = {INFINITY, INFINITY, INFINITY, -INFINITY, -INFINITY, -INFINITY};
  for (int i = blockIdx.x * 256 + tid; i < n; i += 256 * kDcBoundCtas) {
    const double c[3] = {X[i], Y[i], Z[i]};
    for (int k = 0; k < 3; ++k) {
      v[k] = fmin(v[k], c[k]);
      v[3 + k] = fmax(v[3 + k], c[k]);
    }
  }
  for (int o = 16; o > 0; o >>= 1)
    for (int k = 0; k < 3; ++k) {
      v[k] = fmin(v[k], __shfl_xor_sync(0xffffffffu, v[k], o));
      v[3 + k] = fmax(v[3 + k], __shfl_xor_sync(0xffffffffu, v[3 + k], o));
    }
  if (lane == 0)
    for (int k = 0; k < 6; ++k) red[warp][k] = v[k];
  __syncthreads();
  if (tid < 6) {
    double e = red[0][tid];
    for (int w = 1; w < 8; ++w) e = tid < 3 ? fmin(e, red[w][tid]) : fmax(e, red[w][tid]);
    bounds[blockIdx.x * 6 + tid] = e;
  }
}

// Bounding cube: the centre of each coordinate's extent, the largest half-extent (by warp 0).
__device__ __forceinline__ void dc_cube(const double* __restrict__ bounds, double* cube) {
  const int lane = threadIdx.x & 31;
  static_assert(kDcBoundCtas == 32, "one partial per lane");
  double mn[3], mx[3], hs = 0.0;
  for (int k = 0; k < 3; ++k) {
    mn[k] = bounds[lane * 6 + k];
    mx[k] = bounds[lane * 6 + 3 + k];
    for (int o = 16; o > 0; o >>= 1) {
      mn[k] = fmin(mn[k], __shfl_xor_sync(0xffffffffu, mn[k], o));
      mx[k] = fmax(mx[k], __shfl_xor_sync(0xffffffffu, mx[k], o));
    }
    if (lane == 0) cube[k] = __dmul_rn(__dadd_rn(mn[k], mx[k]), 0.5);
    const double e = __dmul_rn(__dsub_rn(mx[k], mn[k]), 0.5);
    if (e > hs) hs = e;
  }
  if (lane == 0) cube[3] = hs;
}

// Packed Morton keys and the float copies of the positions with a bound on their conversion error
// (for the distance filters).
__global__ void __launch_bounds__(256)
k_dc_keys(int n, const double* __restrict__ X, const double* __restrict__ Y, const double* __restrict__ Z,
          const double* __restrict__ bounds, unsigned long long* __restrict__ keys, float4* __restrict__ f4) {
  __shared__ double cube[4];
  if (threadIdx.x < 32) dc_cube(bounds, cube);
  __syncthreads();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double p[3] = {X[i], Y[i], Z[i]};
  double c[3] = {cube[0], cube[1], cube[2]}, h = cube[3];
  unsigned long long kk = 0;
  for (int d = 0; d < kDepth; ++d) {
    h = __dmul_rn(h, 0.5);
    unsigned bits = 0;
    for (int k = 0; k < 3; ++k) {
      const int b = p[k] >= c[k];
      bits = (bits << 1) | (unsigned)b;
      c[k] = b ? __dadd_rn(c[k], h) : __dsub_rn(c[k], h);
    }
    kk = (kk << 3) | bits;
  }
  keys[i] = (kk << kIdxBits) | (unsigned long long)i;
  const float fx = __double2float_rn(p[0]), fy = __double2float_rn(p[1]), fz = __double2float_rn(p[2]);
  f4[i] = make_float4(fx, fy, fz, fmaxf(fabsf(fx), fmaxf(fabsf(fy), fabsf(fz))) * 0x1p-22f + 1e-37f);
}

// The sort, by counting: a key's place is the number of smaller keys (they are distinct: the body's
// index is part of the key), over kDcParts slices of the keys. A bitonic sort in one CTA took 180 us
// at N = 10002, these two kernels 25.
__global__ void __launch_bounds__(128)
k_dc_rank(int n, const unsigned long long* __restrict__ keys, int* __restrict__ rank) {
  __shared__ unsigned long long s[128];
  const int i = blockIdx.x * 128 + threadIdx.x, q = blockIdx.y;
  const int per = (n + kDcParts - 1) / kDcParts, lo = q * per, hi = min(n, lo + per);
  const unsigned long long k = i < n ? keys[i] : 0ull;
  int a = 0;
  for (int t = lo; t < hi; t += 128) {
    __syncthreads();
    s[threadIdx.x] = t + (int)threadIdx.x < hi ? keys[t + threadIdx.x] : ~0ull;
    __syncthreads();
#pragma unroll 8
    for (int j = 0; j < 128; ++j) a += s[j] < k;
  }
  if (i < n) rank[(size_t)q * n + i] = a;
}

// Keys, positions and float copies into sorted order; the local rounds' first state.
__global__ void __launch_bounds__(256)
k_dc_place(int n, int mc, const unsigned long long* __restrict__ keys, const int* __restrict__ rank,
           const double* __restrict__ X, const double* __restrict__ Y, const double* __restrict__ Z,
           const float4* __restrict__ f4, unsigned long long* __restrict__ sorted, double* __restrict__ sx,
           float4* __restrict__ sf4, int* __restrict__ comp, int* __restrict__ nbr, int* __restrict__ lcount,
           int* __restrict__ flags) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < mc) lcount[i] = 0;
  if (i < 4) flags[i] = 0;
  if (i >= n) return;
  int a = 0;
#pragma unroll
  for (int q = 0; q < kDcParts; ++q) a += rank[(size_t)q * n + i];
  sorted[a] = keys[i];
  sx[a] = X[i];
  sx[n + a] = Y[i];
  sx[2 * (size_t)n + a] = Z[i];
  sf4[a] = f4[i];
  comp[a] = a;
  nbr[a] = -1;
}

// First position in [lo, hi) whose Morton digit at `shift` exceeds `dgt` (digits are
// non-decreasing inside a cell).
__device__ int digit_end(const unsigned long long* __restrict__ sorted, int lo, int hi, int shift, unsigned dgt) {
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (((sorted[mid] >> shift) & 7u) <= dgt) lo = mid + 1;
    else hi = mid;
  }
  return lo;
}

// Greedy octree partition (warp 0: the lanes share the search for the most populous cell, and eight
// of them find the ends of its children), then the subgraph of every sorted position and the
// subgraph starts (cells partition [0, n); their starts are flagged and scanned). One thread took
// 104 us at N = 10002 with the scan below, the warp 26.
__global__ void __launch_bounds__(1024, 1)
k_dc_partition(int n, int target, int mc, const unsigned long long* __restrict__ gsorted, int* __restrict__ ncell,
               int* __restrict__ leafid, int* __restrict__ leaf_start) {
  extern __shared__ unsigned long long sorted[];  // n keys
  __shared__ int s_nc;
  __shared__ int wsum[32];
  __shared__ Cell cells[kDcMaxSub + 8];
  const int tid = threadIdx.x;
  for (int p = tid; p < n; p += blockDim.x) sorted[p] = gsorted[p];
  __syncthreads();
  if (tid < 32) {
    const int lane = tid;
    int nc = 1;
    if (lane == 0) cells[0] = Cell{0, 0, n};
    __syncwarp();
    while (nc < target) {
      // the most bodies, the lowest start on ties
      int cnt = -1, lo = INT_MAX, at = 0;
      for (int c = lane; c < nc; c += 32) {
        const int k = cells[c].hi - cells[c].lo;
        if (k > cnt || (k == cnt && cells[c].lo < lo)) {
          cnt = k;
          lo = cells[c].lo;
          at = c;
        }
      }
      const int big = __reduce_max_sync(0xffffffffu, cnt);
      const int first_lo = __reduce_min_sync(0xffffffffu, cnt == big ? lo : INT_MAX);
      const unsigned who = __ballot_sync(0xffffffffu, cnt == big && lo == first_lo);
      const int best = __shfl_sync(0xffffffffu, at, __ffs(who) - 1);
      const Cell b = cells[best];
      if (b.hi - b.lo <= 1 || b.depth == kDepth) break;
      const int shift = 3 * (kDepth - b.depth - 1) + kIdxBits;
      // lane d < 8: the end of child d; a child is non-empty where its end is past the one before
      const int end = lane < 8 ? digit_end(sorted, b.lo, b.hi, shift, (unsigned)lane) : b.hi;
      const int beg0 = __shfl_up_sync(0xffffffffu, end, 1);
      const int beg = lane == 0 ? b.lo : beg0;
      const unsigned kids = __ballot_sync(0xffffffffu, lane < 8 && end > beg);
      const int r = __popc(kids & ((1u << lane) - 1u));  // the first child replaces the cell, the others follow
      if ((kids >> lane) & 1u) {
        const int to = r == 0 ? best : nc + r - 1;
        if (r == 0 || to < mc) cells[to] = Cell{b.depth + 1, beg, end};
      }
      nc = min(mc, nc + __popc(kids) - 1);
      __syncwarp();
    }
    if (lane == 0) {
      s_nc = nc;
      *ncell = nc;
    }
  }
  for (int p = tid; p < n; p += blockDim.x) leafid[p] = 0;
  __syncthreads();
  const int nc = s_nc;
  for (int c = tid; c < nc; c += blockDim.x) leafid[cells[c].lo] = 1;
  __syncthreads();
  // inclusive scan of the start flags over the sorted positions: chunk per thread
  const int ch = (n + blockDim.x - 1) / blockDim.x;
  const int b0 = tid * ch, b1 = min(n, b0 + ch);
  int local = 0;
  for (int p = b0; p < b1; ++p) local += leafid[p];
  int incl = local;
  const int lane = tid & 31, warp = tid >> 5;
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  if (lane == 31) wsum[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    int w = lane < (int)(blockDim.x >> 5) ? wsum[lane] : 0;
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += t;
    }
    wsum[lane] = w;
  }
  __syncthreads();
  int run = incl - local + (warp > 0 ? wsum[warp - 1] : 0);
  for (int p = b0; p < b1; ++p) {
    const int f = leafid[p];
    run += f;
    leafid[p] = run - 1;
    if (f) leaf_start[run - 1] = p;
  }
  if (tid == 0) leaf_start[nc] = n;
}

// Prim inside every subgraph: one CTA of kLpThreads per subgraph. A subgraph of up to
// kLeafSmem bodies is staged in shared memory (positions, their float copies, keys and the
// keys rounded up to float, candidate parents, body indices); larger ones work from global
// memory. The thread that owns a position (its offset from the subgraph start, mod the CTA
// size) keeps its key and candidate parent; kp = -2 marks tree vertices. A relaxation
// computes the exact FP64 distance only when the rigorous float lower bound does not exceed
// the key rounded up: otherwise the distance is certainly above the key and the strict
// update cannot happen.
constexpr int kLeafSmem = 1024;
constexpr int kLpThreads = 128;

__device__ __forceinline__ float dc_lower_bound(const float4& p, const float4& q) {
  const float dx = fabsf(p.x - q.x), dy = fabsf(p.y - q.y), dz = fabsf(p.z - q.z);
  const float e = p.w + q.w;
  const float lx = fmaxf(0.f, fmaf(dx, -0x1p-22f, dx) - e), ly = fmaxf(0.f, fmaf(dy, -0x1p-22f, dy) - e),
              lz = fmaxf(0.f, fmaf(dz, -0x1p-22f, dz) - e);
  const float s = fmaf(lz, lz, fmaf(ly, ly, lx * lx));
  // relative rounding of normal results, and 2^-144 for the absolute rounding (<= 2^-150 per
  // operation) of squares and sums below 2^-126
  return fmaxf(fmaf(s, -0x1p-20f, s) - 0x1p-144f, 0.0f);
}

struct LpCand {
  unsigned long long k;
  int v, q;
};

__device__ __forceinline__ bool lp_less(const LpCand& a, const LpCand& b) {
  return a.k < b.k || (a.k == b.k && a.v < b.v);
}

__global__ void __launch_bounds__(kLpThreads)
k_dc_local_prim(const int* __restrict__ ncell, const int* __restrict__ leaf_start,
                const unsigned long long* __restrict__ sorted, const double* __restrict__ X,
                const double* __restrict__ Y, const double* __restrict__ Z, const float4* __restrict__ f4,
                unsigned long long* __restrict__ gkey, float* __restrict__ gkeyf, int* __restrict__ gkp,
                int* __restrict__ eu, int* __restrict__ ev) {
  extern __shared__ double sm[];
  __shared__ LpCand red[2][kLpThreads / 32];
  const int g = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (g >= *ncell) return;
  const int lo = leaf_start[g], hi = leaf_start[g + 1], cnt = hi - lo;
  const bool shared = cnt <= kLeafSmem;
  double* sx = sm;
  double* sy = sx + kLeafSmem;
  double* sz = sy + kLeafSmem;
  unsigned long long* skey = reinterpret_cast<unsigned long long*>(sz + kLeafSmem);
  float4* sf = reinterpret_cast<float4*>(skey + kLeafSmem);
  float* skeyf = reinterpret_cast<float*>(sf + kLeafSmem);
  int* skp = reinterpret_cast<int*>(skeyf + kLeafSmem);
  int* bid = skp + kLeafSmem;
  unsigned long long* key = shared ? skey : gkey + lo;
  float* keyf = shared ? skeyf : gkeyf + lo;
  int* kp = shared ? skp : gkp + lo;
  LpCand st{~0ull, INT_MAX, -1};
  for (int q = tid; q < cnt; q += kLpThreads) {
    const int b = (int)(sorted[lo + q] & kIdxMask);
    if (shared) {
      sx[q] = X[b];
      sy[q] = Y[b];
      sz[q] = Z[b];
      sf[q] = f4[b];
      bid[q] = b;
    }
    key[q] = kInfBits;
    keyf[q] = INFINITY;
    kp[q] = -1;
    if (b < st.v) st = LpCand{0, b, q};
  }
  // the start vertex: the lowest body index of the subgraph
  for (int o = 16; o > 0; o >>= 1) {
    LpCand c;
    c.k = 0;
    c.v = __shfl_xor_sync(0xffffffffu, st.v, o);
    c.q = __shfl_xor_sync(0xffffffffu, st.q, o);
    if (c.v < st.v) st = c;
  }
  if (lane == 0) red[0][warp] = st;
  __syncthreads();
  for (int w = 0; w < kLpThreads / 32; ++w)
    if (red[0][w].v < st.v) st = red[0][w];
  if ((st.q % kLpThreads) == tid) kp[st.q] = -2;
  int u = st.v;
  double ux = X[u], uy = Y[u], uz = Z[u];
  float4 uf = f4[u];
  const int e0 = lo - g;  // local edges of the earlier subgraphs: sum (size - 1)
  for (int it = 1; it < cnt; ++it) {
    LpCand best{~0ull, INT_MAX, -1};
    for (int q = tid; q < cnt; q += kLpThreads) {
      if (kp[q] == -2) continue;
      const int v = shared ? bid[q] : (int)(sorted[lo + q] & kIdxMask);
      unsigned long long k = key[q];
      const float4 fv = shared ? sf[q] : f4[v];
      if (dc_lower_bound(uf, fv) <= keyf[q]) {
        const double vx = shared ? sx[q] : X[v], vy = shared ? sy[q] : Y[v], vz = shared ? sz[q] : Z[v];
        const double dx = __dsub_rn(ux, vx), dy = __dsub_rn(uy, vy), dz = __dsub_rn(uz, vz);
        const double d2 = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
        const unsigned long long d = key_bits(d2);
        if (d < k) {
          k = d;
          key[q] = d;
          keyf[q] = __double2float_ru(d2);
          kp[q] = u;
        }
      }
      const LpCand c{k, v, q};
      if (lp_less(c, best)) best = c;
    }
    for (int o = 16; o > 0; o >>= 1) {
      LpCand c;
      c.k = __shfl_xor_sync(0xffffffffu, best.k, o);
      c.v = __shfl_xor_sync(0xffffffffu, best.v, o);
      c.q = __shfl_xor_sync(0xffffffffu, best.q, o);
      if (lp_less(c, best)) best = c;
    }
    if (lane == 0) red[it & 1][warp] = best;
    __syncthreads();
    for (int w = 0; w < kLpThreads / 32; ++w)
      if (lp_less(red[it & 1][w], best)) best = red[it & 1][w];
    if ((best.q % kLpThreads) == tid) {
      // (no parent: every distance to the body overflows or is NaN; any edge keeps the tree whole)
      eu[e0 + it - 1] = kp[best.q] >= 0 ? kp[best.q] : st.v;
      ev[e0 + it - 1] = best.v;
      kp[best.q] = -2;
    }
    u = best.v;
    if (shared) {
      ux = sx[best.q];
      uy = sy[best.q];
      uz = sz[best.q];
      uf = sf[best.q];
    } else {
      ux = X[u];
      uy = Y[u];
      uz = Z[u];
      uf = f4[u];
    }
  }
}

// The same trees by Boruvka rounds over the whole GPU, in sorted order: within a subgraph whose
// distances are distinct its MST is unique, so the edges are Prim's; any exact tie sets flags[0],
// and the host then runs k_dc_local_prim instead. One CTA per subgraph is bound by the largest one's
// sequential iterations (1.1-4.9 ms at N = 10002, for subgraphs of 670 to 1050 bodies); the rounds
// take 25 us each there, five of them.
//
// Search of a round: thread p, whose cached neighbour is missing or has become internal, scans its
// subgraph's positions that lie in the q-th slice of the CTA's subgraphs.
constexpr int kDcT = 128;
__global__ void __launch_bounds__(kDcT)
k_dc_nfn(int n, const int* __restrict__ ncell, const int* __restrict__ leafid, const int* __restrict__ leaf_start,
         const double* __restrict__ sx, const float4* __restrict__ sf4, const int* __restrict__ comp,
         const int* __restrict__ nbr, const int* __restrict__ lcount, unsigned long long* __restrict__ partD,
         int* __restrict__ partJ, int* __restrict__ flags) {
  __shared__ float4 sq[kDcT];
  __shared__ int s_emax, s_stop;
  if (threadIdx.x == 0) {
    // read once: other CTAs of this launch may set the tie flag meanwhile, and a CTA whose warps saw
    // different values would go on with part of its warps
    s_stop = flags[0] != 0 || flags[1] >= n - *ncell;
    s_emax = 0;
    if (blockIdx.x == 0 && blockIdx.y == 0 && !s_stop) flags[3] += 1;
  }
  __syncthreads();
  if (s_stop) return;
  const int p0 = blockIdx.x * kDcT, p = p0 + threadIdx.x, q = blockIdx.y;
  const int u_lo = leaf_start[leafid[p0]], u_hi = leaf_start[leafid[min(n, p0 + kDcT) - 1] + 1];
  const int per = (u_hi - u_lo + kDcParts - 1) / kDcParts;
  const int s_lo = u_lo + q * per, s_hi = min(u_hi, s_lo + per);
  bool need = false;
  int cp = -1, lo = 0, hi = 0;
  if (p < n) {
    const int g = leafid[p];
    cp = comp[p];
    lo = max(leaf_start[g], s_lo);
    hi = min(leaf_start[g + 1], s_hi);
    const int b = nbr[p];
    need = lcount[g] < leaf_start[g + 1] - leaf_start[g] - 1 && (b < 0 || comp[b] == cp);
  }
  if (!__syncthreads_or(need)) return;
  const float4 fp = p < n ? sf4[p] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  NearestScan ns;
  ns.clear();
  for (int t0 = s_lo; t0 < s_hi; t0 += kDcT) {
    __syncthreads();
    const int j = t0 + threadIdx.x;
    float4 c = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if (j < s_hi) {
      c = sf4[j];
      sq[threadIdx.x] = make_float4(c.x, c.y, c.z, __int_as_float(comp[j]));
    }
    const int e = __reduce_max_sync(0xffffffffu, __float_as_int(c.w));
    if ((threadIdx.x & 31) == 0) atomicMax(&s_emax, e);
    __syncthreads();
    if (!need) continue;
    const int k1 = min(kDcT, hi - t0);
    for (int k = max(0, lo - t0); k < k1; ++k) {
      const float4 s = sq[k];
      ns.add(fp.x - s.x, fp.y - s.y, fp.z - s.z, __float_as_int(s.w) != cp, t0 + k);
    }
  }
  __syncthreads();
  const float emax = fp.w + __int_as_float(s_emax);
  const double *X = sx, *Y = sx + n, *Z = sx + 2 * (size_t)n;
  auto exact = [&](int a, int b) {
    const double dx = __dsub_rn(X[a], X[b]), dy = __dsub_rn(Y[a], Y[b]), dz = __dsub_rn(Z[a], Z[b]);
    return key_bits(__dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz)));
  };
  unsigned long long bD = ~0ull;
  int bj = -1, mytie = 0;
  const bool found = need && !ns.none();
  const bool sure = !found || ns.certain(emax);
  if (found && sure) {
    bj = ns.j1;
    bD = exact(p, bj);
  }
  const int lane = threadIdx.x & 31;
  for (unsigned todo = __ballot_sync(0xffffffffu, !sure); todo; todo &= todo - 1) {
    const int l = __ffs(todo) - 1;
    const int vp = __shfl_sync(0xffffffffu, p, l), vc = __shfl_sync(0xffffffffu, cp, l);
    const int vlo = __shfl_sync(0xffffffffu, lo, l), vhi = __shfl_sync(0xffffffffu, hi, l);
    const float lim = __shfl_sync(0xffffffffu, ns.limit(emax), l);
    const float vx = __shfl_sync(0xffffffffu, fp.x, l), vy = __shfl_sync(0xffffffffu, fp.y, l),
                vz = __shfl_sync(0xffffffffu, fp.z, l);
    unsigned long long d = ~0ull;
    int dj = -1, tied = 0;
    for (int jj = vlo + lane; jj < vhi; jj += 32) {
      if (comp[jj] == vc) continue;
      const float4 c = sf4[jj];
      const float dx = vx - c.x, dy = vy - c.y, dz = vz - c.z;
      if (fmaf(dz, dz, fmaf(dy, dy, dx * dx)) > lim) continue;
      const unsigned long long db = exact(vp, jj);
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
  partD[(size_t)q * n + p] = bD;
  partJ[(size_t)q * n + p] = bj;
  if (mytie) atomicOr(flags, 1);
}

// The rest of the round, one CTA per subgraph: the slices' neighbours merged, each component's
// cheapest edge, hooking and relabelling (components are labelled by a sorted position of theirs).
constexpr int kDcRoundT = 512;
__global__ void __launch_bounds__(kDcRoundT)
k_dc_round(int n, const int* __restrict__ ncell, const int* __restrict__ leaf_start,
           const unsigned long long* __restrict__ sorted, int* comp, int* nbr, unsigned long long* nbrD, int* cidx,
           int* nxt, const unsigned long long* __restrict__ partD, const int* __restrict__ partJ,
           unsigned long long* cmin, int* lcount, int* __restrict__ eu, int* __restrict__ ev, int* flags) {
  __shared__ int s_tie, s_edges, s_stop;
  const int g = blockIdx.x;
  if (g >= *ncell) return;
  const int lo = leaf_start[g], hi = leaf_start[g + 1];
  if (threadIdx.x == 0) {
    s_stop = flags[0];  // read once, as in the search: it may change during the launch
    s_tie = s_edges = 0;
  }
  __syncthreads();
  const int done = lcount[g];
  if (s_stop || done >= hi - lo - 1) return;
  for (int p = lo + threadIdx.x; p < hi; p += kDcRoundT) {
    cmin[p] = ~0ull;
    cidx[p] = -1;
  }
  __syncthreads();
  for (int p = lo + threadIdx.x; p < hi; p += kDcRoundT) {
    const int c = comp[p];
    int b = nbr[p];
    if (b < 0 || comp[b] == c) {
      unsigned long long bD = ~0ull;
      b = -1;
      for (int q = 0; q < kDcParts; ++q) {
        const unsigned long long d = partD[(size_t)q * n + p];
        const int j = partJ[(size_t)q * n + p];
        if (j < 0) continue;
        if (d < bD) {
          bD = d;
          b = j;
        } else if (d == bD && j != b) {
          s_tie = 1;
        }
      }
      nbr[p] = b;
      nbrD[p] = bD;
    }
    if (b >= 0) atomicMin(&cmin[c], nbrD[p]);
  }
  __syncthreads();
  for (int p = lo + threadIdx.x; p < hi; p += kDcRoundT)
    if (nbr[p] >= 0 && nbrD[p] == cmin[comp[p]] && atomicExch(&cidx[comp[p]], p) >= 0) s_tie = 1;
  __syncthreads();
  if (s_tie) {  // two cheapest edges of equal weight
    if (threadIdx.x == 0) atomicOr(flags, 1);
    return;
  }
  for (int c = lo + threadIdx.x; c < hi; c += kDcRoundT) {
    if (comp[c] != c) continue;
    const int i = cidx[c];
    if (i < 0) {  // only after a tie elsewhere
      nxt[c] = c;
      continue;
    }
    const int j = nbr[i], t = comp[j];
    const int it = cidx[t];
    const bool mutual = it >= 0 && comp[nbr[it]] == c;
    nxt[c] = mutual && c < t ? c : t;
    if (!mutual || c < t) {
      const int k = atomicAdd(&s_edges, 1);
      if (done + k < hi - lo - 1) {  // the subgraph's edges lie at lo - g ...
        eu[lo - g + done + k] = (int)(sorted[i] & kIdxMask);
        ev[lo - g + done + k] = (int)(sorted[j] & kIdxMask);
      }
    }
  }
  __syncthreads();
  for (int p = lo + threadIdx.x; p < hi; p += kDcRoundT) {
    int c = comp[p];
    for (int guard = lo; guard < hi && nxt[c] != c; ++guard) c = nxt[c];
    cidx[p] = c;  // (the new labels are written when every chain has been followed)
  }
  __syncthreads();
  for (int p = lo + threadIdx.x; p < hi; p += kDcRoundT) comp[p] = cidx[p];
  if (threadIdx.x == 0) {
    lcount[g] = done + s_edges;
    atomicAdd(&flags[1], s_edges);
  }
}

// Meta-graph weights: for every pair of subgraphs a < b the least (d^2, i, j) over i in a, j in b.
// The larger subgraph's bodies are taken 32 at a time, one per lane of a warp, against all bodies of
// the smaller one; the warps of kMetaZ CTAs share a pair's groups (most pairs have one to four, the
// largest pair's 33 would keep one CTA busy for 50 us). A first pass finds each lane's least float
// squared distance; only bodies whose least is within the error of the CTA's (as in nearest.cuh)
// are looked at again, by their whole warp, comparing in FP64 every pair that can win or tie. With
// an FP64 distance wherever a float bound beat the thread's best, 457 us at N = 10002 (104
// subgraphs, the largest of 1045 bodies); 130 now.
constexpr int kMetaT = 256;

__global__ void __launch_bounds__(kMetaT)
k_dc_meta_w(int n, const int* __restrict__ ncell, int mc, const int* __restrict__ leaf_start,
            const unsigned long long* __restrict__ sorted, const double* __restrict__ sx,
            const float4* __restrict__ sf4, DcEdge* __restrict__ W) {
  __shared__ DcEdge red[kMetaT / 32];
  __shared__ int s_min, s_emax;
  const int nc = *ncell, z = blockIdx.y;
  if ((int)blockIdx.x >= nc * (nc - 1) / 2) return;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int a, b;
  tile_pair(blockIdx.x, nc - 1, a, b);  // rows of nc - 1 - a pairs
  b += 1;
  const int la = leaf_start[a], sa = leaf_start[a + 1] - la;
  const int lb = leaf_start[b], sb = leaf_start[b + 1] - lb;
  const bool swap = sa > sb;  // outer: the larger subgraph, by lane; inner: the other
  const int lo = swap ? la : lb, so = swap ? sa : sb, li = swap ? lb : la, si = swap ? sb : sa;
  if (threadIdx.x == 0) {
    s_min = 0x7f800000;
    s_emax = 0;
  }
  __syncthreads();
  constexpr int kStep = 32 * (kMetaT / 32) * kMetaZ;  // bodies between a warp's groups
  const int q0 = 32 * (z * (kMetaT / 32) + warp) + lane;
  float mine = __int_as_float(0x7f800000), em = 0.0f;
  for (int q = q0; q - lane < so; q += kStep) {
    const float4 f = sf4[lo + min(q, so - 1)];
    float m1 = __int_as_float(0x7f800000), e = f.w;
#pragma unroll 4
    for (int t = 0; t < si; ++t) {
      const float4 g = __ldg(&sf4[li + t]);
      const float dx = f.x - g.x, dy = f.y - g.y, dz = f.z - g.z;
      m1 = fminf(m1, fmaf(dz, dz, fmaf(dy, dy, dx * dx)));
      e = fmaxf(e, g.w);
    }
    mine = fminf(mine, fminf(m1, 3e38f));  // (an overflow or NaN counts as 3e38)
    em = fmaxf(em, e);
  }
  const int wm = __reduce_min_sync(0xffffffffu, __float_as_int(mine));  // non-negative floats
  const int we = __reduce_max_sync(0xffffffffu, __float_as_int(em));
  if (lane == 0) {
    atomicMin(&s_min, wm);
    atomicMax(&s_emax, we);
  }
  __syncthreads();
  NearestScan ns;
  ns.m1 = __int_as_float(s_min);
  const float lim = ns.limit(2.0f * __int_as_float(s_emax));  // e_i + e_j is at most twice the largest
  DcEdge best{~0ull, INT_MAX, INT_MAX};
  const double *X = sx, *Y = sx + n, *Z = sx + 2 * (size_t)n;
  for (unsigned todo = __ballot_sync(0xffffffffu, mine <= lim); todo; todo &= todo - 1) {
    const int l = __ffs(todo) - 1;
    for (int q = q0 - lane + l; q < so; q += kStep) {  // that lane's bodies, over the warp
      const float4 f = sf4[lo + q];
      for (int t = lane; t < si; t += 32) {
        const float4 g = sf4[li + t];
        const float dx = f.x - g.x, dy = f.y - g.y, dz = f.z - g.z;
        if (fmaf(dz, dz, fmaf(dy, dy, dx * dx)) > lim) continue;
        const int pi = swap ? lo + q : li + t, pj = swap ? li + t : lo + q;
        const double ex = __dsub_rn(X[pi], X[pj]), ey = __dsub_rn(Y[pi], Y[pj]), ez = __dsub_rn(Z[pi], Z[pj]);
        const DcEdge c{key_bits(__dadd_rn(__dadd_rn(__dmul_rn(ex, ex), __dmul_rn(ey, ey)), __dmul_rn(ez, ez))),
                       (int)(sorted[pi] & kIdxMask), (int)(sorted[pj] & kIdxMask)};
        if (dc_less(c, best)) best = c;
      }
    }
  }
  if (__any_sync(0xffffffffu, best.d != ~0ull)) {
    for (int o = 16; o > 0; o >>= 1) {
      DcEdge c;
      c.d = __shfl_xor_sync(0xffffffffu, best.d, o);
      c.i = __shfl_xor_sync(0xffffffffu, best.i, o);
      c.j = __shfl_xor_sync(0xffffffffu, best.j, o);
      if (dc_less(c, best)) best = c;
    }
  }
  if (lane == 0) red[warp] = best;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < kMetaT / 32; ++w)
      if (dc_less(red[w], best)) best = red[w];
    W[((size_t)z * mc + a) * mc + b] = best;
  }
}

// The shares' weights folded into the first share's table.
__global__ void __launch_bounds__(256) k_dc_meta_fold(const int* __restrict__ ncell, int mc, DcEdge* W) {
  const int nc = *ncell, k = blockIdx.x * 256 + threadIdx.x;
  const int a = k / mc, b = k - a * mc;
  if (a >= nc || b >= nc || b <= a) return;
  DcEdge e = W[(size_t)a * mc + b];
  for (int z = 1; z < kMetaZ; ++z) {
    const DcEdge c = W[((size_t)z * mc + a) * mc + b];
    if (dc_less(c, e)) e = c;
  }
  W[(size_t)a * mc + b] = e;
}

// MST of the meta-graph, by Boruvka rounds in one CTA: the weights (d^2, i, j) are distinct triples,
// so the tree is unique whatever the order, and equals that of Prim from subgraph 0, whose one
// warp took 197 us for 104 subgraphs at N = 10002; 30 now. Its edges go after the n - ncell local
// ones.
__global__ void __launch_bounds__(1024, 1)
k_dc_meta_mst(int n, const int* __restrict__ ncell, int mc, const DcEdge* __restrict__ W, int* __restrict__ eu,
              int* __restrict__ ev) {
  constexpr int M = kDcMaxSub + 8;
  __shared__ DcEdge key[M];        // cheapest edge out of each subgraph's component
  __shared__ short far_[M];        // the subgraph at its far end
  __shared__ short comp[M], pick[M], nxt[M];
  __shared__ int s_edges;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nc = *ncell;
  for (int g = tid; g < nc; g += 1024) comp[g] = (short)g;
  if (tid == 0) s_edges = 0;
  __syncthreads();
  for (int round = 0; round < 16; ++round) {  // components at least halve
    if (s_edges >= nc - 1) break;
    for (int g = warp; g < nc; g += 32) {
      const int cg = comp[g];
      DcEdge b{~0ull, INT_MAX, INT_MAX};
      int bh = -1;
      for (int h0 = lane; h0 < nc; h0 += 128) {
        DcEdge e[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          const int h = h0 + 32 * t;
          const bool in = h < nc && comp[h] != cg;
          e[t] = in ? (g < h ? W[(size_t)g * mc + h] : W[(size_t)h * mc + g]) : DcEdge{~0ull, INT_MAX, INT_MAX};
        }
#pragma unroll
        for (int t = 0; t < 4; ++t)
          if (dc_less(e[t], b)) {
            b = e[t];
            bh = h0 + 32 * t;
          }
      }
      for (int o = 16; o > 0; o >>= 1) {
        DcEdge c;
        c.d = __shfl_xor_sync(0xffffffffu, b.d, o);
        c.i = __shfl_xor_sync(0xffffffffu, b.i, o);
        c.j = __shfl_xor_sync(0xffffffffu, b.j, o);
        const int h2 = __shfl_xor_sync(0xffffffffu, bh, o);
        if (dc_less(c, b)) {
          b = c;
          bh = h2;
        }
      }
      if (lane == 0) {
        key[g] = b;
        far_[g] = (short)bh;
      }
    }
    __syncthreads();
    for (int c = tid; c < nc; c += 1024) {
      if (comp[c] != c) continue;
      int p = -1;
      for (int g = 0; g < nc; ++g)
        if (comp[g] == c && far_[g] >= 0 && (p < 0 || dc_less(key[g], key[p]))) p = g;
      pick[c] = (short)p;
    }
    __syncthreads();
    for (int c = tid; c < nc; c += 1024) {
      if (comp[c] != c) continue;
      const int p = pick[c];
      if (p < 0) {
        nxt[c] = (short)c;
        continue;
      }
      const int t = comp[far_[p]], pt = pick[t];
      const bool mutual = pt >= 0 && comp[far_[pt]] == c;
      nxt[c] = (short)(mutual && c < t ? c : t);
      if (!mutual || c < t) {
        const int k = atomicAdd(&s_edges, 1);
        if (k < nc - 1) {
          eu[n - nc + k] = key[p].i;
          ev[n - nc + k] = key[p].j;
        }
      }
    }
    __syncthreads();
    int to[(M + 1023) / 1024];
    int q = 0;
    for (int g = tid; g < nc; g += 1024, ++q) {
      int c = comp[g];
      for (int guard = 0; guard < nc && nxt[c] != c; ++guard) c = nxt[c];
      to[q] = c;
    }
    __syncthreads();
    q = 0;
    for (int g = tid; g < nc; g += 1024, ++q) comp[g] = (short)to[q];
    __syncthreads();
  }
}

// The breadth-first walk of the tree in one warp: the queue is the order. A level's vertices are
// taken 32 at a time, one per lane; every lane appends its children (ascending) after those of the
// lanes before it.
__global__ void __launch_bounds__(32)
k_bfs_order(int n, const int* __restrict__ root, const int* __restrict__ child_off, const int* __restrict__ child_idx,
            int* order) {
  const int lane = threadIdx.x;
  if (lane == 0) order[0] = root[0];
  __syncwarp();
  int tail = 1;
  for (int h = 0; h < tail && h < n;) {
    const int t = min(tail, h + 32);  // vertices appended before this pass, in queue order
    const int v = h + lane < t ? order[h + lane] : -1;
    const int c0 = v >= 0 ? child_off[v] : 0, cnt = v >= 0 ? child_off[v + 1] - c0 : 0;
    int incl = cnt;
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    const int at = tail + incl - cnt;
    for (int k = 0; k < cnt; ++k)
      if (at + k < n) order[at + k] = child_idx[c0 + k];
    tail += __shfl_sync(0xffffffffu, incl, 31);
    h = t;
    __syncwarp();  // this pass's appends are read by the next
  }
}

}  // namespace

size_t dc_scratch_bytes(int n, int nsub) { return dc_layout(n, nsub, nullptr).bytes; }

cudaError_t launch_mst_dc(mstar_ctx* c) {
  const int n = c->n;
  if (!c->d.dc) return cudaErrorInvalidValue;
  const DcLayout L = dc_layout(n, c->p.mst_nsub, c->d.dc);
  const int target = target_of(n, c->p.mst_nsub);
  const double* X = c->d.r;
  const double* Y = X + c->npad;
  const double* Z = Y + c->npad;
  cudaStream_t s = c->stream;
  const int nb = (n + 255) / 256;
  k_dc_bounds<<<kDcBoundCtas, 256, 0, s>>>(n, X, Y, Z, L.bounds);
  k_dc_keys<<<nb, 256, 0, s>>>(n, X, Y, Z, L.bounds, L.keys, L.f4);
  k_dc_rank<<<dim3((n + 127) / 128, kDcParts), 128, 0, s>>>(n, L.keys, L.rank);
  k_dc_place<<<(std::max(n, L.mc) + 255) / 256, 256, 0, s>>>(n, L.mc, L.keys, L.rank, X, Y, Z, L.f4, L.sorted, L.sx,
                                                             L.sf4, L.comp, L.nbr, L.lcount, L.flags);
  const size_t psmem = 8 * (size_t)n;
  cudaError_t e = cudaFuncSetAttribute(k_dc_partition, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)psmem);
  if (e != cudaSuccess) return e;
  k_dc_partition<<<1, 1024, psmem, s>>>(n, target, L.mc, L.sorted, L.ncell, L.leafid, L.leaf_start);
  k_dc_meta_w<<<dim3(L.mc * (L.mc - 1) / 2, kMetaZ), kMetaT, 0, s>>>(n, L.ncell, L.mc, L.leaf_start, L.sorted, L.sx,
                                                                     L.sf4, L.W);
  k_dc_meta_fold<<<(L.mc * L.mc + 255) / 256, 256, 0, s>>>(L.ncell, L.mc, L.W);
  k_dc_meta_mst<<<1, 1024, 0, s>>>(n, L.ncell, L.mc, L.W, L.eu, L.ev);
  c->launches += 8;
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  // the subgraphs' trees: as many rounds as the context's last build ran before the first check of
  // the edge count, then one at a time; Prim's kernel on a tie
  bool tied = false;
  int ncell = 0, edges = -1;
  for (int round = 0; round < 64 && !tied && edges < n - ncell;) {
    const int batch = round == 0 ? (c->mst_rounds > 0 ? c->mst_rounds : 1) : 1;
    for (int k = 0; k < batch; ++k, ++round) {
      k_dc_nfn<<<dim3((n + kDcT - 1) / kDcT, kDcParts), kDcT, 0, s>>>(n, L.ncell, L.leafid, L.leaf_start, L.sx, L.sf4,
                                                                      L.comp, L.nbr, L.lcount, L.partD, L.partJ,
                                                                      L.flags);
      k_dc_round<<<L.mc, kDcRoundT, 0, s>>>(n, L.ncell, L.leaf_start, L.sorted, L.comp, L.nbr, L.nbrD, L.cidx, L.nxt,
                                      L.partD, L.partJ, L.key, L.lcount, L.eu, L.ev, L.flags);
      c->launches += 2;
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    int* h = reinterpret_cast<int*>(c->host_buf);
    if ((e = cudaMemcpyAsync(h, L.flags, sizeof(int) * 4, cudaMemcpyDeviceToHost, s)) != cudaSuccess) return e;
    if ((e = cudaMemcpyAsync(h + 4, L.ncell, sizeof(int), cudaMemcpyDeviceToHost, s)) != cudaSuccess) return e;
    if ((e = cudaStreamSynchronize(s)) != cudaSuccess) return e;
    int fl[5];
    std::memcpy(fl, h, sizeof(fl));
    tied = fl[0] != 0;
    edges = fl[1];
    c->mst_rounds = fl[3];
    ncell = fl[4];
  }
  if (tied || edges != n - ncell) {
    const size_t lsmem =
        (size_t)kLeafSmem * (3 * sizeof(double) + 8 + sizeof(float4) + sizeof(float) + 2 * sizeof(int));
    if ((e = cudaFuncSetAttribute(k_dc_local_prim, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)lsmem)) !=
        cudaSuccess)
      return e;
    k_dc_local_prim<<<L.mc, kLpThreads, lsmem, s>>>(L.ncell, L.leaf_start, L.sorted, X, Y, Z, L.f4, L.key, L.keyf,
                                                     L.kp, L.eu, L.ev);
    MSTAR_LAUNCHED(c);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  return launch_orient(c, L.eu, L.ev);
}

// d.order of a divide-and-conquer tree, from the children lists of launch_tree; only a caller that
// asks for the order (mstar_get_mst) needs it.
cudaError_t launch_bfs_order(mstar_ctx* c) {
  k_bfs_order<<<1, 32, 0, c->stream>>>(c->n, c->d.root, c->d.child_off, c->d.child_idx, c->d.order);
  MSTAR_LAUNCHED(c);
  return cudaGetLastError();
}

}  // namespace mstar
