// The rebuild test of Sec. 3.5 on the GPU: for each job (one system, one coordinate system,
// one deconstruction rule) repeat, `cycles` times, building the relative coordinates from
// the Cartesian state and deconstructing them back, and record the energy at given cycles.
//
// One thread-block cluster per job; every CTA of it holds the whole state, the edge vectors and
// the tree in shared memory.
// - coordinate systems: the MST (Prim, Sec. 3.2, root closest to the centre of mass) or the
//   chain (Sec. 2.2: the shortest pair first, then the particle closest to either end, the
//   tail on a tie), written as a path tree rooted at the tail;
// - building: X_v = w_v - w_parent(v) (0 at the root);
// - deconstruction: per-vertex path sums X_v + X_parent(v) + ... up to the root, then either
//   the centre-of-mass shift (as the integrator's rebuild) or the root's kept position; or
//   from the root outwards (w_v = w_parent(v) + X_v, parents first) with the root kept, then
//   optionally the centre-of-mass shift;
// - the topology is rebuilt every `topo_every` cycles and compared with the previous one;
// - energies E = T - U with Neumaier-compensated sums of the FP64 terms in index order.
// Every operation is the CPU definition's, in its order, so the results are bit-identical to it.
//
// What bounds it is FP64 latency: a dependent addition takes about 62 cycles, and an SM issues one
// FP64 warp instruction per 16 cycles however few lanes it has. So
// - the path sums (N <L> additions per component: half of N^2 for the chain) are dealt out over
//   the cluster's SMs, 32 bodies of about equal level and one component per warp, and written
//   into every CTA's copy of the state (distributed shared memory);
// - the sums that are sequential by definition run in lockstep lanes of one warp: the six
//   components' centre-of-mass sums, and the two chains of a compensated sum (the sum itself and,
//   a chunk behind it, the sum of its rounding errors, which the other warps form from the
//   recorded partial sums);
// - rules 2 and 3 need no cluster: a chain is one running sum per component, a tree goes level
//   by level in one warp per component.
// N = 379, eight jobs (both coordinate systems, all rules), 1000 cycles and two energies: 456 ms
// with one CTA per job and one thread for each sequential sum, 49 ms now. A cycle of the slowest
// jobs, the chain's with the shift, takes 33-37 us (rules 0 and 3; 428 and 242 before): 378
// dependent additions twice over, at 80-100 cycles each. Tree cycles take 5-22 us, an energy
// 3.3 ms (13.5 before), a build 0.5 ms (tree) or 1.1 ms (chain).
#include <climits>
#include <cmath>
#include <new>

#include <cooperative_groups.h>

#include "device.cuh"
#include "internal.h"

namespace mstar {
namespace {

constexpr int kRbThreads = 512;

struct RbArgs {
  int n, cycles, topo_every, nsample;
  const int* sample_at;
  const double *m, *r, *v;  // per job: n, 3n, 3n
  const int *coords, *decon;
  double *E_out, *r_out, *v_out, *mean_level;
  int* topo_changes;
};

__device__ __forceinline__ double norm2_of(const double* x) {
  return __dadd_rn(__dadd_rn(__dmul_rn(x[0], x[0]), __dmul_rn(x[1], x[1])), __dmul_rn(x[2], x[2]));
}

__device__ __forceinline__ double w2_of(const double* r, int u, int v) {
  const double dx = __dsub_rn(r[3 * u], r[3 * v]), dy = __dsub_rn(r[3 * u + 1], r[3 * v + 1]),
               dz = __dsub_rn(r[3 * u + 2], r[3 * v + 2]);
  return __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
}

struct Neu {
  double s, c;
};

// Lexicographic minimum (key bits, a, b) over the CTA; every thread gets the result.
struct Arg3 {
  unsigned long long k;
  int a, b;
};

__device__ __forceinline__ bool arg3_less(const Arg3& x, const Arg3& y) {
  if (x.k != y.k) return x.k < y.k;
  if (x.a != y.a) return x.a < y.a;
  return x.b < y.b;
}

// The warp's minimum, in every lane: the key's two halves and the indices one after another.
__device__ __forceinline__ Arg3 warp_argmin(Arg3 v) {
  const unsigned kh = (unsigned)(v.k >> 32), mh = __reduce_min_sync(0xffffffffu, kh);
  bool in = kh == mh;
  const unsigned ml = __reduce_min_sync(0xffffffffu, in ? (unsigned)v.k : 0xffffffffu);
  in &= (unsigned)v.k == ml;
  const int ma = __reduce_min_sync(0xffffffffu, in ? v.a : INT_MAX);
  in &= v.a == ma;
  const int mb = __reduce_min_sync(0xffffffffu, in ? v.b : INT_MAX);
  return Arg3{((unsigned long long)mh << 32) | ml, ma, mb};
}

// red: 2 x kRbThreads / 32 entries; consecutive calls alternate `half` (one barrier per call).
__device__ Arg3 cta_argmin(Arg3 v, Arg3* red, int half) {
  constexpr int NW = kRbThreads / 32;
  red += half * NW;
  v = warp_argmin(v);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  const int lane = threadIdx.x & 31;
  return warp_argmin(lane < NW ? red[lane] : Arg3{~0ull, INT_MAX, INT_MAX});
}

// Compensated sum of `count` non-negative terms in index order, by the whole CTA; the result in
// every thread. Chunk by chunk (kNeuChunk terms, one per thread of warps 1 ...): in phase p those
// warps form the terms of chunk p + 1 and the rounding errors of chunk p - 1 (from its recorded
// partial sums), while warp 0 adds chunk p's terms in lane 0 and chunk p - 2's errors in lane 1:
// one dependent addition per term. Short chunks are filled with zeros, which change nothing.
constexpr int kNeuChunk = kRbThreads - 32;
constexpr int kNeuBuf = 7 * kNeuChunk;

template <typename Term>
__device__ Neu neumaier_cta(int count, double* buf, double* s_out, Term term) {
  double* xs = buf;                      // 3 chunks of terms
  double* ts = xs + 3 * kNeuChunk;       // 2 chunks of partial sums
  double* es = ts + 2 * kNeuChunk;       // 2 chunks of errors
  __shared__ double s_start[4];          // the sum before chunk p (p mod 4)
  const int tid = threadIdx.x, q = tid - 32;
  const int nch = (count + kNeuChunk - 1) / kNeuChunk;
  if (q >= 0) xs[q] = q < count ? term(q) : 0.0;
  double acc = 0.0;  // lane 0: the sum; lane 1: the sum of the errors
  __syncthreads();
  for (int p = 0; p < nch + 2; ++p) {
    if (tid < 32) {
      if (tid == 0) s_start[p & 3] = acc;
      const bool go = tid == 0 ? p < nch : (tid == 1 && p >= 2);
      const double* src = tid == 0 ? xs + (p % 3) * kNeuChunk : es + (p & 1) * kNeuChunk;
      double* dst = ts + (p & 1) * kNeuChunk;
      if (go) {
        // eight at a time; the partial sums are stored after the eight additions, each of which
        // would otherwise wait for the store before it
        for (int k = 0; k < kNeuChunk; k += 8) {
          double x[8];
#pragma unroll
          for (int j = 0; j < 8; ++j) x[j] = src[k + j];
#pragma unroll
          for (int j = 0; j < 8; ++j) x[j] = acc = __dadd_rn(acc, x[j]);
          asm volatile("" ::: "memory");
          if (tid == 0) {
#pragma unroll
            for (int j = 0; j < 8; ++j) dst[k + j] = x[j];
          }
        }
      }
    } else {
      if (p + 1 < nch) {
        const int g = (p + 1) * kNeuChunk + q;
        xs[((p + 1) % 3) * kNeuChunk + q] = g < count ? term(g) : 0.0;
      }
      if (p >= 1 && p <= nch) {
        const double* t = ts + ((p - 1) & 1) * kNeuChunk;
        const double x = xs[((p - 1) % 3) * kNeuChunk + q], tk = t[q];
        const double s = q ? t[q - 1] : s_start[(p - 1) & 3];
        const bool big = fabs(s) >= fabs(x);
        es[((p - 1) & 1) * kNeuChunk + q] = __dadd_rn(__dsub_rn(big ? s : x, tk), big ? x : s);
      }
    }
    __syncthreads();
  }
  if (tid < 2) s_out[tid] = acc;
  __syncthreads();
  const Neu r{s_out[0], s_out[1]};
  __syncthreads();
  return r;
}

// E = T - U with compensated sums, the terms and the order of the CPU definition (U over the
// pairs i < j, row by row).
__device__ double energy_comp(int n, const double* m, const double* r, const double* v, double* buf, double* s_out) {
  const Neu T = neumaier_cta(n, buf, s_out, [&](int i) {
    return __dmul_rn(0.5, __dmul_rn(m[i], norm2_of(v + 3 * i)));
  });
  const Neu U = neumaier_cta(n * (n - 1) / 2, buf, s_out, [&](int q) {
    int i, j;
    tile_pair(q, n - 1, i, j);  // rows of n - 1 - i pairs
    return __ddiv_rn(__dmul_rn(1.0, __dmul_rn(m[i], m[j + 1])), __dsqrt_rn(w2_of(r, i, j + 1)));
  });
  return __dsub_rn(__dadd_rn(T.s, T.c), __dadd_rn(U.s, U.c));
}

// Prim's MST (exact keys; root closest to the origin, lowest index on ties).
__device__ void cta_prim(int n, const double* r, int* parent, int* level, int* order, unsigned long long* key,
                         unsigned char* in, Arg3* red) {
  Arg3 b{~0ull, INT_MAX, 0};
  for (int i = threadIdx.x; i < n; i += kRbThreads) {
    const Arg3 c{key_bits(norm2_of(r + 3 * i)), i, 0};
    if (arg3_less(c, b)) b = c;
    key[i] = 0x7ff0000000000000ull;
    parent[i] = -1;
    in[i] = 0;
  }
  b = cta_argmin(b, red, 0);
  const int root = b.a;
  __syncthreads();
  if (threadIdx.x == 0) {
    in[root] = 1;
    level[root] = 0;
    order[0] = root;
  }
  __syncthreads();
  int u = root;
  for (int it = 1; it < n; ++it) {
    b = Arg3{~0ull, INT_MAX, 0};
    for (int w = threadIdx.x; w < n; w += kRbThreads) {
      if (in[w]) continue;
      const unsigned long long d = key_bits(w2_of(r, u, w));
      if (d < key[w]) {
        key[w] = d;
        parent[w] = u;
      }
      const Arg3 c{key[w], w, 0};
      if (arg3_less(c, b)) b = c;
    }
    b = cta_argmin(b, red, it & 1);
    u = b.a;
    if (threadIdx.x == 0) {
      in[u] = 1;
      order[it] = u;
      if (parent[u] < 0) parent[u] = root;
      level[u] = level[parent[u]] + 1;
    }
    __syncthreads();
  }
}

// The chain as a path tree rooted at its tail.
__device__ void cta_chain(int n, const double* r, int* parent, int* level, int* order, int* dq, unsigned char* in,
                          Arg3* red) {
  // the shortest pair (lowest (i, j) on ties)
  Arg3 b{~0ull, INT_MAX, INT_MAX};
  for (int i = 0; i < n - 1; ++i)
    for (int j = i + 1 + threadIdx.x; j < n; j += kRbThreads) {
      const Arg3 c{key_bits(w2_of(r, i, j)), i, j};
      if (arg3_less(c, b)) b = c;
    }
  for (int i = threadIdx.x; i < n; i += kRbThreads) in[i] = 0;
  b = cta_argmin(b, red, 0);
  __shared__ int s_lo, s_hi;
  if (threadIdx.x == 0) {
    s_lo = n;
    s_hi = n + 1;
    dq[n] = b.a;
    dq[n + 1] = b.b;
    in[b.a] = 1;
    in[b.b] = 1;
  }
  __syncthreads();
  for (int added = 2; added < n; ++added) {
    const int tail = dq[s_lo], head = dq[s_hi];
    Arg3 c0{~0ull, INT_MAX, 0};
    for (int p = threadIdx.x; p < n; p += kRbThreads) {
      if (in[p]) continue;
      const double dt = w2_of(r, p, tail), dh = w2_of(r, p, head);
      const int end = dh < dt ? 1 : 0;
      const Arg3 c{key_bits(end ? dh : dt), p, end};
      if (arg3_less(c, c0)) c0 = c;
    }
    c0 = cta_argmin(c0, red, added & 1);
    if (threadIdx.x == 0) {
      in[c0.a] = 1;
      if (c0.b) dq[++s_hi] = c0.a;
      else dq[--s_lo] = c0.a;
    }
    __syncthreads();
  }
  for (int k = threadIdx.x; k < n; k += kRbThreads) {
    const int p = dq[s_lo + k];
    order[k] = p;
    parent[p] = k ? dq[s_lo + k - 1] : -1;
    level[p] = k;
  }
  __syncthreads();
}

// The edge vectors of r and v: six planes of n in path order for the chain (the path's k-th edge,
// 0 for the root), else two n x 3 arrays by body.
__device__ void edge_vectors(int n, int coords, const int* parent, const int* bylev, const double* r, const double* v,
                             double* X) {
  if (coords == 1) {
    for (int t = threadIdx.x; t < 6 * n; t += kRbThreads) {
      const int c = t / n, k = t - c * n;
      const double* w = c < 3 ? r + c : v + (c - 3);
      X[t] = k ? __dsub_rn(w[3 * bylev[k]], w[3 * bylev[k - 1]]) : 0.0;
    }
    return;
  }
  for (int t = threadIdx.x; t < 6 * n; t += kRbThreads) {
    const int h = t < 3 * n ? 0 : 3 * n, i = (t - h) / 3, k = (t - h) - 3 * i;
    const double* w = h ? v : r;
    const int p = parent[i];
    X[t] = p < 0 ? 0.0 : __dsub_rn(w[3 * i + k], w[3 * p + k]);
  }
}

// Deconstruction of r and v from the edge vectors by per-vertex path sums (rules 0 and 1, without
// the shift): the groups of 32 bodies in level order (bylev) times the six components, one per
// warp, dealt out over the cluster; each result goes to every CTA's copy. The chain's sums run
// down the path's planes, so that no parent has to be looked up on the way.
template <int C>
__device__ void cluster_path_sums(int n, int coords, const int* parent, const int* bylev, const double* X, double* r,
                                  double* v, int decon, int rank) {
  namespace cg = cooperative_groups;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int groups = (n + 31) >> 5, root = bylev[0];
  // the deepest groups first
  for (int t = rank + C * warp; t < 6 * groups; t += C * (kRbThreads / 32)) {
    const int g = groups - 1 - t / 6, c = t - (t / 6) * 6;
    double* w = c < 3 ? r + c : v + (c - 3);
    const int k = 32 * g + lane;
    const int b = k < n ? bylev[k] : root;
    double s = 0.0;
    if (coords == 1) {
      const double* W = X + (size_t)c * n;
      int j = k < n ? k : 0;
      for (; j >= 8; j -= 8) {
        double x[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) x[q] = W[j - q];
#pragma unroll
        for (int q = 0; q < 8; ++q) s = __dadd_rn(s, x[q]);
      }
      for (; j >= 1; --j) s = __dadd_rn(s, W[j]);
    } else {
      const double* W = c < 3 ? X + c : X + 3 * n + (c - 3);
      for (int u = b; parent[u] >= 0; u = parent[u]) s = __dadd_rn(s, W[3 * u]);
    }
    // the root's kept position: other bodies' entries of this CTA's copy may already be written, the
    // root's is written only after the barrier that follows
    if (decon == 1) s = __dadd_rn(s, w[3 * root]);
    if (k < n && b != root) {
      if constexpr (C > 1) {
#pragma unroll
        for (int q = 0; q < C; ++q) cg::this_cluster().map_shared_rank(w, q)[3 * b] = s;
      } else {
        w[3 * b] = s;
      }
    }
  }
}

// From the root outwards, w_v = w_parent(v) + W_v with the root kept (rules 2 and 3, without the
// shift). The chain is one running sum per component, in six lanes of a warp, over the path's
// planes; a tree goes level by level, warp c < 6 taking component c and its lanes a level's bodies.
// Every thread of the CTA calls it (it holds a barrier for the chain).
__device__ void outward_sums(int n, int coords, const int* parent, const int* level, const int* bylev, double* X,
                             double* r, double* v) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (coords == 1) {
    if (threadIdx.x < 6) {
      const int c = threadIdx.x;
      double* W = X + (size_t)c * n;
      double s = c < 3 ? r[3 * bylev[0] + c] : v[3 * bylev[0] + c - 3];
      W[0] = s;
      int k = 1;
      for (; k + 8 <= n; k += 8) {
        double x[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) x[j] = W[k + j];
#pragma unroll
        for (int j = 0; j < 8; ++j) x[j] = s = __dadd_rn(s, x[j]);
        asm volatile("" ::: "memory");  // the stores after the eight additions
#pragma unroll
        for (int j = 0; j < 8; ++j) W[k + j] = x[j];
      }
      for (; k < n; ++k) W[k] = s = __dadd_rn(s, W[k]);
    }
    __syncthreads();
    for (int t = threadIdx.x; t < 6 * n; t += kRbThreads) {
      const int c = t / n, b = bylev[t - c * n];
      (c < 3 ? r + c : v + (c - 3))[3 * b] = X[t];
    }
    return;
  }
  if (warp >= 6) return;
  const double* W = warp < 3 ? X + warp : X + 3 * n + (warp - 3);
  double* w = warp < 3 ? r + warp : v + (warp - 3);
  for (int k = 1; k < n;) {
    const int l = level[bylev[k]];
    const int b = k + lane < n ? bylev[k + lane] : -1;
    const unsigned in = __ballot_sync(0xffffffffu, b >= 0 && level[b >= 0 ? b : 0] == l);
    if ((in >> lane) & 1u) w[3 * b] = __dadd_rn(w[3 * parent[b]], W[3 * b]);
    __syncwarp();
    k += __popc(in);  // the level's bodies are consecutive: its first lanes
  }
}

// w -= (sum m w) / M for r and v, with the sums in index order. M is the sum of the masses in index
// order. Every thread forms products (into pr, 6 x n), then lane c < 6 of warp 0 adds component c:
// the sums cost one dependent addition per body. The caller synchronises before and after.
__device__ void com_shift(int n, const double* m, double M, double* r, double* v, double* pr, double* sc) {
  for (int t = threadIdx.x; t < 6 * n; t += kRbThreads) {
    const int c = t / n, i = t - c * n;
    pr[t] = __dmul_rn(m[i], c < 3 ? r[3 * i + c] : v[3 * i + c - 3]);
  }
  __syncthreads();
  if (threadIdx.x < 32) {
    const double* p = pr + (size_t)(threadIdx.x < 6 ? threadIdx.x : 5) * n;
    double s = 0.0, x[8], y[8];
    const int nb = n >> 3;  // blocks of eight, each loaded while the one before is added
#pragma unroll
    for (int j = 0; j < 8; ++j) x[j] = nb ? p[j] : 0.0;
    for (int k = 0; k < nb; ++k) {
#pragma unroll
      for (int j = 0; j < 8; ++j) y[j] = k + 1 < nb ? p[8 * (k + 1) + j] : 0.0;
#pragma unroll
      for (int j = 0; j < 8; ++j) s = __dadd_rn(s, x[j]);
#pragma unroll
      for (int j = 0; j < 8; ++j) x[j] = y[j];
    }
    for (int i = 8 * nb; i < n; ++i) s = __dadd_rn(s, p[i]);
    if (threadIdx.x < 6) sc[threadIdx.x] = __ddiv_rn(s, M);
  }
  __syncthreads();
  for (int t = threadIdx.x; t < 3 * n; t += kRbThreads) {
    const int c = t % 3;
    r[t] = __dsub_rn(r[t], sc[c]);
    v[t] = __dsub_rn(v[t], sc[3 + c]);
  }
}

template <int C>
__global__ void __launch_bounds__(kRbThreads, 2) k_rebuild_jobs(RbArgs A) {
  namespace cg = cooperative_groups;
  extern __shared__ double smem[];
  __shared__ Arg3 red[2 * (kRbThreads / 32)];
  __shared__ double sc[8], s_M;
  const int job = blockIdx.x / C, rank = blockIdx.x - (blockIdx.x / C) * C, n = A.n;
  const int coords = A.coords[job], decon = A.decon[job];
  // rules 2 and 3 run on the first CTA alone: no CTA of their clusters waits for another
  if (decon >= 2 && rank > 0) return;
  double* m = smem;
  double* r = m + n;
  double* v = r + 3 * n;
  double* X = v + 3 * n;  // edge vectors, 6 n
  double* buf = X + 6 * n;
  unsigned long long* key = reinterpret_cast<unsigned long long*>(buf + kNeuBuf);
  int* parent = reinterpret_cast<int*>(key + n);
  int* prev = parent + n;
  int* level = prev + n;
  int* order = level + n;
  int* bylev = order + n;
  int* dq = bylev + n;                                 // 2n + 2
  unsigned char* in = reinterpret_cast<unsigned char*>(dq + 2 * n + 2);
  for (int i = threadIdx.x; i < n; i += kRbThreads) m[i] = A.m[(size_t)job * n + i];
  for (int t = threadIdx.x; t < 3 * n; t += kRbThreads) {
    r[t] = A.r[(size_t)job * 3 * n + t];
    v[t] = A.v[(size_t)job * 3 * n + t];
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double M = 0.0;
    for (int i = 0; i < n; ++i) M = __dadd_rn(M, m[i]);
    s_M = M;
  }
  __syncthreads();
  const double M = s_M;
  int s = 0, changes = 0, builds = 0;
  double lsum = 0.0;
  double* E = A.E_out + (size_t)job * A.nsample;
  auto samples = [&](int c) {  // every CTA keeps count, the first one evaluates
    while (s < A.nsample && A.sample_at[s] == c) {
      if (rank == 0) {
        const double e = energy_comp(n, m, r, v, buf, sc + 6);
        if (threadIdx.x == 0) E[s] = e;
      }
      ++s;
    }
  };
  samples(0);
  for (int c = 1; c <= A.cycles; ++c) {
    if ((c - 1) % A.topo_every == 0) {
      if (coords == 0) cta_prim(n, r, parent, level, order, key, in, red);
      else cta_chain(n, r, parent, level, order, dq, in, red);
      __syncthreads();
      int diff = 0, lev = 0;
      for (int i = threadIdx.x; i < n; i += kRbThreads) {
        diff |= parent[i] != prev[i];
        prev[i] = parent[i];
        lev += level[i];
        // rank in order of (level, index)
        int k = 0;
        const int li = level[i];
        for (int u = 0; u < n; ++u) k += level[u] < li || (level[u] == li && u < i);
        bylev[k] = i;
      }
      diff = __syncthreads_or(diff);
      if (builds && diff) ++changes;
      lev = __reduce_add_sync(0xffffffffu, lev);
      if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5].a = lev;
      __syncthreads();
      if (threadIdx.x == 0)  // whole numbers: exact in any order
        for (int w = 0; w < kRbThreads / 32; ++w) lsum += red[w].a;
      ++builds;
      __syncthreads();
    }
    edge_vectors(n, coords, parent, bylev, r, v, X);
    if (decon >= 2) {
      __syncthreads();
      outward_sums(n, coords, parent, level, bylev, X, r, v);
    } else {
      // every CTA has read its copy before another writes into it
      if constexpr (C > 1) cg::this_cluster().sync();
      else __syncthreads();
      cluster_path_sums<C>(n, coords, parent, bylev, X, r, v, decon, rank);
      if constexpr (C > 1) cg::this_cluster().sync();
      else __syncthreads();
      // the root's path sum is empty; with the root kept it stays 0 + its position
      if (threadIdx.x < 6) {
        double* w = threadIdx.x < 3 ? r + threadIdx.x : v + (threadIdx.x - 3);
        const int o = 3 * bylev[0];
        w[o] = decon == 0 ? 0.0 : __dadd_rn(0.0, w[o]);
      }
    }
    __syncthreads();
    if (decon == 0 || decon == 3) {
      com_shift(n, m, M, r, v, X, sc);  // (the edge vectors, 6 n doubles, are free again)
      __syncthreads();
    }
    samples(c);
  }
  __syncthreads();
  // no CTA leaves while another may still write into its copy: the last barrier of the last cycle
  // follows every such write
  if (rank > 0) return;
  for (int t = threadIdx.x; t < 3 * n; t += kRbThreads) {
    A.r_out[(size_t)job * 3 * n + t] = r[t];
    A.v_out[(size_t)job * 3 * n + t] = v[t];
  }
  if (threadIdx.x == 0) {
    A.topo_changes[job] = changes;
    A.mean_level[job] = builds ? lsum / ((double)builds * n) : 0.0;
  }
}

size_t rb_smem(int n) {
  return sizeof(double) * (size_t)(13 * n + kNeuBuf) + 8 * (size_t)n + sizeof(int) * (size_t)(5 * n + 2 * n + 2) +
         (size_t)n + 16;
}

// A launch of njobs clusters of C CTAs, and how many of them the device can hold at once (0: none).
template <int C>
cudaError_t rb_config(int njobs, size_t smem, cudaStream_t st, cudaLaunchConfig_t* cfg, cudaLaunchAttribute* attr,
                      int* resident) {
  *cfg = {};
  cfg->gridDim = dim3(njobs * C);
  cfg->blockDim = dim3(kRbThreads);
  cfg->dynamicSmemBytes = smem;
  cfg->stream = st;
  attr->id = cudaLaunchAttributeClusterDimension;
  attr->val.clusterDim.x = C;
  attr->val.clusterDim.y = 1;
  attr->val.clusterDim.z = 1;
  cfg->attrs = attr;
  cfg->numAttrs = 1;
  cudaError_t e = cudaFuncSetAttribute(k_rebuild_jobs<C>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e == cudaSuccess && C > 8) e = cudaFuncSetAttribute(k_rebuild_jobs<C>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) return e;
  *resident = 1;
  if (C > 1 && cudaOccupancyMaxActiveClusters(resident, k_rebuild_jobs<C>, cfg) != cudaSuccess) {
    cudaGetLastError();
    *resident = 0;
  }
  return cudaSuccess;
}

// Launches with clusters of C CTAs if the device can hold them all at once (beyond that the jobs
// would only queue behind one another's centre-of-mass sums), else of C / 2. Clusters of 16 against
// 8: 18 against 24 us for the chain's path sums at N = 379 (an SM's share of the additions, at one
// FP64 warp instruction per 16 cycles, falls to their latency).
template <int C>
cudaError_t rb_launch(int njobs, size_t smem, cudaStream_t st, const RbArgs& A) {
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr;
  int resident = 0;
  const cudaError_t e = rb_config<C>(njobs, smem, st, &cfg, &attr, &resident);
  if (e != cudaSuccess) return e;
  if constexpr (C > 1) {
    if (resident < njobs) return rb_launch<C / 2>(njobs, smem, st, A);
  }
  return cudaLaunchKernelEx(&cfg, k_rebuild_jobs<C>, A);
}

}  // namespace
}  // namespace mstar

extern "C" int mstar_rebuild_test(int njobs, int n, const double* m, const double* r, const double* v,
                                  const int* coords, const int* deconstruct, int cycles, int topo_every, int nsample,
                                  const int* sample_at, double* E_out, double* r_out, double* v_out, int* topo_changes,
                                  double* mean_level, void* cuda_stream) {
  using namespace mstar;
  if (njobs < 1 || n < 2 || n > MSTAR_REBUILD_MAX_N || cycles < 0 || topo_every < 1 || nsample < 0 || !m || !r ||
      !v || !coords || !deconstruct || (nsample && (!sample_at || !E_out)))
    return MSTAR_ERR_INVALID_ARG;
  for (int j = 0; j < njobs; ++j)
    if ((coords[j] != 0 && coords[j] != 1) || deconstruct[j] < 0 || deconstruct[j] > 3)
      return MSTAR_ERR_INVALID_ARG;
  for (int s = 0; s < nsample; ++s)
    if (sample_at[s] < 0 || sample_at[s] > cycles || (s && sample_at[s] < sample_at[s - 1]))
      return MSTAR_ERR_INVALID_ARG;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  const size_t nm = (size_t)njobs * n, n3 = 3 * nm;
  const size_t bytes = sizeof(double) * (nm + 4 * n3 + (size_t)njobs * nsample + 2 * njobs) +
                       sizeof(int) * (size_t)(2 * njobs + nsample + njobs) + 1024;
  char* buf = nullptr;
  if (cudaMalloc(&buf, bytes) != cudaSuccess) {
    cudaGetLastError();
    return MSTAR_ERR_NOMEM;
  }
  size_t off = 0;
  auto take = [&](size_t b) {
    off = (off + 15) & ~size_t(15);
    char* p = buf + off;
    off += b;
    return p;
  };
  RbArgs A{};
  A.n = n;
  A.cycles = cycles;
  A.topo_every = topo_every;
  A.nsample = nsample;
  double* dm = reinterpret_cast<double*>(take(sizeof(double) * nm));
  double* dr = reinterpret_cast<double*>(take(sizeof(double) * n3));
  double* dv = reinterpret_cast<double*>(take(sizeof(double) * n3));
  double* dro = reinterpret_cast<double*>(take(sizeof(double) * n3));
  double* dvo = reinterpret_cast<double*>(take(sizeof(double) * n3));
  double* dE = reinterpret_cast<double*>(take(sizeof(double) * ((size_t)njobs * nsample + 1)));
  double* dml = reinterpret_cast<double*>(take(sizeof(double) * njobs));
  int* dco = reinterpret_cast<int*>(take(sizeof(int) * njobs));
  int* dde = reinterpret_cast<int*>(take(sizeof(int) * njobs));
  int* dsa = reinterpret_cast<int*>(take(sizeof(int) * (nsample + 1)));
  int* dtc = reinterpret_cast<int*>(take(sizeof(int) * njobs));
  int rc = MSTAR_OK;
  auto cp = [&](void* dst, const void* src, size_t b) {
    if (!rc && cudaMemcpyAsync(dst, src, b, cudaMemcpyDefault, st) != cudaSuccess) rc = MSTAR_ERR_CUDA;
  };
  cp(dm, m, sizeof(double) * nm);
  cp(dr, r, sizeof(double) * n3);
  cp(dv, v, sizeof(double) * n3);
  cp(dco, coords, sizeof(int) * njobs);
  cp(dde, deconstruct, sizeof(int) * njobs);
  if (nsample) cp(dsa, sample_at, sizeof(int) * nsample);
  if (!rc) {
    A.m = dm;
    A.r = dr;
    A.v = dv;
    A.coords = dco;
    A.decon = dde;
    A.sample_at = dsa;
    A.E_out = dE;
    A.r_out = dro;
    A.v_out = dvo;
    A.mean_level = dml;
    A.topo_changes = dtc;
    if (rb_launch<16>(njobs, rb_smem(n), st, A) != cudaSuccess) rc = MSTAR_ERR_CUDA;
  }
  if (nsample) cp(E_out, dE, sizeof(double) * (size_t)njobs * nsample);
  if (r_out) cp(r_out, dro, sizeof(double) * n3);
  if (v_out) cp(v_out, dvo, sizeof(double) * n3);
  if (topo_changes) cp(topo_changes, dtc, sizeof(int) * njobs);
  if (mean_level) cp(mean_level, dml, sizeof(double) * njobs);
  if (cudaStreamSynchronize(st) != cudaSuccess && !rc) rc = MSTAR_ERR_CUDA;
  cudaFree(buf);
  return rc;
}
