// mstar_accelerations_noalloc: the Cartesian pair loop for callers that cannot allocate
// device memory.
//
// Some callers must not call cudaMalloc: a sub-integrator embedded in a larger code whose
// memory manager owns the whole device heap (and would see a private allocation as a leak
// or a fragmentation hazard), or a host loop that cannot afford cudaMalloc's implicit
// device synchronisation. This entry point needs no context and allocates nothing: its
// scratch (the per-tile partial sums) is one file-scope
// static __device__ array of fixed size, which every GPU that loads the library keeps for
// the life of the process. The caller passes inputs and outputs.
//
// Consequences documented in include/mstar.h: every call shares that array, so calls that
// overlap on the GPU (on different streams, or from different host threads) race; each
// call writes all that it reads; sizes above MSTAR_NOALLOC_MAX_N are
// rejected. The first call on a device looks up the array's device address.
#include <mutex>

#include "device.cuh"
#include "internal.h"
#include "pairtile.cuh"

namespace {

constexpr int kNaMax = MSTAR_NOALLOC_MAX_N;
constexpr int kNaFin = 128;  // threads of a finishing block

// Scratch layout (doubles): partials [slot][3 npad], one slot per tile, then one force-function
// sum per tile pair.
// The tile grows with n so that at most 136 CTAs, one per SM, hold all the tile pairs: one wave, and
// scratch for 16 slots. Smaller tiles past these sizes make a second wave: 31 us against 23 at
// n = 1024 (32 instead of 64 bodies), 55 against 35 at n = 1600 (64 instead of 128).
constexpr int kNaMaxN1 = 512, kNaMaxN2 = 1024;  // largest n with tiles of 32, 64 bodies
constexpr size_t na_doubles(int npad, int T) {
  return 3 * (size_t)npad * (npad / T) + (size_t)(npad / T) * (npad / T + 1) / 2;
}
constexpr size_t kNaDoubles = na_doubles(kNaMax, 128);
static_assert(na_doubles(kNaMaxN1, 32) <= kNaDoubles && na_doubles(kNaMaxN2, 64) <= kNaDoubles, "scratch too small");

static __device__ __align__(256) double g_noalloc_scratch[kNaDoubles];

struct DevAddr {
  double* ptr = nullptr;
  bool done = false;
};
std::mutex g_mu;
DevAddr g_addr[64];

// Device address of the scratch array on the current device (looked up once per device).
int scratch_address(double** out) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return MSTAR_ERR_CUDA;
  if (dev < 0 || dev >= 64) return MSTAR_ERR_UNSUPPORTED;
  std::lock_guard<std::mutex> lock(g_mu);
  if (!g_addr[dev].done) {
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess) return MSTAR_ERR_CUDA;
    g_addr[dev].ptr = static_cast<double*>(p);
    g_addr[dev].done = true;
  }
  *out = g_addr[dev].ptr;
  return MSTAR_OK;
}

__device__ __forceinline__ void na_tile_pair(int tp, int NT, int& I, int& J) {
  int i = 0;
  int start = 0;
  while (start + (NT - i) <= tp) {
    start += NT - i;
    ++i;
  }
  I = i;
  J = i + (tp - start);
}

// Symmetric tiled pair loop over Cartesian separations (every pair far) in the arithmetic of
// pairtile.cuh: one CTA per pair of tiles of 32 W bodies, one warp per pair of 32-body sub-tiles and
// range of 32 / S rotation steps. Bound by the integer pipe above n = 1024 (22 us of 42 at n = 2047),
// by latency below: prologue, one short chain of steps, the sums, two launches. The FP64 loop over
// four-warp CTAs this replaced took 103 us at n = 100, 127 at 1024 and 130 at 2047 for four launches
// (calls back to back on the stream); now 8.8, 17.0 and 42.5.
template <int W, int S>
__global__ void __launch_bounds__(32 * W * W * S, 1)
    k_na_tiles(int n, int npad, int NT, const double* __restrict__ m, const double* __restrict__ r,
               double* __restrict__ P, double* __restrict__ Upart) {
  constexpr int T = 32 * W, NW = W * W * S;
  __shared__ double sx[T], sy[T], sz[T], sm[T];
  __shared__ long long sfx[T], sfy[T], sfz[T];
  __shared__ unsigned long long smm[T];
  __shared__ int sme[T], sbox[NW][8], scj[NW][32];
  __shared__ float4 sf[T];
  __shared__ double sj3[NW][3][32], si3[NW][3][32], su[NW];  // si3 holds the integer sums before
  using namespace mstar;
  int I, J;
  na_tile_pair(blockIdx.x, NT, I, J);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int wj = warp % W, wi = warp / W % W, s = warp / (W * W);
  const int i = I * T + wi * 32 + lane, jt = wj * 32 + lane, j = J * T + jt;
  const bool i_pad = i >= n, j_pad = j >= n, diag = I == J;
  double pi3[3], pj3[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    pi3[c] = i_pad ? 0.0 : r[3 * (size_t)i + c];
    pj3[c] = j_pad ? 0.0 : r[3 * (size_t)j + c];
  }
  const double mi = i_pad ? 0.0 : m[i], mj = j_pad ? 0.0 : m[j], m0 = m[I * T];
  bool eq;
  FixWindow fw = tile_window<NW>(pi3, pj3, mi, mj, i_pad, j_pad, m0, sbox, &eq);
  // masses that are not positive are legal here: FP64 throughout (zero is outside the window's range)
  fw.ok = __all_sync(0xffffffffu, fw.ok && (i_pad || __double2hiint(mi) >= 0) && (j_pad || __double2hiint(mj) >= 0));
  if (tid < T) {  // the warps of wi = 0, s = 0
    sx[tid] = pj3[0];
    sy[tid] = pj3[1];
    sz[tid] = pj3[2];
    sm[tid] = mj;
    sfx[tid] = fix_of(pj3[0], fw.u);
    sfy[tid] = fix_of(pj3[1], fw.u);
    sfz[tid] = fix_of(pj3[2], fw.u);
    sf[tid] = make_float4(float_of(pj3[0]), float_of(pj3[1]), float_of(pj3[2]), sqrtf(float_of(mj)));
    const MassSplit ms = fix_mass(mj);
    smm[tid] = ms.m;
    sme[tid] = ms.e;
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) sj3[warp][c][lane] = 0.0;
  TileBody body;
  body.set(pi3[0], pi3[1], pi3[2], mi, fw);
  __syncthreads();
  const bool self = diag && wi == wj;
  if (!(diag && wj < wi)) {
    const int js = wj * 32;
    const int k0 = self ? 1 + s * (16 / S) : s * (32 / S), k1 = k0 + (self ? 16 : 32) / S;
    const unsigned mw = mask_word(nullptr, i_pad, n - J * T - js, self, lane);
    long long* sb = reinterpret_cast<long long*>(&si3[warp][0][0]);
    const SubTile t{sx + js,       sy + js,       sz + js,       sfx + js,      sfy + js,      sfz + js,
                    smm + js,      sme + js,      sf + js,       sm + js,       sj3[warp][0],  sj3[warp][1],
                    sj3[warp][2],  sb,            sb + 32,       sb + 64,       scj[warp]};
    subtile_pairs<Fallback::plain, S < 4 ? 8 : 16 / S, 2>(body, t, fw, eq, m0, mw, k0, k1, lane, [&] {
      return i_pad ? BodyPos{0.0, 0.0, 0.0, 0.0}
                   : BodyPos{r[3 * (size_t)i], r[3 * (size_t)i + 1], r[3 * (size_t)i + 2], mi};
    });
  }
  __syncwarp();
  si3[warp][0][lane] = body.ax;
  si3[warp][1][lane] = body.ay;
  si3[warp][2][lane] = body.az;
  double um = i_pad ? 0.0 : mi * body.u;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) um += __shfl_down_sync(0xffffffffu, um, o);
  if (lane == 0) su[warp] = um;
  __syncthreads();
  // sums over the warps, in warp order: thread q of 3 T holds component q mod 3 of body q / 3
  for (int q = tid; q < 3 * T; q += 32 * NW) {
    const int b = q / 3, c = q - 3 * b, sub = b >> 5, l = b & 31;
    double fi = 0.0, fj = 0.0;
#pragma unroll
    for (int w = 0; w < W * S; ++w) {
      const int o = w % W, st = w / W * W * W;
      fi += si3[st + sub * W + o][c][l];
      fj += sj3[st + o * W + sub][c][l];
    }
    if (diag) {
      P[(size_t)I * 3 * npad + 3 * (size_t)I * T + q] = fi - fj;
    } else {
      P[(size_t)J * 3 * npad + 3 * (size_t)I * T + q] = fi;
      P[(size_t)I * 3 * npad + 3 * (size_t)J * T + q] = -fj;
    }
  }
  if (tid == 0) {
    double u = 0.0;
#pragma unroll
    for (int w = 0; w < NW; ++w) u += su[w];
    Upart[blockIdx.x] = u;
  }
}

// a = G times the sums over the slots; the last block sums the force function.
__global__ void __launch_bounds__(kNaFin) k_na_finish(int n, int npad, int NT, double G, const double* __restrict__ P,
                                                      const double* __restrict__ Upart, double* __restrict__ a,
                                                      double* __restrict__ U) {
  __shared__ double scratch[32];
  if (blockIdx.x == gridDim.x - 1) {
    double u = 0.0;
    for (int t = threadIdx.x; t < NT * (NT + 1) / 2; t += kNaFin) u += Upart[t];
    u = mstar::block_sum(u, scratch);
    if (threadIdx.x == 0) *U = G * u;
    return;
  }
  const int q = blockIdx.x * kNaFin + threadIdx.x;
  if (q >= 3 * n) return;
  double s = 0.0;
#pragma unroll 4
  for (int t = 0; t < NT; ++t) s += P[(size_t)t * 3 * npad + q];
  a[q] = G * s;
}

template <int W, int S>
void na_run(int n, const double* m, const double* r, double G, double* a, double* U, double* base, cudaStream_t s) {
  const int NT = (n + 32 * W - 1) / (32 * W), npad = 32 * W * NT;
  double* Upart = base + (size_t)3 * npad * NT;
  k_na_tiles<W, S><<<NT * (NT + 1) / 2, 32 * W * W * S, 0, s>>>(n, npad, NT, m, r, base, Upart);
  k_na_finish<<<(3 * n + kNaFin - 1) / kNaFin + 1, kNaFin, 0, s>>>(n, npad, NT, G, base, Upart, a, U);
}

bool is_device_pointer(const void* p) {
  cudaPointerAttributes at;
  if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged;
}

}  // namespace

extern "C" MSTAR_API int mstar_accelerations_noalloc(int n, const double* m, const double* r, double G,
                                                     double* a, double* U, void* cuda_stream) {
  if (n < 2 || !m || !r || !a || !U || !(G > 0.0)) return MSTAR_ERR_INVALID_ARG;
  if (n > MSTAR_NOALLOC_MAX_N) return MSTAR_ERR_UNSUPPORTED;
  if (!is_device_pointer(m) || !is_device_pointer(r) || !is_device_pointer(a) || !is_device_pointer(U))
    return MSTAR_ERR_INVALID_ARG;
  double* base = nullptr;
  int rc = scratch_address(&base);
  if (rc != MSTAR_OK) return rc;
  cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
  // Every partial and every force-function sum that is read was written by the same call: nothing
  // to clear.
  if (n <= kNaMaxN1)
    na_run<1, 8>(n, m, r, G, a, U, base, s);
  else if (n <= kNaMaxN2)
    na_run<2, 4>(n, m, r, G, a, U, base, s);
  else
    na_run<4, 1>(n, m, r, G, a, U, base, s);
  if (cudaGetLastError() != cudaSuccess) return MSTAR_ERR_CUDA;
  return MSTAR_OK;
}
