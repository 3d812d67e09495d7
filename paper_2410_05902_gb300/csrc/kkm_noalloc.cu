// kkm_distances_noalloc: the FP32 distance pass without a context and without
// any allocation.
//
// Some callers cannot call cudaMalloc. Two kinds are common. One is a caller
// whose device memory is owned entirely by a framework's caching allocator or
// a pre-sized arena: a serving process that reserved the free memory at
// start-up, where a stray cudaMalloc fails or fragments that reservation. The
// other is a caller on a latency-critical loop, where cudaMalloc and cudaFree
// can synchronise the device and stall for milliseconds. This entry point lets
// such callers score query points against k centers that they hold
// themselves. They pass the inputs and the outputs. The only scratch is one
// file-scope __device__ array of fixed size (KKM_NOALLOC_SCRATCH_BYTES in
// kkm.h).
//
// CUDA loads modules lazily by default, so that array, and the code of this
// file's kernels, come onto a device when the first call on that device looks
// up the array's address and launches the kernels. The first call on each
// device therefore reserves the memory; a call with m = 0 does exactly that
// and nothing else. It must come before the caller reserves the rest of the
// device memory and before any stream capture. Later calls reserve nothing.
//
// Host code never dereferences the array's name: on the host that name is only
// a stand-in. Every call shares the one array, so two calls whose kernels
// overlap on the GPU (for example on two streams without ordering between
// them) race on it. Calls queued on one stream, one after another, are safe.
// Each call writes every scratch entry it later reads (tile list, norms,
// partial sums, the offsets' check), so nothing left over from an earlier call
// is ever used.
//
// A small call is a chain of launches, so it is three: tile list and norms,
// Gram tiles, distances and argmin. 64 queries against 50 centers of about 216
// rows each, d = 64: 77.8 us as five launches with FP64 norm reductions and a
// thread per row in the argmin, now 20.3 us (5.2, 10.1 and 11.2 us alone with
// cold caches).
#include <algorithm>
#include <mutex>
#include <string>

#include "kkm_internal.cuh"
#include "../../include/kkm.h"

#define KKM_API extern "C" __attribute__((visibility("default")))

namespace {

constexpr int NA_ROWS = KKM_NOALLOC_MAX_ROWS_PER_PASS;   // query rows per internal pass
constexpr int NA_TILE = 64;                               // support rows per tile
constexpr int NA_MAX_TILES = KKM_NOALLOC_MAX_TILES;
constexpr int NA_MAX_S = KKM_NOALLOC_MAX_SUPPORT;
constexpr int BK = 16, NT = 256;

struct Scratch {
  float part[NA_MAX_TILES * NA_ROWS];   // per-tile weighted kernel sums of each query row
  float yn[NA_MAX_S];                   // ||y||^2 of the support rows
  float qn[NA_ROWS];                    // ||q||^2 of the pass's query rows
  int4 tiles[NA_MAX_TILES];             // (center, first support row, rows, -)
  int32_t tile_first[1024];
  int32_t tile_cnt[1024];
  int32_t ntiles;                       // tiles written by this call's k_na_tiles
  int32_t bad;                          // the call's offsets were not non-decreasing within [0, S]
};
static_assert(sizeof(Scratch) <= KKM_NOALLOC_SCRATCH_BYTES, "scratch layout exceeds its declared size");

static __device__ __align__(256) unsigned char kkm_noalloc_scratch[KKM_NOALLOC_SCRATCH_BYTES];

std::mutex g_na_mutex;
void* g_na_addr[256] = {};
bool g_na_loaded[256] = {};
thread_local std::string g_na_error;

kkm_status na_fail(kkm_status st, const char* msg) {
  g_na_error = msg;
  return st;
}

// Launches one kernel and returns that launch's own status. A failed launch's
// error is cleared from the thread's last-error record once it is returned
// here; an error left there by someone else's earlier launch is neither
// reported as this call's nor cleared. The kernels wait for everything queued
// before them at their first statement, so each may be set up during the one ahead.
template <typename... Params, typename... Args>
cudaError_t na_launch(void (*kern)(Params...), int grid, int block, cudaStream_t st, Args... args) {
  const cudaError_t e = kkm::launch_pdl(kern, dim3((unsigned)grid), dim3((unsigned)block), 0, st, args...);
  if (e != cudaSuccess) (void)cudaGetLastError();
  return e;
}

// The tile list of the support segments, by one block of NT threads (four
// centers each, k <= 1024). Offsets that are not non-decreasing within [0, S]
// (or whose tiles would not fit the list, which well-formed offsets under the
// host's size check never do) set `bad` and leave an empty list, so no later
// kernel reads a tile.
__device__ void na_tiles(Scratch* sc, const int32_t* __restrict__ seg_off, int k, int S) {
  __shared__ int wsum[NT / 32];
  constexpr int PER = 1024 / NT;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  int a[PER], size[PER], nt[PER], mine = 0, bad_here = 0;
#pragma unroll
  for (int u = 0; u < PER; ++u) {
    const int j = tid * PER + u;
    a[u] = size[u] = nt[u] = 0;
    if (j < k) {
      const int s0 = seg_off[j], s1 = seg_off[j + 1];
      bad_here |= s0 < 0 || s1 < s0 || s1 > S;
      a[u] = min(max(s0, 0), S);
      size[u] = min(max(s1, a[u]), S) - a[u];
      nt[u] = (size[u] + NA_TILE - 1) / NA_TILE;
      mine += nt[u];
    }
  }
  int x = mine;
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) wsum[warp] = x;
  const int any_bad = __syncthreads_or(bad_here);
  int before = 0, total = 0;
  for (int w = 0; w < NT / 32; ++w) {
    if (w < warp) before += wsum[w];
    total += wsum[w];
  }
  const bool bad = any_bad || total > NA_MAX_TILES;
  int first = x - mine + before;                // every first + nt <= total when !bad
  if (tid == 0) {
    sc->ntiles = bad ? 0 : total;
    sc->bad = bad ? 1 : 0;
  }
#pragma unroll
  for (int u = 0; u < PER; ++u) {
    const int j = tid * PER + u;
    if (j < k) {
      sc->tile_first[j] = bad ? 0 : first;
      sc->tile_cnt[j] = bad ? 0 : nt[u];
      if (!bad)
        for (int t = 0; t < nt[u]; ++t)
          sc->tiles[first + t] = make_int4(j, a[u] + t * NA_TILE, min(NA_TILE, size[u] - t * NA_TILE), 0);
      first += nt[u];
    }
  }
}

// A sum kept as h + l in two FP32 words, every rounding error carried.
__device__ __forceinline__ void pair_add(float& h, float& l, float bh, float bl) {
  const float s = __fadd_rn(h, bh);
  const float t = __fsub_rn(s, h);
  const float e = __fadd_rn(__fsub_rn(h, __fsub_rn(s, t)), __fsub_rn(bh, t));
  l = __fadd_rn(__fadd_rn(l, bl), e);
  h = s;
}
__device__ __forceinline__ void pair_square(float& h, float& l, float v) {
  const float p = __fmul_rn(v, v);
  pair_add(h, l, p, __fmaf_rn(v, v, -p));
}

// What a call's Gram pass needs, in one launch: the tile list (block 0, when
// tiles is set; the host then passes k >= 1) and ||row||^2 of the support rows
// Y and of a pass's query rows Q, FP32-rounded, eight lanes a row. The squares
// are summed as FP32 pairs (48 bits): FP64 issues at 1/64 of the FP32 rate on
// this chip, and a warp per row with a 32-lane FP64 reduction took longer than
// the Gram tiles of a small call. A pair only stands where every sum within
// its error rounds to the same FP32 value, so that the norms are those of FP64
// sums to the bit; the others (one row in thousands), sums near the ends of the
// FP32 range (where a square's error term leaves it), zeros and non-finite ones
// are taken again in FP64. VEC: rows on 16-byte boundaries (as NaGram's).
template <bool VEC>
__global__ void __launch_bounds__(NT) k_na_prepare(Scratch* sc, int tiles, const int32_t* __restrict__ seg_off,
                                                   int k, int S, const float* __restrict__ Y, int64_t ldy, int ny,
                                                   const float* __restrict__ Q, int64_t ldq, int nq, int d) {
  KKM_GRID_DEP_WAIT();
  KKM_LAUNCH_DEPENDENTS();
  if (tiles && blockIdx.x == 0) {
    na_tiles(sc, seg_off, k, S);
    return;
  }
  const int sub = threadIdx.x & 7;
  const int r = ((int)blockIdx.x - (tiles ? 1 : 0)) * (NT / 8) + (int)(threadIdx.x >> 3);
  const bool live = r < ny + nq;
  const float* p = r < ny ? Y + (int64_t)r * ldy : live ? Q + (int64_t)(r - ny) * ldq : nullptr;
  const int dl = live ? d : 0;
  float h = 0.0f, l = 0.0f;
  int c = VEC ? 4 * sub : sub;
  if constexpr (VEC) {
#pragma unroll 2
    for (; c + 3 < dl; c += 32) {
      const float4 v = *reinterpret_cast<const float4*>(p + c);
      pair_square(h, l, v.x);
      pair_square(h, l, v.y);
      pair_square(h, l, v.z);
      pair_square(h, l, v.w);
    }
    for (; c < dl; ++c) pair_square(h, l, p[c]);   // at most one lane has a partial vector
  } else {
#pragma unroll 4
    for (; c < dl; c += 8) pair_square(h, l, p[c]);
  }
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) {
    const float bh = __shfl_xor_sync(0xffffffffu, h, o), bl = __shfl_xor_sync(0xffffffffu, l, o);
    pair_add(h, l, bh, bl);
  }
  float out = __fadd_rn(h, l);
  // m additions into a pair: each rounds l, at most m 2^-24 h, by 2^-24 of it;
  // twice that bounds their sum and the roundings of the bound itself
  const float m = (float)(d / 8 + 8), err = __fmul_rn(h, m * m * 0x1p-47f);
  const bool redo = live && (!(h > 1e-25f && h < 1e37f) || __fadd_rn(h, __fsub_rn(l, err)) != __fadd_rn(h, __fadd_rn(l, err)));
  if (__any_sync(0xffffffffu, redo)) {
    double acc = 0.0;
    for (int q = sub; q < dl; q += 8) acc += (double)p[q] * (double)p[q];
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (redo) out = (float)acc;
  }
  if (live && sub == 0) (r < ny ? sc->yn[r] : sc->qn[r - ny]) = out;
}

// Persistent over (16 MR-row query tile, 64-row support tile): FP32 Gram, then
// the kernel values and the weighted sum of each query row over the tile's
// support rows. A thread holds MR x 4 products; the next 16 columns are loaded
// into registers while the current ones are multiplied from shared memory
// (two buffers, one barrier per 16 columns). VEC: both matrices' rows start on
// 16-byte boundaries and are read four columns at a time; otherwise
// (any leading dimension) by single bounds-checked loads.
// DIFF (Laplacian kernel): the tile accumulates ||q - y||^2 from the
// differences instead of <q, y>. Through ||q||^2 + ||y||^2 - 2 <q, y> a query
// equal to a support row would get d2 of the order of the FP32 rounding of
// its norm instead of 0, and the square root magnifies that into an error of
// its square root; the difference form has no such cancellation.
template <bool VEC>
__device__ __forceinline__ void na_load4(const float* p, bool ok, int c, int d, float (&v)[4]) {
  if (VEC && ok && c + 3 < d) {
    const float4 q = *reinterpret_cast<const float4*>(p + c);
    v[0] = q.x;
    v[1] = q.y;
    v[2] = q.z;
    v[3] = q.w;
    return;
  }
#pragma unroll
  for (int e = 0; e < 4; ++e) v[e] = (ok && c + e < d) ? p[c + e] : 0.0f;
}

template <bool DIFF, int MR, bool VEC>
__global__ void __launch_bounds__(NT) k_na_gram(Scratch* sc, const float* __restrict__ Q, int64_t ldq, int rows,
                                                const float* __restrict__ Y, int64_t ldy,
                                                const float* __restrict__ w, int d, int kind, float negc,
                                                float coef0, int degree) {
  constexpr int TR = 16 * MR, NA = TR / 64;     // rows per tile, 64-row slices a loader thread fills
  __shared__ __align__(16) float As[2][BK][TR + 4];
  __shared__ __align__(16) float Bs[2][BK][64 + 4];
  KKM_GRID_DEP_WAIT();
  KKM_LAUNCH_DEPENDENTS();
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int lr = tid >> 2, lk = (tid & 3) * 4;
  const int R = (rows + TR - 1) / TR;
  const int ntiles = sc->ntiles;
  for (int item = blockIdx.x; item < R * ntiles; item += gridDim.x) {
    const int t = item / R, rt = item % R;
    const int4 T = sc->tiles[t];
    const float* ap[NA];
    bool a_ok[NA];
#pragma unroll
    for (int q = 0; q < NA; ++q) {
      const int arow = rt * TR + q * 64 + lr;
      a_ok[q] = arow < rows;
      ap[q] = Q + (int64_t)(a_ok[q] ? arow : 0) * ldq;
    }
    const bool b_ok = lr < T.z;
    const float* bp = Y + (int64_t)(T.y + (b_ok ? lr : 0)) * ldy;
    float acc[MR][4] = {};
    float av[NA][4], bv[4];
    auto load = [&](int k0) {
#pragma unroll
      for (int q = 0; q < NA; ++q) na_load4<VEC>(ap[q], a_ok[q], k0 + lk, d, av[q]);
      na_load4<VEC>(bp, b_ok, k0 + lk, d, bv);
    };
    auto store = [&](int b) {
#pragma unroll
      for (int e = 0; e < 4; ++e) {
#pragma unroll
        for (int q = 0; q < NA; ++q) As[b][lk + e][q * 64 + lr] = av[q][e];
        Bs[b][lk + e][lr] = bv[e];
      }
    };
    load(0);
    __syncthreads();                            // the previous item's readers are done
    store(0);
    int buf = 0;
    for (int k0 = 0; k0 < d; k0 += BK, buf ^= 1) {
      const bool more = k0 + BK < d;
      if (more) load(k0 + BK);
      __syncthreads();                          // this buffer is filled, the other one read
#pragma unroll
      for (int kk = 0; kk < BK; ++kk) {
        float ar[MR];
#pragma unroll
        for (int i = 0; i < MR; i += 4) {
          const float4 a4 = *reinterpret_cast<const float4*>(&As[buf][kk][ty * MR + i]);
          ar[i] = a4.x;
          ar[i + 1] = a4.y;
          ar[i + 2] = a4.z;
          ar[i + 3] = a4.w;
        }
        const float4 b4 = *reinterpret_cast<const float4*>(&Bs[buf][kk][tx * 4]);
        const float br[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
        for (int i = 0; i < MR; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            if constexpr (DIFF) {
              const float df = ar[i] - br[j];
              acc[i][j] = fmaf(df, df, acc[i][j]);
            } else {
              acc[i][j] = fmaf(ar[i], br[j], acc[i][j]);
            }
          }
      }
      if (more) store(buf ^ 1);
    }
    float yn[4], wy[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int c = tx * 4 + j;
      const bool ok = c < T.z;
      yn[j] = ok ? sc->yn[T.y + c] : 0.0f;
      wy[j] = ok ? w[T.y + c] : 0.0f;
    }
#pragma unroll
    for (int i = 0; i < MR; ++i) {
      const int r = rt * TR + ty * MR + i;
      const float xn = r < rows ? sc->qn[r] : 0.0f;
      float sum = 0.0f;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float kv = DIFF ? exp2f(sqrtf(acc[i][j]) * negc)
                              : kkm::kernel_from_gram(kind, acc[i][j], xn, yn[j], false, negc, coef0, degree);
        sum += (tx * 4 + j < T.z) ? wy[j] * kv : 0.0f;
      }
      sum += __shfl_xor_sync(0xffffffffu, sum, 8);
      sum += __shfl_xor_sync(0xffffffffu, sum, 4);
      sum += __shfl_xor_sync(0xffffffffu, sum, 2);
      sum += __shfl_xor_sync(0xffffffffu, sum, 1);
      if (tx == 0 && r < rows) sc->part[(int64_t)t * NA_ROWS + r] = sum;
    }
  }
}

// Delta(q, C_j) = K(q,q) - 2 <phi(q), C_j> + ||C_j||^2 and the argmin (ties to
// the lowest j). Rejected offsets give NaN distances and the assignment -1 on
// every row. A block takes AR rows; thread (g, r) takes row r's centers
// g, g + NT/AR, ... : as one thread per row the chain of a row's k center sums
// was the longest part of a small call.
constexpr int AR = 8;
__global__ void __launch_bounds__(NT) k_na_argmin(const Scratch* sc, int rows, int k,
                                                  const double* __restrict__ cnorm, int kind, double coef0,
                                                  int degree, float* __restrict__ dist_out,
                                                  int32_t* __restrict__ assign_out) {
  __shared__ double sbest[NT];
  __shared__ int sj[NT];
  KKM_GRID_DEP_WAIT();
  KKM_LAUNCH_DEPENDENTS();
  const int r = threadIdx.x % AR, g = threadIdx.x / AR;
  const int x = blockIdx.x * AR + r;
  const bool bad = sc->bad != 0;
  double best = 1e300;
  int bj = 0x7fffffff;
  if (x < rows) {
    const double kxx = bad ? 0.0 : kkm::kernel_self(kind, (double)sc->qn[x], coef0, degree);
    for (int j = g; j < k; j += NT / AR) {
      double dist = 0.0;
      if (!bad) {
        double inner = 0.0;
        const int t0 = sc->tile_first[j], nt = sc->tile_cnt[j];
        const float* part = sc->part + (int64_t)t0 * NA_ROWS + x;
#pragma unroll 4
        for (int t = 0; t < nt; ++t) inner += (double)part[(int64_t)t * NA_ROWS];
        dist = kxx - 2.0 * inner + cnorm[j];
      }
      if (dist_out) dist_out[(int64_t)x * k + j] = bad ? __int_as_float(0x7fc00000) : (float)dist;
      if (dist < best) {
        best = dist;
        bj = j;
      }
    }
  }
  sbest[threadIdx.x] = best;
  sj[threadIdx.x] = bj;
  __syncthreads();
  if (threadIdx.x < AR && x < rows && assign_out) {
    for (int q = 1; q < NT / AR; ++q) {
      const double o = sbest[q * AR + r];
      const int oj = sj[q * AR + r];
      if (o < best || (o == best && oj < bj)) {
        best = o;
        bj = oj;
      }
    }
    assign_out[x] = bad ? -1 : bj == 0x7fffffff ? 0 : bj;   // no distance below the bound: center 0
  }
}

using NaGram = void (*)(Scratch*, const float*, int64_t, int, const float*, int64_t, const float*, int, int, float,
                        float, int);
// Query tiles of 128 rows once a pass fills more than one 64-row tile and the
// larger tiles still give every SM two items; smaller passes are bound by
// latency and take the 64-row tile. [DIFF][128 rows][VEC].
NaGram na_gram_kernel(bool diff, bool wide, bool vec) {
  static const NaGram table[2][2][2] = {
      {{k_na_gram<false, 4, false>, k_na_gram<false, 4, true>}, {k_na_gram<false, 8, false>, k_na_gram<false, 8, true>}},
      {{k_na_gram<true, 4, false>, k_na_gram<true, 4, true>}, {k_na_gram<true, 8, false>, k_na_gram<true, 8, true>}}};
  return table[diff][wide][vec];
}

}  // namespace

KKM_API const char* kkm_noalloc_last_error(void) { return g_na_error.c_str(); }

KKM_API kkm_status kkm_distances_noalloc(const float* Q, int64_t m, int64_t ldq, int32_t d, const float* Y,
                                         int64_t S, int64_t ldy, const float* w, const int32_t* seg_off,
                                         const double* cnorm, int32_t k, const kkm_kernel* kernel,
                                         float* dist_out, int32_t* assign_out, void* stream) {
  if (m < 0) return na_fail(KKM_EINVAL, "m must be >= 0");
  if (m > 0) {
    if (!kernel) return na_fail(KKM_EINVAL, "kernel is required");
    if (!Q) return na_fail(KKM_EINVAL, "Q must be given when m > 0");
    if (d < 1 || d > 4096) return na_fail(KKM_EINVAL, "d must be in [1, 4096]");
    if (ldq < d) return na_fail(KKM_EINVAL, "ldq must be >= d");
    if (k < 1 || k > 1024) return na_fail(KKM_EINVAL, "k must be in [1, 1024]");
    if (S < 0 || S > NA_MAX_S)
      return na_fail(KKM_EINVAL, "S exceeds the scratch limit KKM_NOALLOC_MAX_SUPPORT (65536 support rows)");
    if ((S + NA_TILE - 1) / NA_TILE + k > NA_MAX_TILES)
      return na_fail(KKM_EINVAL,
                     "ceil(S/64) + k exceeds the scratch limit KKM_NOALLOC_MAX_TILES (1024 support tiles)");
    if (S > 0 && (!Y || !w || ldy < d)) return na_fail(KKM_EINVAL, "Y and w are required and ldy must be >= d");
    if (!seg_off || !cnorm) return na_fail(KKM_EINVAL, "seg_off and cnorm are required");
    if (kernel->kind < KKM_GAUSSIAN || kernel->kind > KKM_POLY) return na_fail(KKM_EINVAL, "unknown kernel kind");
    if ((kernel->kind == KKM_GAUSSIAN || kernel->kind == KKM_LAPLACIAN) && !(kernel->param > 0.0))
      return na_fail(KKM_EINVAL, "kernel param must be > 0");
    if (kernel->kind == KKM_POLY && (kernel->degree < 1 || kernel->degree > 8))
      return na_fail(KKM_EINVAL, "polynomial degree must be in [1, 8]");
  }

  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 256) return na_fail(KKM_ECUDA, "cudaGetDevice failed");
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  void* base = nullptr;
  bool load = false;
  {
    std::lock_guard<std::mutex> lock(g_na_mutex);
    if (!g_na_addr[dev]) {
      void* p = nullptr;
      const cudaError_t e = cudaGetSymbolAddress(&p, kkm_noalloc_scratch);
      if (e != cudaSuccess || !p) {
        (void)cudaGetLastError();
        return na_fail(KKM_ECUDA, "cudaGetSymbolAddress of the scratch array failed");
      }
      g_na_addr[dev] = p;
    }
    base = g_na_addr[dev];
    load = m == 0 && !g_na_loaded[dev];
    if (load) g_na_loaded[dev] = true;
  }
  Scratch* sc = static_cast<Scratch*>(base);
  if (m == 0) {
    // The first empty call on a device launches every kernel of this file on
    // empty work (no row, no center), so that their code is loaded now
    // rather than on the first call with queries.
    cudaError_t e = cudaSuccess;
    if (load) {
      for (int v = 0; v < 2 && e == cudaSuccess; ++v)
        e = na_launch(v ? k_na_prepare<true> : k_na_prepare<false>, 1, NT, st, sc, 1, (const int32_t*)nullptr, 0, 0,
                      (const float*)nullptr, (int64_t)0, 0, (const float*)nullptr, (int64_t)0, 0, 1);
      for (int v = 0; v < 8 && e == cudaSuccess; ++v)
        e = na_launch(na_gram_kernel(v & 4, v & 2, v & 1), 1, NT, st, sc, (const float*)nullptr, (int64_t)0, 0,
                      (const float*)nullptr, (int64_t)0, (const float*)nullptr, 1, (int)KKM_LINEAR, 0.0f, 0.0f, 1);
      if (e == cudaSuccess)
        e = na_launch(k_na_argmin, 1, NT, st, (const Scratch*)sc, 0, 0, (const double*)nullptr, (int)KKM_LINEAR,
                      0.0, 1, (float*)nullptr, (int32_t*)nullptr);
      if (e != cudaSuccess) {
        std::lock_guard<std::mutex> lock(g_na_mutex);
        g_na_loaded[dev] = false;
      }
    }
    return e == cudaSuccess ? KKM_OK : na_fail(KKM_ECUDA, cudaGetErrorString(e));
  }

  int sms = 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) {
    (void)cudaGetLastError();
    sms = 148;
  }
  const bool normalised = kernel->kind == KKM_GAUSSIAN || kernel->kind == KKM_LAPLACIAN;
  const float negc = normalised ? (float)(-1.4426950408889634 / kernel->param) : 0.0f;
  const int Si = (int)S;
  const int max_tiles = (Si + NA_TILE - 1) / NA_TILE + k;   // bound on the tiles k_na_tiles writes

  auto aligned = [](const float* p, int64_t ld) { return ((uintptr_t)p & 15) == 0 && ld % 4 == 0; };
  const bool vec = aligned(Q, ldq) && (Si == 0 || aligned(Y, ldy));
  const bool diff = kernel->kind == KKM_LAPLACIAN;
  cudaError_t e = cudaSuccess;
  for (int64_t r0 = 0; r0 < m && e == cudaSuccess; r0 += NA_ROWS) {
    const int rows = (int)std::min<int64_t>(NA_ROWS, m - r0);
    const int first = r0 == 0, ny = first ? Si : 0;   // the tile list and the support norms: once a call
    const float* Qr = Q + r0 * ldq;
    e = na_launch(vec ? k_na_prepare<true> : k_na_prepare<false>, first + (ny + rows + NT / 8 - 1) / (NT / 8), NT, st,
                  sc, first, seg_off, (int)k, Si, Y, ldy, ny, Qr, ldq, rows, (int)d);
    if (e == cudaSuccess && Si > 0) {
      const bool wide = rows > 64 && ((rows + 127) / 128) * max_tiles >= 2 * sms;
      const int items = (wide ? (rows + 127) / 128 : (rows + 63) / 64) * max_tiles;
      const int grid = std::max(1, std::min(items, sms * 4));
      e = na_launch(na_gram_kernel(diff, wide, vec), grid, NT, st, sc, Qr, ldq, rows, Y, ldy, w, (int)d,
                    (int)kernel->kind, negc, (float)kernel->coef0, (int)kernel->degree);
    }
    if (e == cudaSuccess)
      e = na_launch(k_na_argmin, (rows + AR - 1) / AR, NT, st, (const Scratch*)sc, rows, (int)k, cnorm,
                    (int)kernel->kind, kernel->coef0, (int)kernel->degree, dist_out ? dist_out + r0 * k : nullptr,
                    assign_out ? assign_out + r0 : nullptr);
  }
  if (e != cudaSuccess) return na_fail(KKM_ECUDA, cudaGetErrorString(e));
  return KKM_OK;
}
