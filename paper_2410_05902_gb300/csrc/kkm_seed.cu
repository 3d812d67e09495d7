// Kernel k-means++ seeding on the GPU (kkm_kmeanspp).
//
// Secs. 1 and 5 start from k-means++ (Arthur and Vassilvitskii, 2007) run in
// feature space, so every initial center is a data point. D^2 sampling:
//   1. the first center is uniform over X;
//   2. each later center is x with probability proportional to
//      D(x)^2 = min over the chosen c of Delta(x, c),
//      Delta(x, c) = K(x,x) - 2 K(x,c) + K(c,c).
// The uniform variate of draw t is u_t = (h_t >> 11) * 2^-53 with h_t output t
// of SplitMix64 seeded with `seed`; the draw picks the first x whose running
// sum of D^2 exceeds u_t * total. Draw 0 (the first center) maps h_0 onto
// [0, n) by Lemire's multiply-high; so does a draw whose total is 0.
//
// Each draw is one launch: every block refreshes D^2 against the newest center
// for its points (one, two, four or eight lanes a point) and writes its FP64
// sum, and the last block to finish finds the crossing point. The chosen index
// stays on the device, so the k draws need no host round trip.
//
// What bounds it: FP64. The chip issues about 2 FP64 operations per clock and
// SM, 1/64 of its FP32 rate, conversions included. The squared distance is
// therefore summed in FP32 triples (hi + mid + lo, every rounding error of the
// large terms carried exactly by two-sums and FMA products), about 40 FP32
// operations per feature in place of three FP64 ones, with a smaller error
// than an FP64 sum has; and a point has few lanes, so the FP64 exponential (or
// square root) runs once per lane of it, not on 32. Measured at 200000 x 64,
// k = 50: 38.2 ms per call with a warp per point, four FP64 sums, the
// exponential on every lane and two launches per draw, 1.62 ms now.
// At d = 3 .. 784 the triples end at most 1.0e-16 (relative) off the exact
// sum, the FP64 sums they replace 2.3e-16.
//
// Lanes per point: one where the points alone fill the chip. Fewer points than
// two blocks' worth for every SM are spread over more lanes as long as each
// keeps a tile of features of its own. One draw at 5000 x 784: Gaussian kernel
// 60 us with one lane a point and 35 with eight (107 with a warp), polynomial
// 158 and 79 (101 with a warp).
#include <algorithm>
#include <type_traits>

#include "kkm_internal.cuh"

namespace kkm {
namespace {

constexpr int PP_NT = 128;                  // threads per block
constexpr int PP_STATIC = 21 * 1024;        // a block's shared memory aside from the center's row
constexpr int PP_F = 32;                    // features per lane of a staged tile
constexpr int PP_PITCH = PP_F + 4;          // floats per lane of a tile's row: float4 reads without bank conflicts

__device__ __forceinline__ double uniform01(uint64_t seed, uint64_t counter) {
  return (double)(splitmix64(seed, counter) >> 11) * (1.0 / 9007199254740992.0);
}

__device__ double kernel_fp64(int kind, double d2, double xy, double param, double coef0, int degree) {
  if (kind == K_GAUSS) return exp(-d2 / param);
  if (kind == K_LAPLACE) return exp(-sqrt(d2) / param);
  if (kind == K_LINEAR) return xy;
  double base = xy + coef0, r = 1.0;
  for (int p = 0; p < degree; ++p) r *= base;
  return r;
}

struct PPArgs {
  const float* X;
  int64_t n, ldx;
  int d, kind, degree;
  double param, coef0;
  uint64_t seed;
  double* d2;          // [n] current D^2
  double* part;        // [nblk] block sums of D^2
  int64_t* chosen;     // [k] chosen indices (device)
  unsigned* done;      // finished blocks of the current draw (0 between draws)
  int vec;             // rows may be read 16 bytes at a time
};

// hi + mid + lo += (x - c)^2. x - c = s + e exactly; s^2 = p + q and 2 s e =
// t + u exactly (FMA products); hi and mid collect their terms by two-sums, lo
// the errors of mid's sums and the terms below 2^-46 s^2 in plain FP32. nz
// stays 0 while every difference is 0.
__device__ __forceinline__ void add_square(float x, float c, float& hi, float& mid, float& lo, unsigned& nz) {
  float e, g, h;
  const float s = two_sum(x, -c, e);
  nz |= __float_as_uint(s);
  const float p = __fmul_rn(s, s), q = __fmaf_rn(s, s, -p);
  const float s2 = __fadd_rn(s, s);
  const float t = __fmul_rn(s2, e), u = __fmaf_rn(s2, e, -t);
  hi = two_sum(hi, p, g);
  mid = two_sum(mid, g, h);
  lo = __fadd_rn(lo, h);
  mid = two_sum(mid, q, h);
  lo = __fadd_rn(lo, h);
  mid = two_sum(mid, t, h);
  lo = __fadd_rn(lo, __fadd_rn(h, __fmaf_rn(e, e, u)));
}

// The sum of two triples.
__device__ __forceinline__ void add_triple(float& hi, float& mid, float& lo, float bh, float bm, float bl) {
  float g, h, e;
  hi = two_sum(hi, bh, g);
  mid = two_sum(mid, bm, h);
  mid = two_sum(mid, g, e);
  lo = __fadd_rn(__fadd_rn(lo, bl), __fadd_rn(h, e));
}

// Features [f0, f0 + 32 LP) of the warp's 32 / LP points (rows row0 ..) into
// its tile (rows of LP * PP_PITCH floats), zero past d and past the last point.
template <int LP>
__device__ __forceinline__ void stage_tile(const PPArgs& a, int64_t row0, int f0, float* tile) {
  const unsigned lane = threadIdx.x & 31u;
  if (a.vec) {                              // a row's features are 8 LP 16-byte words
    float4 v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const unsigned i = 32u * u + lane, r = i / (8u * LP), f = f0 + 4u * (i % (8u * LP));
      v[u] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      if (row0 + r < a.n && f < (unsigned)a.d)
        v[u] = __ldg(reinterpret_cast<const float4*>(a.X + (row0 + r) * a.ldx + f));
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const unsigned i = 32u * u + lane;
      *reinterpret_cast<float4*>(tile + i / (8u * LP) * (LP * PP_PITCH) + 4u * (i % (8u * LP))) = v[u];
    }
  } else {
#pragma unroll 8
    for (int u = 0; u < 32; ++u) {
      const unsigned i = 32u * u + lane, r = i / (PP_F * LP), f = i % (PP_F * LP);
      tile[r * (LP * PP_PITCH) + f] =
          (row0 + r < a.n && f0 + f < (unsigned)a.d) ? __ldg(a.X + (row0 + r) * a.ldx + f0 + f) : 0.0f;
    }
  }
  __syncwarp();
}

// First index i in [lo, hi) with base + (v[lo] + ... + v[i]) > target, by one
// warp (32 values per round, warp scan, ballot); hi - 1 if none. Returns the
// index and leaves in *before the running sum before it.
template <typename Load>
__device__ int64_t warp_crossing(int64_t lo, int64_t hi, double base, double target, Load load, double* before) {
  const int lane = threadIdx.x & 31;
  for (int64_t i0 = lo; i0 < hi; i0 += 32) {
    const int64_t i = i0 + lane;
    const double v = i < hi ? load(i) : 0.0;
    double incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const double y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    const unsigned hit = __ballot_sync(0xffffffffu, i < hi && base + incl > target);
    if (hit) {
      const int l = __ffs(hit) - 1;
      const double inc_l = __shfl_sync(0xffffffffu, incl, l);
      const double v_l = __shfl_sync(0xffffffffu, v, l);
      *before = base + inc_l - v_l;
      return i0 + l;
    }
    base += __shfl_sync(0xffffffffu, incl, 31);
  }
  *before = base;
  return hi - 1;
}

// Draw t + 1 by the last block to finish, after draw t's center is in D^2:
// total = sum of the block sums (fixed order); the first point whose running
// sum exceeds u * total (points in index order) becomes chosen[t + 1]. The
// search narrows run -> block -> point, each step by one warp.
// points: per block.
__device__ __forceinline__ void select_next(const PPArgs& a, int nblk, int points, int t) {
  __shared__ double pre[PP_NT];
  const int tid = threadIdx.x, lane = tid & 31;
  const int per = (nblk + PP_NT - 1) / PP_NT;   // thread r sums run r of `per` consecutive block sums
  const int b0 = min(tid * per, nblk), b1 = min(b0 + per, nblk);
  double mine = 0.0;
  for (int q = b0; q < b1; ++q) mine += __ldcg(a.part + q);
  pre[tid] = mine;
  __syncthreads();
  if (tid >= 32) return;
  double total = 0.0;
#pragma unroll
  for (int g = 0; g < PP_NT / 32; ++g) {            // the same scan order as the search below
    double v = pre[32 * g + lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const double y = __shfl_up_sync(0xffffffffu, v, o);
      if (lane >= o) v += y;
    }
    total += __shfl_sync(0xffffffffu, v, 31);
  }
  int64_t c;
  if (!(total > 0.0)) {
    c = (int64_t)index_below(splitmix64(a.seed, (uint64_t)(t + 1)), (uint64_t)a.n);
  } else {
    const double target = uniform01(a.seed, (uint64_t)(t + 1)) * total;
    double before = 0.0;
    const int64_t r = warp_crossing(0, PP_NT, 0.0, target, [&](int64_t i) { return pre[i]; }, &before);
    const int64_t q0 = min((int64_t)r * per, (int64_t)nblk), q1 = min(q0 + per, (int64_t)nblk);
    const int64_t q = warp_crossing(q0, q1 > q0 ? q1 : q0 + 1, before, target,
                                    [&](int64_t i) { return i < nblk ? __ldcg(a.part + i) : 0.0; }, &before);
    const int64_t x0 = q * points, x1 = min(x0 + points, a.n);
    const int64_t x = warp_crossing(x0, x1 > x0 ? x1 : x0 + 1, before, target,
                                    [&](int64_t i) { return i < a.n ? __ldcg(a.d2 + i) : 0.0; }, &before);
    c = x < a.n ? x : a.n - 1;
  }
  if (lane == 0) a.chosen[t + 1] = c;
}

// D^2(x) = min(D^2(x), Delta(x, c)) for c = chosen[t] (first draw: = Delta),
// then (last block) draw t + 1. LP lanes share a point: lane p of it takes the
// tile's float4 words p, p + LP, .. and the lanes' sums meet by shuffles.
// DOT (linear and polynomial kernels): <x, c>, ||x||^2 and ||c||^2 in FP64, all
// three in the same order, so that Delta of a row that equals the center's is
// exactly 0. The lane's words go to four sums in turn, and the block's four
// warps take one of ||c||^2's each. The center's row is kept in FP64, which
// leaves three FP64 operations per feature and lane and a quarter of one:
// 200000 x 256, linear kernel: 523 us a draw with ||c||^2 in one warp and the
// center's row converted by every lane, 421 now.
// Otherwise ||x - c||^2 in FP32 triples; a warp with a sum that left the range
// where every product is exact (below 2^-60 but not 0, above 2^120, or not
// finite) sums that tile again in FP64.
template <bool DOT, int LP>
__global__ void __launch_bounds__(PP_NT) k_pp_draw(PPArgs a, int t) {
  using C = std::conditional_t<DOT, double, float>;
  extern __shared__ __align__(16) unsigned char smem[];
  C* const crow = reinterpret_cast<C*>(smem);         // [round_up(d, 32 LP)] the center's row
  __shared__ __align__(16) float tiles[PP_NT / 32][32 * PP_PITCH];
  __shared__ double red[PP_NT / 32], cself[PP_NT / 32][32];
  __shared__ bool last;
  constexpr int TF = PP_F * LP;                       // features of a tile
  const unsigned lane = threadIdx.x & 31u, w = threadIdx.x >> 5, p = lane % LP;
  const int64_t row0 = (int64_t)blockIdx.x * (PP_NT / LP) + 32 / LP * w, x = row0 + lane / LP;
  const int dp = (a.d + TF - 1) / TF * TF;
  float* const tile = tiles[w];
  const float* const mine = tile + lane / LP * (LP * PP_PITCH);
  stage_tile<LP>(a, row0, 0, tile);                   // X does not depend on the draw before
  KKM_GRID_DEP_WAIT();
  KKM_LAUNCH_DEPENDENTS();
  const float* cr = a.X + a.chosen[t] * a.ldx;
  for (int f = threadIdx.x; f < dp; f += PP_NT) crow[f] = (C)(f < a.d ? cr[f] : 0.0f);
  __syncthreads();
  double delta;
  if constexpr (DOT) {
    double qxy[4] = {}, qxx[4] = {}, qcc = 0.0;
    for (int f0 = 0; f0 < dp; f0 += TF) {
      if (f0 > 0) {
        __syncwarp();
        stage_tile<LP>(a, row0, f0, tile);
      }
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float4 xv = *reinterpret_cast<const float4*>(mine + 4 * (i * LP + p));
        const double2* cq = reinterpret_cast<const double2*>(&crow[f0 + 4 * (i * LP + p)]);
        const double2 c0 = cq[0], c1 = cq[1];
        const double xd[4] = {xv.x, xv.y, xv.z, xv.w}, cd[4] = {c0.x, c0.y, c1.x, c1.y};
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          qxy[i & 3] = fma(xd[u], cd[u], qxy[i & 3]);
          qxx[i & 3] = fma(xd[u], xd[u], qxx[i & 3]);
        }
        if ((i & 3) == w)
#pragma unroll
          for (int u = 0; u < 4; ++u) qcc = fma(cd[u], cd[u], qcc);
      }
    }
    static_assert(PP_NT / 32 == 4, "a warp per sum of ||c||^2");
    cself[w][lane] = qcc;
    __syncthreads();
    double sxy = (qxy[0] + qxy[1]) + (qxy[2] + qxy[3]);
    double sxx = (qxx[0] + qxx[1]) + (qxx[2] + qxx[3]);
    double scc = (cself[0][lane] + cself[1][lane]) + (cself[2][lane] + cself[3][lane]);
#pragma unroll
    for (int o = 1; o < LP; o <<= 1) {
      sxy += __shfl_xor_sync(0xffffffffu, sxy, o);
      sxx += __shfl_xor_sync(0xffffffffu, sxx, o);
      scc += __shfl_xor_sync(0xffffffffu, scc, o);
    }
    delta = kernel_fp64(a.kind, 0.0, sxx, a.param, a.coef0, a.degree) -
            2.0 * kernel_fp64(a.kind, 0.0, sxy, a.param, a.coef0, a.degree) +
            kernel_fp64(a.kind, 0.0, scc, a.param, a.coef0, a.degree);
  } else {
    float hi = 0.0f, mid = 0.0f, lo = 0.0f;
    unsigned nz = 0u;
    for (int f0 = 0; f0 < dp; f0 += TF) {
      if (f0 > 0) {
        __syncwarp();
        stage_tile<LP>(a, row0, f0, tile);
      }
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float4 xv = *reinterpret_cast<const float4*>(mine + 4 * (i * LP + p));
        const float4 cv = *reinterpret_cast<const float4*>(&crow[f0 + 4 * (i * LP + p)]);
        add_square(xv.x, cv.x, hi, mid, lo, nz);
        add_square(xv.y, cv.y, hi, mid, lo, nz);
        add_square(xv.z, cv.z, hi, mid, lo, nz);
        add_square(xv.w, cv.w, hi, mid, lo, nz);
      }
    }
#pragma unroll
    for (int o = 1; o < LP; o <<= 1) {
      add_triple(hi, mid, lo, __shfl_xor_sync(0xffffffffu, hi, o), __shfl_xor_sync(0xffffffffu, mid, o),
                 __shfl_xor_sync(0xffffffffu, lo, o));
      nz |= __shfl_xor_sync(0xffffffffu, nz, o);
    }
    double s2 = (double)hi + ((double)mid + (double)lo);
    const bool redo = nz != 0u && !(hi >= 0x1p-60f && hi <= 0x1p120f);
    if (__any_sync(0xffffffffu, redo)) {
      double s = 0.0;
      for (int f0 = 0; f0 < dp; f0 += TF) {
        __syncwarp();
        stage_tile<LP>(a, row0, f0, tile);
        for (int i = 0; i < PP_F; ++i) {
          const int f = 4 * (i / 4 * LP + p) + i % 4;
          const double df = (double)mine[f] - (double)crow[f0 + f];
          s = fma(df, df, s);
        }
      }
#pragma unroll
      for (int o = 1; o < LP; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (redo) s2 = s;
    }
    delta = 2.0 - 2.0 * kernel_fp64(a.kind, s2, 0.0, a.param, 0.0, 0);
  }
  delta = fmax(delta, 0.0);
  double v = 0.0;
  if (x < a.n && p == 0) {
    v = (t == 0) ? delta : fmin(a.d2[x], delta);
    a.d2[x] = v;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if (lane == 0) red[w] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int q = 0; q < PP_NT / 32; ++q) s += red[q];
    a.part[blockIdx.x] = s;
  }
  // D^2 and the block sum become visible before the block counts as finished
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(a.done, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  select_next(a, (int)gridDim.x, PP_NT / LP, t);
  if (threadIdx.x == 0) *a.done = 0u;                 // ready for the next draw
}

using PPDraw = void (*)(PPArgs, int);
template <bool DOT> PPDraw draw_kernel(int lanes) {
  return lanes == 1   ? k_pp_draw<DOT, 1>
         : lanes == 2 ? k_pp_draw<DOT, 2>
         : lanes == 4 ? k_pp_draw<DOT, 4>
                      : k_pp_draw<DOT, 8>;
}

}  // namespace

// Lanes per point (see the header comment).
static int kmeanspp_lanes(int64_t n, int d, int num_sms) {
  int lanes = 1;
  while (lanes < 8 && n * lanes < 2 * (int64_t)PP_NT * num_sms && d > PP_F * lanes) lanes *= 2;
  return lanes;
}

int64_t kmeanspp_blocks(int64_t n, int d, int num_sms) {
  return (n * kmeanspp_lanes(n, d, num_sms) + PP_NT - 1) / PP_NT;
}

cudaError_t launch_kmeanspp(const float* X, int64_t n, int d, int64_t ldx, int k, int kind, double param,
                            double coef0, int degree, uint64_t seed, int num_sms, double* d2, double* part,
                            int64_t* chosen, unsigned* done, cudaStream_t st) {
  const int vec = d % 4 == 0 && ldx % 4 == 0 && reinterpret_cast<uintptr_t>(X) % 16 == 0;
  PPArgs a{X, n, ldx, d, kind, degree, param, coef0, seed, d2, part, chosen, done, vec};
  const int lanes = kmeanspp_lanes(n, d, num_sms);
  const int64_t nblk = kmeanspp_blocks(n, d, num_sms);
  if (nblk > (int64_t)0x7fffffff) return cudaErrorInvalidValue;
  // draw 0: uniform
  const int64_t first = (int64_t)index_below(splitmix64(seed, 0), (uint64_t)n);
  cudaError_t e = cudaMemcpyAsync(chosen, &first, sizeof(first), cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaMemsetAsync(done, 0, sizeof(unsigned), st);
  const bool dot = kind == K_LINEAR || kind == K_POLY;
  const PPDraw draw = dot ? draw_kernel<true>(lanes) : draw_kernel<false>(lanes);
  size_t smem = (size_t)round_up(d, PP_F * lanes) * (dot ? sizeof(double) : sizeof(float));   // at most 32 KB
  // Blocks of the next draw take their places while this one's finish, wherever
  // there is room, and then stay: with more room than its share an SM ends up
  // with nine of 782 blocks that others have five of. Shared memory past the
  // row's keeps every SM to its share (at most eight). 100000 points, d = 64 and
  // 256: 33.0 and 82 us a draw without, 29.1 and 65 with.
  const int64_t share = std::min<int64_t>(8, (nblk + num_sms - 1) / num_sms);
  if (share >= 2) smem = std::max<size_t>(smem, (228 * 1024 / share - 1024 - PP_STATIC) / 128 * 128);
  if (e == cudaSuccess && smem > 24 * 1024)   // with the staged tiles more than a kernel has by default
    e = cudaFuncSetAttribute(draw, cudaFuncAttributeMaxDynamicSharedMemorySize, 100 * 1024);   // the same for every call
  for (int t = 0; t + 1 < k && e == cudaSuccess; ++t)
    e = launch_pdl(draw, dim3((unsigned)nblk), dim3(PP_NT), smem, st, a, t);
  return e;
}

}  // namespace kkm
