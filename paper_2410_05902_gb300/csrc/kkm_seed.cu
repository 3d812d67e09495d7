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
// for its 128 points (a thread per point) and writes its FP64 sum, and the
// last block to finish finds the crossing point. The chosen index stays on
// the device, so the k draws need no host round trip.
//
// What bounds it: FP64. The chip issues about 2 FP64 operations per clock and
// SM, 1/64 of its FP32 rate, conversions included. The squared distance is
// therefore summed in FP32 triples (hi + mid + lo, every rounding error of the
// large terms carried exactly by two-sums and FMA products), about 40 FP32
// operations per feature in place of three FP64 ones, with a smaller error
// than an FP64 sum has; and a thread owns a point, so the FP64 exponential
// (or square root) runs once per point, not once per lane. Measured at
// 200000 x 64, k = 50: 38.2 ms per call before (a warp per point, four FP64
// sums and the exponential on every lane, two launches per draw), 1.75 ms now.
// At d = 3 .. 784 the triples end at most 1.0e-16 (relative) off the exact
// sum, the FP64 sums they replace 2.3e-16.
#include "kkm_internal.cuh"

namespace kkm {
namespace {

constexpr int PP_ROWS = 128;                // points per block, a thread each
constexpr int PP_F = 32;                    // features per staged tile
constexpr int PP_PITCH = PP_F + 4;          // float4 reads of 32 different rows without bank conflicts

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

// s + e = a + b exactly (Knuth's two-sum).
__device__ __forceinline__ float two_sum(float a, float b, float& e) {
  const float s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
  return s;
}

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

// Features [f0, f0 + 32) of the warp's 32 points (rows row0 ..) into its tile,
// zero past d and past the last point.
__device__ __forceinline__ void stage_tile(const PPArgs& a, int64_t row0, int f0, float (*tile)[PP_PITCH]) {
  const int lane = threadIdx.x & 31;
  if (a.vec) {                              // a row's 32 features are eight 16-byte words
    float4 v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int r = 4 * u + (lane >> 3), f = f0 + 4 * (lane & 7);
      v[u] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      if (row0 + r < a.n && f < a.d)
        v[u] = __ldg(reinterpret_cast<const float4*>(a.X + (row0 + r) * a.ldx + f));
    }
#pragma unroll
    for (int u = 0; u < 8; ++u)
      *reinterpret_cast<float4*>(&tile[4 * u + (lane >> 3)][4 * (lane & 7)]) = v[u];
  } else {
    const int f = f0 + lane;
#pragma unroll 8
    for (int r = 0; r < 32; ++r)
      tile[r][lane] = (row0 + r < a.n && f < a.d) ? __ldg(a.X + (row0 + r) * a.ldx + f) : 0.0f;
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
__device__ __forceinline__ void select_next(const PPArgs& a, int nblk, int t) {
  __shared__ double pre[PP_ROWS];
  const int tid = threadIdx.x, lane = tid & 31;
  const int per = (nblk + PP_ROWS - 1) / PP_ROWS;   // thread r sums run r of `per` consecutive block sums
  const int b0 = min(tid * per, nblk), b1 = min(b0 + per, nblk);
  double mine = 0.0;
  for (int q = b0; q < b1; ++q) mine += __ldcg(a.part + q);
  pre[tid] = mine;
  __syncthreads();
  if (tid >= 32) return;
  double total = 0.0;
#pragma unroll
  for (int g = 0; g < PP_ROWS / 32; ++g) {          // the same scan order as the search below
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
    const int64_t r = warp_crossing(0, PP_ROWS, 0.0, target, [&](int64_t i) { return pre[i]; }, &before);
    const int64_t q0 = min((int64_t)r * per, (int64_t)nblk), q1 = min(q0 + per, (int64_t)nblk);
    const int64_t q = warp_crossing(q0, q1 > q0 ? q1 : q0 + 1, before, target,
                                    [&](int64_t i) { return i < nblk ? __ldcg(a.part + i) : 0.0; }, &before);
    const int64_t x0 = q * PP_ROWS, x1 = min(x0 + PP_ROWS, a.n);
    const int64_t x = warp_crossing(x0, x1 > x0 ? x1 : x0 + 1, before, target,
                                    [&](int64_t i) { return i < a.n ? __ldcg(a.d2 + i) : 0.0; }, &before);
    c = x < a.n ? x : a.n - 1;
  }
  if (lane == 0) a.chosen[t + 1] = c;
}

// D^2(x) = min(D^2(x), Delta(x, c)) for c = chosen[t] (first draw: = Delta),
// then (last block) draw t + 1. DOT (linear and polynomial kernels): <x, c>,
// ||x||^2 and ||c||^2 in FP64, all three in the same order, so that Delta of a
// row that equals the center's is exactly 0 (||c||^2 is the block's first
// warp's). Otherwise ||x - c||^2 in FP32 triples; a warp with a sum that left
// the range where every product is exact (below 2^-60 but not 0, above 2^120,
// or not finite) sums that tile again in FP64.
template <bool DOT>
__global__ void __launch_bounds__(PP_ROWS) k_pp_draw(PPArgs a, int t) {
  extern __shared__ __align__(16) float crow[];       // [round_up(d, 32)] the center's row
  __shared__ __align__(16) float tiles[PP_ROWS / 32][32][PP_PITCH];
  __shared__ double red[PP_ROWS / 32], cself;
  __shared__ bool last;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t row0 = (int64_t)blockIdx.x * PP_ROWS + 32 * w, x = row0 + lane;
  const int dp = (a.d + PP_F - 1) / PP_F * PP_F;
  float(*tile)[PP_PITCH] = tiles[w];
  stage_tile(a, row0, 0, tile);                       // X does not depend on the draw before
  KKM_GRID_DEP_WAIT();
  KKM_LAUNCH_DEPENDENTS();
  const float* cr = a.X + a.chosen[t] * a.ldx;
  for (int f = threadIdx.x; f < dp; f += PP_ROWS) crow[f] = f < a.d ? cr[f] : 0.0f;
  __syncthreads();
  double delta;
  if constexpr (DOT) {
    double sxy = 0.0, sxx = 0.0, scc = 0.0;
    for (int f0 = 0; f0 < dp; f0 += PP_F) {
      if (f0 > 0) {
        __syncwarp();
        stage_tile(a, row0, f0, tile);
      }
      for (int f = 0; f < PP_F; ++f) {
        const double xv = tile[lane][f], cv = crow[f0 + f];
        sxy = fma(xv, cv, sxy);
        sxx = fma(xv, xv, sxx);
        if (w == 0) scc = fma(cv, cv, scc);
      }
    }
    if (threadIdx.x == 0) cself = scc;
    __syncthreads();
    scc = cself;
    delta = kernel_fp64(a.kind, 0.0, sxx, a.param, a.coef0, a.degree) -
            2.0 * kernel_fp64(a.kind, 0.0, sxy, a.param, a.coef0, a.degree) +
            kernel_fp64(a.kind, 0.0, scc, a.param, a.coef0, a.degree);
  } else {
    float hi = 0.0f, mid = 0.0f, lo = 0.0f;
    unsigned nz = 0u;
    for (int f0 = 0; f0 < dp; f0 += PP_F) {
      if (f0 > 0) {
        __syncwarp();
        stage_tile(a, row0, f0, tile);
      }
#pragma unroll
      for (int f = 0; f < PP_F; f += 4) {
        const float4 xv = *reinterpret_cast<const float4*>(&tile[lane][f]);
        const float4 cv = *reinterpret_cast<const float4*>(&crow[f0 + f]);
        add_square(xv.x, cv.x, hi, mid, lo, nz);
        add_square(xv.y, cv.y, hi, mid, lo, nz);
        add_square(xv.z, cv.z, hi, mid, lo, nz);
        add_square(xv.w, cv.w, hi, mid, lo, nz);
      }
    }
    double s2 = (double)hi + ((double)mid + (double)lo);
    const bool redo = nz != 0u && !(hi >= 0x1p-60f && hi <= 0x1p120f);
    if (__any_sync(0xffffffffu, redo)) {
      double s = 0.0;
      for (int f0 = 0; f0 < dp; f0 += PP_F) {
        __syncwarp();
        stage_tile(a, row0, f0, tile);
        for (int f = 0; f < PP_F; ++f) {
          const double df = (double)tile[lane][f] - (double)crow[f0 + f];
          s = fma(df, df, s);
        }
      }
      if (redo) s2 = s;
    }
    delta = 2.0 - 2.0 * kernel_fp64(a.kind, s2, 0.0, a.param, 0.0, 0);
  }
  delta = fmax(delta, 0.0);
  double v = 0.0;
  if (x < a.n) {
    v = (t == 0) ? delta : fmin(a.d2[x], delta);
    a.d2[x] = v;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if (lane == 0) red[w] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int q = 0; q < PP_ROWS / 32; ++q) s += red[q];
    a.part[blockIdx.x] = s;
  }
  // D^2 and the block sum become visible before the block counts as finished
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(a.done, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  select_next(a, (int)gridDim.x, t);
  if (threadIdx.x == 0) *a.done = 0u;                 // ready for the next draw
}

}  // namespace

cudaError_t launch_kmeanspp(const float* X, int64_t n, int d, int64_t ldx, int k, int kind, double param,
                            double coef0, int degree, uint64_t seed, double* d2, double* part, int64_t* chosen,
                            unsigned* done, cudaStream_t st) {
  const int vec = d % 4 == 0 && ldx % 4 == 0 && reinterpret_cast<uintptr_t>(X) % 16 == 0;
  PPArgs a{X, n, ldx, d, kind, degree, param, coef0, seed, d2, part, chosen, done, vec};
  const int64_t nblk = (n + PP_ROWS - 1) / PP_ROWS;
  if (nblk > (int64_t)0x7fffffff) return cudaErrorInvalidValue;
  // draw 0: uniform
  const int64_t first = (int64_t)index_below(splitmix64(seed, 0), (uint64_t)n);
  cudaError_t e = cudaMemcpyAsync(chosen, &first, sizeof(first), cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaMemsetAsync(done, 0, sizeof(unsigned), st);
  const bool dot = kind == K_LINEAR || kind == K_POLY;
  const size_t smem = (size_t)round_up(d, PP_F) * sizeof(float);   // at most 16 KB
  for (int t = 0; t + 1 < k && e == cudaSuccess; ++t)
    e = launch_pdl(dot ? k_pp_draw<true> : k_pp_draw<false>, dim3((unsigned)nblk), dim3(PP_ROWS), smem, st, a, t);
  return e;
}

}  // namespace kkm
