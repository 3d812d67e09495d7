// FP32 CUDA-core form of the two Gram passes.
//
// Distance pass: for each (64-row batch tile, 64-row support tile of center j),
// G = X_B Y^T in FP32, then in registers
//   K = kernel(||x||^2 + ||y||^2 - 2G) and part[tile][x] = sum_y w_y K(x, y),
// the per-tile share of <phi(x), C_j> (Sec. 1: <phi(x), c> for a center held
// as a weighted sum of feature vectors; Sec. 4.1 cost O(kb(b+tau))).
//
// Window pass (norm recurrence of Sec. 4 with the drops of Eq. (1)): for each
// center with a new block, the weighted sums
//   A   = sum_{p in D, q in W} w_p w_q K(p, q)   = <C, D>
//   Bdd = sum_{p in D, q in D} w_p w_q K(p, q)   = ||D||^2
//   E   = sum_{p in D, q in B} w_p K(p, q)       = b_j <D, cm(B_j)>
//   M   = sum_{p in B, q in B} K(p, q)           = b_j^2 ||cm(B_j)||^2
// where W is the old window, D its dropped prefix (old weights) and B the new
// block. Each tile writes its four FP64 partial sums, which are added in tile
// order (NormReports; run groups: k_finalize).
#include <algorithm>

#include "kkm_internal.cuh"

namespace kkm {
namespace {

constexpr int BM = 64, BN = 64, BK = 16, NT = 256;

// Operand chunks of BK columns, two buffers: columns of 16 MR rows of A and 64 of B.
template <int MR> struct GramSmem {
  float A[2][BK][16 * MR + 4];
  float B[2][BK][BN + 4];
};

// acc[i][j] = sum_k A[ty*MR+i][k] * B[tx*4+j][k] for a 16 MR x 64 tile. A and B
// point at the tiles' first rows; rows are `ld` elements apart and the product
// runs over all of them (zero padded, a multiple of BK).
// DIFF: acc[i][j] = sum_k (A[ty*MR+i][k] - B[tx*4+j][k])^2 instead. The next BK
// columns are loaded into registers while the current ones are multiplied out of
// shared memory, with one barrier per BK columns. Each sum is one chain over k
// whatever MR is.
template <int MR, bool DIFF>
__device__ __forceinline__ void gram_tile(const float* __restrict__ A, const float* __restrict__ B, int ld,
                                          float (&acc)[MR][4], GramSmem<MR>& sm) {
  constexpr int NA = MR / 4;                     // 64-row slices of A a loader thread fills
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int lr = tid >> 2, lk = (tid & 3) * 4;   // loader: row, k offset
  const float* arow = A + (int64_t)lr * ld + lk;
  const float* brow = B + (int64_t)lr * ld + lk;
#pragma unroll
  for (int i = 0; i < MR; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.0f;
  float4 a[NA], b;
  auto load = [&](int k0) {
#pragma unroll
    for (int q = 0; q < NA; ++q) a[q] = *reinterpret_cast<const float4*>(arow + (int64_t)q * 64 * ld + k0);
    b = *reinterpret_cast<const float4*>(brow + k0);
  };
  auto store = [&](int buf) {
#pragma unroll
    for (int q = 0; q < NA; ++q) {
      const int r = q * 64 + lr;
      sm.A[buf][lk + 0][r] = a[q].x; sm.A[buf][lk + 1][r] = a[q].y;
      sm.A[buf][lk + 2][r] = a[q].z; sm.A[buf][lk + 3][r] = a[q].w;
    }
    sm.B[buf][lk + 0][lr] = b.x; sm.B[buf][lk + 1][lr] = b.y;
    sm.B[buf][lk + 2][lr] = b.z; sm.B[buf][lk + 3][lr] = b.w;
  };
  load(0);
  __syncthreads();                               // the previous tile's readers are done
  store(0);
  int buf = 0;
  for (int k0 = 0; k0 < ld; k0 += BK, buf ^= 1) {
    const bool more = k0 + BK < ld;
    if (more) load(k0 + BK);
    __syncthreads();                             // this buffer is filled, the other one read
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      float ar[MR];
#pragma unroll
      for (int i = 0; i < MR; i += 4) {
        const float4 av = *reinterpret_cast<const float4*>(&sm.A[buf][kk][ty * MR + i]);
        ar[i] = av.x; ar[i + 1] = av.y; ar[i + 2] = av.z; ar[i + 3] = av.w;
      }
      const float4 bv = *reinterpret_cast<const float4*>(&sm.B[buf][kk][tx * 4]);
      const float br[4] = {bv.x, bv.y, bv.z, bv.w};
#pragma unroll
      for (int i = 0; i < MR; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          if constexpr (DIFF) {
            const float t = ar[i] - br[j];
            acc[i][j] = fmaf(t, t, acc[i][j]);
          } else {
            acc[i][j] = fmaf(ar[i], br[j], acc[i][j]);
          }
        }
    }
    if (more) store(buf ^ 1);
  }
}

// One level of the row sums' tree: N rows' values, half of them handed to the
// lane across `o`, which keeps the other half. The lane whose bit o is set keeps the upper half.
template <int N>
__device__ __forceinline__ void fold_rows(float (&v)[N], int o) {
  const bool up = (threadIdx.x & o) != 0;
#pragma unroll
  for (int i = 0; i < N / 2; ++i) {
    const float keep = up ? v[i + N / 2] : v[i], give = up ? v[i] : v[i + N / 2];
    v[i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
  }
}

// The weighted kernel sums of a tile's rows (16 MR rows, 64 columns): per thread
// four columns in order, then the 16 threads of a row in a tree over lane bits
// 3, 2, 1, 0. The tree works on all of a thread's rows at once, each level
// halving the rows a lane holds: MR + 16 / MR - 1 shuffles or so instead of 4 MR.
template <int KIND, int MR>
__device__ __forceinline__ void dist_simt_sums(const Dev& s, int rows, int t, int row0, const Tile& T,
                                               const float (&acc)[MR][4]) {
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  float yn[4], wy[4];
  int yi[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int c = tx * 4 + j;
    const bool ok = c < T.ncols;
    const int64_t g = (int64_t)T.row0 + (ok ? c : 0);
    yn[j] = s.yn[g];
    yi[j] = s.yi[g];
    wy[j] = ok ? s.w32[g] : 0.0f;
  }
  float v[MR];
#pragma unroll
  for (int i = 0; i < MR; ++i) {
    const int r = row0 + ty * MR + i;
    const int rr = r < rows ? r : 0;
    const float xn = s.xbn[rr];
    const int xi = s.xbi[rr];
    float sum = 0.0f;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const bool same = xi >= 0 && xi == yi[j];
      const float kv = KIND == K_LAPLACE ? exp2f(sqrtf(same ? 0.0f : acc[i][j]) * s.negc)
                                         : kernel_from_gram(KIND, acc[i][j], xn, yn[j], same, s.negc, (float)s.coef0,
                                                            s.degree);
      sum += (tx * 4 + j < T.ncols) ? wy[j] * kv : 0.0f;
    }
    v[i] = sum;
  }
  int row = 0, o = 8;                            // the row this lane ends up with; lanes left to add over
  if constexpr (MR == 8) {
    float (&v8)[8] = v;
    fold_rows(v8, 8);
    row = (tx & 8) >> 1;
    o = 4;
  }
  float v4[4] = {v[0], v[1], v[2], v[3]};
  fold_rows(v4, o);
  row += (tx & o) ? 2 : 0;
  o >>= 1;
  float v2[2] = {v4[0], v4[1]};
  fold_rows(v2, o);
  row += (tx & o) ? 1 : 0;
  o >>= 1;
  float sum = v2[0];
  const int mask = 2 * o - 1;                    // lanes that end up with the same row
  for (; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  const int r = row0 + ty * MR + row;
  if ((tx & mask) == 0 && r < rows) s.part[(int64_t)t * s.bpad + r] = sum;
}

// Item w of a run's distance pass (row tile w % R of support tile w / R; 16 MR rows a tile).
template <int MR>
__device__ __forceinline__ void dist_simt_item(const Dev& s, int rows, int R, int w, GramSmem<MR>& sm) {
  const int t = w / R, row0 = (w % R) * 16 * MR;
  const Tile T = s.tiles[t];
  const float *A = s.xb32 + (int64_t)row0 * s.ld, *B = s.y32 + (int64_t)T.row0 * s.ld;
  float acc[MR][4];
  // Laplacian kernel: ||x - y||^2 from the differences. Through ||x||^2 +
  // ||y||^2 - 2 <x, y> a query row equal to a support row (no data index to
  // recognise it by) keeps d2 ~ eps ||x||^2, which the square root magnifies.
  if (s.kind == K_LAPLACE) {
    gram_tile<MR, true>(A, B, s.ld, acc, sm);
    dist_simt_sums<K_LAPLACE, MR>(s, rows, t, row0, T, acc);
    return;
  }
  gram_tile<MR, false>(A, B, s.ld, acc, sm);
  if (s.kind == K_GAUSS) dist_simt_sums<K_GAUSS, MR>(s, rows, t, row0, T, acc);
  else if (s.kind == K_LINEAR) dist_simt_sums<K_LINEAR, MR>(s, rows, t, row0, T, acc);
  else dist_simt_sums<K_POLY, MR>(s, rows, t, row0, T, acc);
}

template <int MR>
__global__ void __launch_bounds__(NT) k_dist_simt(Dev s, int rows) {
  KKM_GRID_DEP_WAIT();
  KKM_LAUNCH_DEPENDENTS();
  __shared__ __align__(16) GramSmem<MR> sm;
  const int R = (rows + 16 * MR - 1) / (16 * MR);
  const int total = R * (*s.ntiles);
  for (int w = blockIdx.x; w < total; w += gridDim.x) dist_simt_item<MR>(s, rows, R, w, sm);
}

// Pair w of a run's window pass; its four sums go to wpart[w].
__device__ __forceinline__ void wgram_simt_item(const Dev& s, int w, GramSmem<4>& sm, double (*red)[NT / 32]) {
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4, lane = tid & 31, warp = tid >> 5;
  {
    const WPair pr = s.wpairs[w];
    const Plan P = s.plan[pr.j];
    const int64_t base = (int64_t)pr.j * s.cap;
    // row and column ranges, as positions inside the center's region
    int r0, rn, c0, cn;
    if (pr.kind == 0) { r0 = P.head_c; rn = P.ndrop; c0 = P.head_c; cn = P.tail_new - P.head_c; }
    else { r0 = P.tail_c; rn = P.cnt; c0 = P.tail_c; cn = P.cnt; }
    const int rs = r0 + pr.rt * BM, cs = c0 + pr.ct * BN;
    float acc[4][4];
    gram_tile<4, false>(s.y32 + (base + rs) * s.ld, s.y32 + (base + cs) * s.ld, s.ld, acc, sm);
    // FP64 issues at 1/64 of the FP32 rate on this chip. The row weight is taken
    // out of the column sums, and a thread's 16 kernel values go through FP64 once
    // for every class of columns that the item has (0 dropped rows, 1 the rest of
    // the old window, 2 the new block; most items have one): a conversion and one
    // FMA a value. With every value's class decided in the FP64 code 90 % of 8192
    // rows in one of two centers, d = 64, took 2460 us a step, 2000 now.
    const int c1 = pr.kind == 0 ? P.head_new : c0, c2 = pr.kind == 0 ? P.tail_c : c0, cend = c0 + cn;
    float kv[4][4];
    {
      float yn[4];
      int yi[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int64_t q = base + min(cs + tx * 4 + j, cend - 1);
        yn[j] = s.yn[q];
        yi[j] = s.yi[q];
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int64_t p = base + rs + ty * 4 + i;
        const float xn = s.yn[p];
        const int xi = s.yi[p];
#pragma unroll
        for (int j = 0; j < 4; ++j)
          kv[i][j] = kernel_from_gram(s.kind, acc[i][j], xn, yn[j], xi == yi[j], s.negc, (float)s.coef0, s.degree);
      }
    }
    double sum[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int cls = 0; cls < 3; ++cls) {
      const int lo = cls == 0 ? c0 : cls == 1 ? c1 : c2, hi = cls == 0 ? c1 : cls == 1 ? c2 : cend;
      if (max(lo, cs) >= min(hi, cs + BN)) continue;   // the item has no such columns
      double yw[4];
      bool in[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int c = cs + tx * 4 + j;
        in[j] = c >= lo && c < hi;
        yw[j] = cls < 2 && in[j] ? s.wwin64[base + c] : 1.0;
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        if (pr.rt * BM + ty * 4 + i >= rn) continue;
        double r = 0.0;
#pragma unroll
        for (int j = 0; j < 4; ++j) r = fma(yw[j], (double)(in[j] ? kv[i][j] : 0.0f), r);
        sum[cls] = pr.kind == 0 ? fma(s.wwin64[base + rs + ty * 4 + i], r, sum[cls]) : sum[cls] + r;
      }
    }
    const double sA = sum[0] + sum[1], sB = sum[0], sE = pr.kind == 0 ? sum[2] : 0.0, sM = pr.kind == 0 ? 0.0 : sum[2];
    // fixed-order block reduction of the four sums: two levels hand half of them
    // to the other lane, so that lanes 0, 8, 16, 24 end with sA, sE, sB, sM
    {
      const bool hi = lane & 16, up = lane & 8;
      double k0 = hi ? sB : sA, k1 = hi ? sM : sE;
      k0 += __shfl_xor_sync(0xffffffffu, hi ? sA : sB, 16);
      k1 += __shfl_xor_sync(0xffffffffu, hi ? sE : sM, 16);
      double v = up ? k1 : k0;
      v += __shfl_xor_sync(0xffffffffu, up ? k0 : k1, 8);
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      // red[0..3]: sA, sB, sE, sM
      if ((lane & 7) == 0) red[(hi ? 1 : 0) + (up ? 2 : 0)][warp] = v;
    }
    __syncthreads();
    if (tid < 4) {
      double v = 0.0;
      if (tid < 4)
        for (int q = 0; q < NT / 32; ++q) v += red[tid][q];
      s.wpart[(int64_t)w * 4 + tid] = v;
    }
    __syncthreads();
  }
}

__device__ __forceinline__ void wgram_simt_body(const Dev& s, bool norms, int bid, int nblk) {
  KKM_GRID_DEP_WAIT();
  KKM_LAUNCH_DEPENDENTS();
  __shared__ __align__(16) GramSmem<4> sm;
  __shared__ double red[4][NT / 32];
  const int total = *s.nwpairs;
  // Norms are reported by the first warp, whose first four lanes wrote the sums.
  // Many items a block: a contiguous range each, so that its reports are few;
  // few: strided, so that a center's items spread over the chip. FP32, d = 64,
  // 90 % of the batch in one of 10 centers, us a step strided and contiguous:
  // b = 1024 (1.5 items a block) 85 and 92, b = 2048 (6) 221 and 208, b = 8192
  // (75) 2649 and 2459.
  if (total < 4 * nblk) {
    for (int w = bid; w < total; w += nblk) {
      wgram_simt_item(s, w, sm, red);
      if (norms && threadIdx.x < 32) norm_report(s, ItemPlace(s, w, s.wpairs[w].j), 1);
    }
    return;
  }
  const int lo = (int)((int64_t)bid * total / nblk), hi = (int)((int64_t)(bid + 1) * total / nblk);
  NormReports reports(hi);
  for (int w = lo; w < hi; ++w) {
    wgram_simt_item(s, w, sm, red);
    if (norms && threadIdx.x < 32) {
      reports.next(s, w);
      reports.done(s, true);
    }
  }
}

__global__ void __launch_bounds__(NT) k_wgram_simt(Dev s, int norms) {
  wgram_simt_body(s, norms != 0, blockIdx.x, gridDim.x);
}

// Run groups: the items of all the launch's runs laid end to end (distance
// pass: row tiles x support tiles; window pass: pairs), block-strided, so the
// blocks stay busy until the last item of any run. Item w of the flat space is
// item w - off[r] of run r; every item writes only its own partials, so each
// run computes what its own launch would.
constexpr int GROUP_MAX_RUNS = 1024;

template <int MODE>
__global__ void __launch_bounds__(NT) k_group_simt(GroupPhase g) {
  KKM_GRID_DEP_WAIT();
  KKM_LAUNCH_DEPENDENTS();
  __shared__ __align__(16) GramSmem<4> sm;
  __shared__ double red[4][NT / 32];
  __shared__ int off[GROUP_MAX_RUNS + 1];
  const int nr = g.nruns < GROUP_MAX_RUNS ? g.nruns : GROUP_MAX_RUNS;
  for (int r = threadIdx.x; r < nr; r += NT) {
    const Dev& s = g.runs[r].s;
    off[r + 1] = MODE == 0 ? ((s.b + BM - 1) / BM) * (*s.ntiles) : *s.nwpairs;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    off[0] = 0;
    for (int r = 0; r < nr; ++r) off[r + 1] += off[r];
  }
  __syncthreads();
  const int total = off[nr];
  for (int w = blockIdx.x; w < total; w += gridDim.x) {
    int lo = 0, hi = nr;                         // the run r with off[r] <= w < off[r + 1]
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (off[mid] <= w) lo = mid;
      else hi = mid;
    }
    const Dev& s = g.runs[lo].s;
    if constexpr (MODE == 0) dist_simt_item<4>(s, s.b, (s.b + BM - 1) / BM, w - off[lo], sm);
    else wgram_simt_item(s, w - off[lo], sm, red);
  }
}

}  // namespace

// 2048 x 64 batch rows against about 11000 support rows (k = 50): the whole
// iteration took 188 us, 131 of it this pass, with 64-row tiles, one buffer and
// a runtime kernel kind; now 150 us with the window pass's fewer FP64 operations.
// 128-row tiles where the pass still has two items for every SM: a thread's 8 x
// 4 products take three shared-memory reads per 32 FMAs, the 64-row tile's 4 x 4
// two per 16. The number of support tiles is known on the device only; a full
// window has at least tau / 64 of them, a center without one at most none.
cudaError_t launch_dist_simt(const Dev& s, int rows, cudaStream_t st) {
  if (rows <= 0) return cudaSuccess;
  const int64_t tiles = (int64_t)s.k * std::max(1, s.tau / BN);
  if (rows > BM && (rows + 127) / 128 * tiles >= 2 * s.num_sms)
    return launch_pdl(k_dist_simt<8>, dim3(s.num_sms * 3), dim3(NT), 0, st, s, rows);
  return launch_pdl(k_dist_simt<4>, dim3(s.num_sms * 4), dim3(NT), 0, st, s, rows);
}

cudaError_t launch_wgram(const Dev& s, cudaStream_t st, bool norms) {
  return launch_pdl(k_wgram_simt, dim3(s.num_sms * 4), dim3(NT), 0, st, s, norms ? 1 : 0);
}

cudaError_t launch_group_simt(const GroupPhase& g, int mode, int blocks, cudaStream_t st) {
  const dim3 grid(blocks > 0 ? blocks : 1), block(NT);
  return launch_pdl(mode == 0 ? k_group_simt<0> : k_group_simt<1>, grid, block, 0, st, g);
}

}  // namespace kkm
