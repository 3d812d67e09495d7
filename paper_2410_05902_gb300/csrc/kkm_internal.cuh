// Internal declarations shared by the libkkm translation units.
//
// Device state of one run. Everything lives in HBM and is sized at kkm_init;
// nothing is allocated per step.
//
//   support store  k regions of `cap` rows, one per center. Center j's
//                  window (Eq. (1)) occupies rows [head_j, tail_j) of region j,
//                  laid out as C_1 (while kept), then blocks oldest -> newest,
//                  each block in batch order. Appends go at tail. Drops advance
//                  head. When an append would pass the region's end, the
//                  window is first copied down to row 0 ("compaction"). With
//                  cap - REGION_PAD = 2*tau + 4*b + 8 usable rows the source
//                  and destination rows of that copy never overlap, because a
//                  window holds at most tau + b rows. The last REGION_PAD rows
//                  of a region are never used, so a tile (at most 256 rows)
//                  that starts inside the window never reaches the next region.
//   row data       FP32 form: FP32 rows, ld = round_up(d, 16), zero padded.
//                  TF32 form: FP32 rows rounded to TF32, ld = dp = round_up(d, 32).
//                  BF16 forms: BF16 rows [hi(0..dp) | lo(0..dp)], dp =
//                  round_up(d, 64), zero padded; ld = 2*dp.
//   yn             FP32 ||y||^2 of the values the Gram product actually uses
//   yi             int32 data index of the row (the key that forces K(x,x)=1
//                  when a batch point meets its own support copy)
//   w64 / w32      FP64 master weight and its FP32 copy for the distance kernel.
//                  Invariant: both are 0 on every row outside its window, so a
//                  tile may cover rows on either side of a window and read
//                  their weights as they are.
//
// Per-center block ring: (iteration, count) of the window's blocks, oldest
// first, at most tau + 2 entries. C_1 is not in the ring; c1[j] flags it.
#pragma once
#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <stdint.h>
#include <atomic>
#include <type_traits>

namespace kkm {

enum Form : int { FORM_FP32 = 0, FORM_BF16 = 1, FORM_BF16X3 = 2, FORM_TF32 = 3 };

// forms whose row buffers hold FP32 values (xb32 / y32)
__host__ __device__ inline bool f32_rows(int form) { return form == FORM_FP32 || form == FORM_TF32; }
enum KernelKind : int { K_GAUSS = 0, K_LAPLACE = 1, K_LINEAR = 2, K_POLY = 3 };

// device status bits (sticky until the context is destroyed)
constexpr int ST_BAD_BATCH_INDEX = 1;
constexpr int ST_BAD_ASSIGN = 2;
constexpr int ST_CAPACITY = 4;
constexpr int ST_TIMEOUT = 8;

constexpr int REGION_PAD = 256;   // unused rows at the end of each support region (the widest tile)
constexpr int WPASS_TNV = 128;    // tcgen05 window pass: support rows per column tile

// Column tile of the distance pass: support rows [row0, row0 + ncols) of center j.
struct Tile {
  int32_t j;
  int32_t row0;   // global support row
  int32_t ncols;
  int32_t pad;
};

// Tile pair of the window Gram pass (norm recurrence terms), see kkm_step.cu.
struct WPair {
  int32_t j;
  int32_t kind;   // 0: dropped rows x (old window + new block); 1: new block x new block
  int32_t rt;     // row tile index within the row range
  int32_t ct;     // column tile index within the column range
};

// Per-center plan of one update, written by the sort/plan kernel.
struct Plan {
  int32_t head_c;    // window start after compaction
  int32_t tail_c;    // window end after compaction (= start of the new block)
  int32_t head_new;  // window start after the drops
  int32_t tail_new;  // window end after the append
  int32_t src_head;  // compaction source start (-1 when not compacting)
  int32_t cnt;       // b_i^j
  int32_t ndrop;     // rows dropped (C_1 included)
  int32_t c1_new;    // C_1 kept after this update
};

struct alignas(16) Dev {
  // problem
  int64_t n;
  int32_t d, k, b, tau, cap, nbcap;
  int64_t ldx;
  int32_t ld;        // row stride of batch and support rows, in elements
  int32_t dp;        // BF16 forms: padded d (hi part length)
  int32_t form, kind, degree, lr;
  double param, coef0, eta;
  double inv_b;      // 1 / b
  float negc;        // -log2(e) / param (Gaussian, Laplacian)
  int32_t num_sms;
  uint64_t seed;
  int32_t tn;        // support rows per distance tile
  int32_t ppt;       // partials per distance tile in part[] (2 for 256-row tcgen05 tiles: one per column half)
  int32_t pre_b;     // tcgen05 passes: read the tile and pair lists before the grid-dependency wait
                     // (set per launch, where the kernel just ahead writes neither)
  int32_t pair_rows, pair_cols; // window-pass tile: row and column counts (64x64 SIMT, 128x128 tcgen05)
  int32_t walign;    // window-pass tiles start at range starts rounded down to this many rows (1 SIMT, 4 tcgen05)
  int32_t bpad;      // rows of the batch buffers (>= b, multiple of 128)
  int32_t max_tiles, max_pairs;
  const float* X;
  // batch
  float* xb32;       // [bpad * ld]   FP32 form
  __nv_bfloat16* xbh;// [bpad * ld]   BF16 forms
  float* xbn;        // [bpad]
  int32_t* xbi;      // [bpad] data index, -1 for query rows
  // support store
  float* y32;
  __nv_bfloat16* ybh;
  float* yn;
  int32_t* yi;
  double* w64;
  float* w32;
  float* wo32;       // FP32 weights before the last update (k_update), for its window pass
  double* wo64;      // the same in FP64 (FP32 form only, whose window pass reads FP64 weights)
  const float* wwin; // the weights the window pass reads: wo32, or w32 where the pass runs before the update
  const double* wwin64;   // FP32 form: wo64 or w64
  // per center
  int32_t* head;
  int32_t* tail;
  int32_t* c1;
  int32_t* wsum;     // sum of block counts in the window (C_1 excluded)
  double* cnorm;
  float* cnorm32;    // FP32 copy of cnorm for the argmin
  int32_t* blk_iter; // [k * nbcap]
  int32_t* blk_cnt;  // [k * nbcap]
  int32_t* blk_first;
  int32_t* blk_num;
  // step workspaces
  int32_t* assign;   // [bpad] assignment used by the update
  float* mind;       // [bpad]
  float* inner_a;    // [bpad] <phi(x), C_a> at the used assignment a
  int32_t* counts;   // [k]
  double* alpha;     // [k]
  int32_t* coff;     // [k + 1] exclusive offsets of the center-sorted batch
  int32_t* perm;     // [b] batch rows sorted by center (stable)
  int64_t* mvdst;    // [b] support row that sorted batch row w moves to (k_sort_plan), -1 past capacity
  double* cmc;       // [k] <C_j, cm(B_j)>
  Plan* plan;        // [k]
  int32_t* comp_off; // [k] first flat row of each center's compaction copy
  int32_t* comp_total; // [1] rows copied by this step's compactions
  Tile* tiles;       // [max_tiles]
  int32_t* ntiles;   // [1]
  int2* split;       // [nsplit + 1] first window item and first distance item of each CTA of a step's launch
  int32_t nsplit;    // its CTAs
  int32_t tile_floor;  // least work of a tile: its operand copies (see tile_work)
  int32_t win_floor;   // least work of a window item (see window_work)
  int32_t* tile_first; // [k]
  int32_t* tile_cnt;   // [k]
  float* part;       // [max_tiles * ppt * bpad] per-tile weighted kernel sums (ppt partials per tile)
  WPair* wpairs;     // [max_pairs]
  int32_t* nwpairs;  // [1]
  int32_t* wpair_first; // [k]
  int32_t* wpair_cnt;   // [k]
  double* ncum;      // [k] points assigned to each center so far (N^j of the sklearn rate)
  const double* rtab; // [2 (b + 1)]: 1/n at [n] and sqrt(n / b) at [b + 1 + n], n = 0..b (host-computed)
  double* wpart;     // [max_pairs][4 sums]: A, Bdd, E, M partials per window item
  double* wseg;      // [win_segment_slots][4 sums]: the same per segment of a center's items
  int64_t* iter;     // [1] next iteration number
  int32_t* status;   // [1] sticky device status bits
  int32_t* wdone;    // [win_segment_slots] finished items of each segment (k_sort_plan clears them)
  int32_t* cdone;    // [k] finished segments (k_sort_plan clears them)
  int64_t* gnext;    // [1] the iteration whose batch has been scored (its successor's batch may be gathered)
  int64_t* stats;    // [3] steps, support rows, tiles
  double* obj;       // [1] last batch objective
  float* cmpart;     // [k][32] FP32 lane partials of sum_{x in B_j} <phi(x), C_j>
};

// Programmatic dependent launch: every step kernel is launched so that it may
// be scheduled while its predecessor drains. It must wait here before it reads
// anything the predecessor writes (a no-op when launched without the attribute).
#define KKM_GRID_DEP_WAIT() asm volatile("griddepcontrol.wait;" ::: "memory")
// Lets the next kernel in the stream start its pre-wait part. Issued only after
// this kernel's own wait, so that every kernel before it has completed, and by
// every block of it, so that the pre-wait part of the next kernel runs beside
// this one and beside nothing earlier. It may therefore read what kernels before
// this one wrote, and write what only they read. Before their wait work:
//   the tcgen05 passes: set up shared memory and TMEM and read the tile and pair
//     lists (where the kernel ahead writes none of them: Dev::pre_b)
//   k_argmin: the tile tables, the batch rows' norms, forced assignments
//   k_finalize (run groups): plans, counts, norms and partials of the sort/plan
//   k_update, its gather of the next batch into the other buffer set: beside it
//     runs the sort/plan, which reads no batch rows. The last readers of that set
//     were the previous step's row moves, and the distance pass and the argmin of
//     this step have completed since. It reads the data, the caller's indices and
//     the counter that the argmin left (gnext)
//   k_gather_query, ahead of a chunk, into the other buffer set: beside it runs a
//     chunk's distance pass, which reads its own set; the last readers of the
//     other one, the kernels of the chunk before, have completed
//   k_pp_draw: stages rows of the data
// All others wait at their first statement.
#define KKM_LAUNCH_DEPENDENTS() asm volatile("griddepcontrol.launch_dependents;" ::: "memory")

// Raises `kern`'s dynamic shared-memory limit to `bytes` on the current device,
// once per device: the attribute belongs to the function on that device.
// `done` is the caller's per-kernel mask of devices already set.
template <typename Kern>
inline cudaError_t smem_limit_once(Kern kern, int bytes, std::atomic<uint64_t>& done) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const uint64_t bit = dev < 64 ? (uint64_t)1 << dev : 0;
  if (bit && (done.load(std::memory_order_relaxed) & bit)) return cudaSuccess;
  e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess) done.fetch_or(bit, std::memory_order_relaxed);
  return e;
}

// Launches `kern` with the programmatic-stream-serialization attribute.
template <typename... Params, typename... Args>
inline cudaError_t launch_pdl(void (*kern)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                              Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, static_cast<Params>(args)...);
}

// ---------------------------------------------------------------- helpers
// Work of a distance tile in units of one 16-column chunk of an epilogue group
// (about 470 cycles): five for what an item costs whatever its width, one per
// chunk of its wider column half, and at least what its operand copies take.
// With the items split by count the CTAs of the 1e6 x 128 workload's launch
// ended 44.9 to 56.8 us after its start, split by work 41 to 49.
__host__ __device__ inline int tile_work(int ncols, int tn, int floor_) {
  const int half = tn == 256 ? 128 : tn;
  const int w = 5 + ((ncols < half ? ncols : half) + 15) / 16;
  return w > floor_ ? w : floor_;
}

// Work of a window item beside tiles of tn rows, on the same scale: a 128 x 128
// item takes a CTA about 4380 cycles where a full 256-row distance tile takes
// 3690 (8192 x 64, BF16), narrow ones hardly less (weights by their columns made
// the 1e6 x 128 workload 3 to 5 % slower), and all of them at least their
// operand copies. few: the launch has so few items that all epilogue groups
// work on each; then its reductions weigh most.
__host__ __device__ inline int window_work(int tn, bool few, int floor_) {
  const int w = few ? 22 : tn == 256 ? 15 : 30;
  return w > floor_ ? w : floor_;
}

__device__ __forceinline__ double warp_sum_f64(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// alpha_i^j for b_j = n > 0 points, N points in all (this batch included), beta = sqrt(b_j / b).
__device__ __forceinline__ double learning_rate(const Dev& s, double n, double N, double beta) {
  if (s.lr == 0) return beta;
  return s.lr == 2 ? n / N : s.eta;    // sklearn: the running-mean rate
}

// Sec. 4: ||C'||^2 = (1-a)^2 ||R||^2 + 2a(1-a) <R, m> + a^2 ||m||^2 with m =
// cm(B_j) and R = C - D, the part of the old center Eq. (1) keeps. cmc =
// <C, m>, inv_n = 1 / b_j. One function for every caller, so that a run's
// norms come out the same to the bit however its launches are grouped.
static __device__ __noinline__ double norm_recurrence(double a, double cmc, double inv_n, double cn_old, double A,
                                                      double Bdd, double E, double M) {
  const double keep = 1.0 - a;
  const double m2 = M * inv_n * inv_n;
  const double R2 = cn_old - 2.0 * A + Bdd;
  const double Rm = cmc - E * inv_n;
  return keep * keep * R2 + 2.0 * a * keep * Rm + a * a * m2;
}

// The window items of a center are added up in segments of WSEG items, then the
// segments' sums: a center's items grow with the square of its rows (two at 40
// rows, 768 at 1900), and as one list read by the warp that finishes the last
// of them the sum was tens of microseconds that the argmin waits for. A segment
// is summed by the warp that finishes the last item in it, wherever that runs,
// with all its loads in flight at once. 90 % of the batch in one of 10 centers,
// d = 64, us a step with one list and with segments: BF16 b = 4096 120 and 88,
// b = 8192 392 and 276; FP32 b = 2048 346 and 208, b = 8192 4683 and 2459.
constexpr int WSEG = 64;
__host__ __device__ inline int win_segments(int items) { return (items + WSEG - 1) / WSEG; }
// Place of the first segment of center j, whose items start at `first`: no two
// centers' segments meet, and all lie below win_segment_slots.
__host__ __device__ inline int win_segment_slot(int first, int j) { return first / WSEG + j; }
__host__ __device__ inline int win_segment_slots(int items, int k) { return items / WSEG + k + 1; }

// Sums of n / 4 partials of four values each by a warp (element e belongs to
// value e & 3): lane l ends with value l & 3. One order for every caller.
__device__ __forceinline__ double sum_partials(const double* p, int n) {
  const int lane = threadIdx.x & 31;
  double acc = 0.0;
  for (int e0 = 0; e0 < n; e0 += 256) {
    double v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int e = e0 + 32 * u + lane;
      v[u] = e < n ? __ldcg(p + e) : 0.0;
    }
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (e0 + 32 * u < n) acc += v[u];
  }
#pragma unroll
  for (int o = 4; o < 32; o <<= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  return acc;
}

// Whether this warp's `m` arrivals are the last of `of` on the counter; what
// the earlier ones wrote before theirs is then visible. (Release and acquire on
// the atomic itself.)
__device__ __forceinline__ bool last_arrival(int32_t* counter, int m, int of) {
  int last = 0;
  __syncwarp();
  if ((threadIdx.x & 31) == 0) {
    int before;
    asm volatile("atom.add.acq_rel.gpu.global.s32 %0, [%1], %2;" : "=r"(before) : "l"(counter), "r"(m) : "memory");
    last = before + m == of;
  }
  last = __shfl_sync(0xffffffffu, last, 0);
  __syncwarp();
  return last != 0;
}

// Where a window item's sums go.
struct ItemPlace {
  int j, first, cnt, q;   // its center, that center's first item and their number, its segment
  __device__ ItemPlace() {}
  __device__ ItemPlace(const Dev& s, int item, int j_)
      : j(j_), first(s.wpair_first[j_]), cnt(s.wpair_cnt[j_]), q((item - first) / WSEG) {}
};

// A warp's report of m finished window items of a segment (their sums are in
// wpart): the last of a segment adds it up, the last of a center's segments adds
// those and carries ||C_j||^2 through the update. A fence and an atomic take
// longer than an item's arithmetic, so consecutive items of a segment are
// reported together (NormReports).
__device__ __forceinline__ void norm_report(const Dev& s, const ItemPlace& at, int m) {
  const int lane = threadIdx.x & 31, j = at.j, q = at.q, first = at.first;
  const int nseg = win_segments(at.cnt), slot = win_segment_slot(first, j), here = min(WSEG, at.cnt - q * WSEG);
  if (!last_arrival(s.wdone + slot + q, m, here)) return;
  const int n = s.plan[j].cnt;
  const double part = (double)s.cmpart[(int64_t)j * 32 + lane];
  const double inv_n = s.rtab[n], a = s.alpha[j], cn_old = s.cnorm[j];
  double qt = sum_partials(s.wpart + (int64_t)(first + q * WSEG) * 4, here * 4);
  if (nseg > 1) {
    if (lane < 4) __stcg(s.wseg + (int64_t)(slot + q) * 4 + lane, qt);
    __syncwarp();
    if (!last_arrival(s.cdone + j, 1, nseg)) return;
    qt = sum_partials(s.wseg + (int64_t)slot * 4, nseg * 4);
  }
  const double A = __shfl_sync(0xffffffffu, qt, 0), Bdd = __shfl_sync(0xffffffffu, qt, 1);
  const double E = __shfl_sync(0xffffffffu, qt, 2), M = __shfl_sync(0xffffffffu, qt, 3);
  const double cmc = warp_sum_f64(part) * inv_n;
  if (lane == 0) {
    const double cn = norm_recurrence(a, cmc, inv_n, cn_old, A, Bdd, E, M);
    s.cmc[j] = cmc;
    s.cnorm[j] = cn;
    s.cnorm32[j] = (float)cn;
  }
}

// Gathers the reports of a warp that finishes items in order up to hi - 1: one
// per segment. next: the item it waits for; done: that item is finished (ok) or
// was skipped, and then its center keeps its norm.
struct NormReports {
  int hi, m = 0;
  ItemPlace at;
  bool send = false;
  __device__ explicit NormReports(int hi_) : hi(hi_) {}
  __device__ __forceinline__ void next(const Dev& s, int item) {
    const int j = s.wpairs[item].j, jn = item + 1 < hi ? s.wpairs[item + 1].j : -1;
    at = ItemPlace(s, item, j);
    send = jn != j || (item + 1 - at.first) % WSEG == 0;
  }
  __device__ __forceinline__ void done(const Dev& s, bool ok) {
    m += ok ? 1 : 0;
    if (!send) return;
    if (m > 0) norm_report(s, at, m);
    m = 0;
  }
};

__host__ __device__ inline int64_t round_up(int64_t a, int64_t m) { return (a + m - 1) / m * m; }

// SplitMix64 (Steele, Lea, Flood 2014): output `counter` of the sequential
// generator seeded with `seed`, i.e. the finaliser applied to
// seed + (counter + 1) * golden gamma.
__host__ __device__ inline uint64_t splitmix64(uint64_t seed, uint64_t counter) {
  uint64_t z = seed + (counter + 1ull) * 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

// Lemire's multiply-high reduction of a 64-bit value onto [0, n).
__host__ __device__ inline int64_t index_below(uint64_t h, uint64_t n) {
#ifdef __CUDA_ARCH__
  return (int64_t)__umul64hi(h, n);
#else
  return (int64_t)(((unsigned __int128)h * n) >> 64);
#endif
}

// Kernel value from the Gram entry g = <x,y> and the squared norms, in FP32.
// `same` forces ||x - y|| = 0 when x and y are the same data point.
__device__ __forceinline__ float kernel_from_gram(int kind, float g, float xn, float yn, bool same,
                                                  float negc, float coef0, int degree) {
  if (kind == K_GAUSS || kind == K_LAPLACE) {
    float d2 = fmaxf(fmaf(-2.0f, g, xn + yn), 0.0f);
    if (same) d2 = 0.0f;
    float arg = (kind == K_GAUSS) ? d2 : sqrtf(d2);
    return exp2f(arg * negc);       // negc = -log2(e) / param
  }
  if (kind == K_LINEAR) return g;
  float base = g + coef0, r = 1.0f;
  for (int p = 0; p < degree; ++p) r *= base;
  return r;
}

// K(x, x) from ||x||^2 (FP64, for the distance formula).
__host__ __device__ inline double kernel_self(int kind, double xn, double coef0, int degree) {
  if (kind == K_GAUSS || kind == K_LAPLACE) return 1.0;
  if (kind == K_LINEAR) return xn;
  double base = xn + coef0, r = 1.0;
  for (int p = 0; p < degree; ++p) r *= base;
  return r;
}

// Table form of Algorithm 1 (kkm_config.algo = KKM_ALGO_TABLE).
struct TabBuf {
  float* T;            // [k][n] <phi(x), C_j>, center-major
  int32_t* bs_off;     // [k+1] start of each center's rows in the support buffer (whole tiles)
  const float* part;   // the Gram view's per-tile partials, [tiles][npad]
  int64_t npad;        // row stride of part (round_up(n, 128))
  int32_t bs_rows;     // rows of the support buffer (k * cap + 256)
};

// s + e = a + b exactly (Knuth's two-sum).
__device__ __forceinline__ float two_sum(float a, float b, float& e) {
  const float s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
  return s;
}

// ------------------------------------------------------------ launchers
// All return cudaGetLastError() of their launches.
cudaError_t launch_gather_batch(const Dev& s, const int32_t* idx, cudaStream_t st);
// id0 >= 0: the rows are the data points id0 ..; ahead: see k_gather_query
cudaError_t launch_gather_query(const Dev& s, const float* Q, int64_t ldq, int rows, int64_t id0, bool ahead,
                                cudaStream_t st);
cudaError_t launch_dist_simt(const Dev& s, int rows, cudaStream_t st);
// obj_acc: each block's FP64 sum of its rows' minima goes to obj_acc[block], or (obj_first false) is added to it
cudaError_t launch_argmin(const Dev& s, int rows, const int32_t* forced, int32_t* assign_out,
                          float* mind_out, float* dist_out, bool update, cudaStream_t st, double* obj_acc = nullptr,
                          bool obj_first = false);
cudaError_t launch_sum(const double* a, int n, double* out, cudaStream_t st);   // sum of n doubles
cudaError_t launch_sort_plan(const Dev& s, double* obj_out, cudaStream_t st);
cudaError_t launch_move(const Dev& s, cudaStream_t st);
// The row moves and the weight update in one launch; with next, the gather of
// the following batch beside them, into next's batch buffers (next_idx: its
// indices, or NULL for the built-in sampler).
cudaError_t launch_update(const Dev& s, const Dev* next, const int32_t* next_idx, cudaStream_t st);
// norms: every center's norm follows its last item (after k_update)
cudaError_t launch_wgram(const Dev& s, cudaStream_t st, bool norms = false);
cudaError_t launch_finalize(const Dev& s, cudaStream_t st);
// batch objective at fixed assignments and its adjoint (kkm_grad.cu): two
// launches. ws holds grad_workspace_doubles(s, m) doubles, zeroed when it is
// allocated (its first int is the row kernel's finished-block counter, which
// every call leaves at zero). With grad_q == NULL only the forward runs
// (loss, delta); otherwise the adjoint (grad_q, grad_s).
// kernel k-means++ seeding (kkm_seed.cu): chosen[0..k) on the device;
// d2 holds n doubles, part kmeanspp_blocks doubles, done one word
int64_t kmeanspp_blocks(int64_t n, int d, int num_sms);
cudaError_t launch_kmeanspp(const float* X, int64_t n, int d, int64_t ldx, int k, int kind, double param,
                            double coef0, int degree, uint64_t seed, int num_sms, double* d2, double* part,
                            int64_t* chosen, unsigned* done, cudaStream_t st);
size_t grad_workspace_doubles(const Dev& s, int64_t m);
cudaError_t launch_objective(const Dev& s, double log_sigma, const float* Q, int64_t m, int64_t ldq,
                             const int32_t* assign, double* loss, float* delta, const double* grad_loss,
                             float* grad_q, int64_t ldg, double* grad_s, double* ws, cudaStream_t st);
cudaError_t launch_build_tiles(const Dev& s, cudaStream_t st);
cudaError_t launch_init_centers(const Dev& s, const int32_t* init_idx, cudaStream_t st);
cudaError_t launch_load_rows(const Dev& s, int32_t rows_total, cudaStream_t st);
cudaError_t launch_tab_batch_dist(const Dev& s, const TabBuf& q, int rows, const int32_t* forced,
                                  int32_t* assign_out, float* mind_out, float* dist_out, bool update, cudaStream_t st);
cudaError_t launch_tab_plan(const Dev& s, const TabBuf& q, double* obj_out, cudaStream_t st);
cudaError_t launch_tab_fill(const Dev& s, const TabBuf& q, cudaStream_t st);
cudaError_t launch_tab_center(const Dev& s, const TabBuf& q, cudaStream_t st);
cudaError_t launch_tab_update(const Dev& s, const TabBuf& q, bool init, cudaStream_t st);
cudaError_t launch_tab_init(const Dev& s, const Dev& g, const TabBuf& q, const int32_t* init_idx, cudaStream_t st);
cudaError_t launch_tab_objective(const Dev& s, const TabBuf& q, const float* xn, double* blk, int nblk,
                                 cudaStream_t st);
cudaError_t launch_mind_sum(const Dev& s, int rows, double scale, double* out, cudaStream_t st);  // scale * sum of mind

// --------------------------------------------------------------- run groups
// A run of a group as the group's launches see it: its four TMA descriptors
// (tc_prepare's layout, used in place by the tcgen05 passes) and its Dev.
struct alignas(64) GroupRun {
  unsigned char maps[512];
  Dev s;
};
static_assert(sizeof(GroupRun) % 64 == 0, "descriptors of consecutive runs stay 64-byte aligned");
// One launch over several runs. The step phases: runs[r] owns blocks
// [first[r], first[r + 1]) and each of them plays one block of that run's own
// launch. The Gram passes read no `first`: they spread the runs' items over
// the launch on the device (kkm_gram_tc.cuh, kkm_gram_simt.cu).
struct GroupPhase {
  const GroupRun* runs;   // device
  const int32_t* first;   // device, nruns + 1 entries, non-decreasing, first[0] = 0
  int32_t nruns;
};
cudaError_t launch_group_gather(const GroupPhase& g, int blocks, cudaStream_t st);
cudaError_t launch_group_argmin(const GroupPhase& g, int blocks, cudaStream_t st);
cudaError_t launch_group_sort_plan(const GroupPhase& g, int smem, cudaStream_t st);   // one block per run
cudaError_t launch_group_move(const GroupPhase& g, int blocks, cudaStream_t st);
cudaError_t launch_group_finalize(const GroupPhase& g, int blocks, cudaStream_t st);
// distance pass (mode 0) or window pass (mode 1) of runs that share the form,
// kernel kind and distance tile: tcgen05 (ctas persistent CTAs) ...
cudaError_t launch_group_tc(const GroupPhase& g, int mode, int form, int kind, int tn, int ctas, cudaStream_t st);
// ... or the FP32 CUDA-core passes
cudaError_t launch_group_simt(const GroupPhase& g, int mode, int blocks, cudaStream_t st);
int sort_plan_smem(int k, int b);

// ------------------------------------------------ full-batch kernel Lloyd
// The Gram view's Dev (xb*: every row of X in the operand form, y*: the
// support buffer of X sorted by center) plus these buffers (kkm_lloyd.cu).
constexpr int LLOYD_RANK_ROWS = 1024;   // rows per chunk of the counting sort's ranking
struct LloydBuf {
  float* T;               // [k][n] <phi(x), C_j>, center-major
  int32_t* assign;        // [n] assignment at the current centers
  float* mind;            // [n] min_j Delta(x, C_j) at the current centers
  int32_t* rank;          // [n] rank of x among the rows of its center within its ranking chunk
  int32_t* ccnt;          // [nrk][k] rows of center j in ranking chunk c (chunk-major)
  int32_t* cbase;         // [nrk][k] position of chunk c's first row of center j within center j
  int32_t* bs_off;        // [k + 1] first support-buffer row of each center (blocks of whole tiles)
  double* blk;            // [nblk] objective partials of the assignment pass
  int32_t* blk_changed;   // [nblk] changed-assignment partials
  double* obj;            // [1] f_X at the current centers
  int64_t* changed;       // [1] rows whose assignment the last assignment pass changed
  int32_t nrk;            // ranking chunks, ceil(n / LLOYD_RANK_ROWS)
  int32_t nblk;           // blocks of the assignment pass
};
// counting sort of X by assignment: ranks, then offsets, tiles and weights 1/n_j
cudaError_t launch_lloyd_sort(const Dev& g, const LloydBuf& L, cudaStream_t st);
// the center-sorted rows into the support buffer
cudaError_t launch_lloyd_scatter(const Dev& g, const LloydBuf& L, cudaStream_t st);
// T[j][row0 + r] from the Gram pass partials of one chunk of rows (gc: the chunk's view);
// all: every center (initial centers), else only centers with rows
cudaError_t launch_lloyd_reduce(const Dev& gc, const LloydBuf& L, int64_t row0, int rows, bool all, cudaStream_t st);
// ||C_j||^2 = (1/n_j) sum_{x in X_j} T[j][x] for the centers with rows
cudaError_t launch_lloyd_cnorm(const Dev& g, const LloydBuf& L, cudaStream_t st);
// argmin over the centers for every row, f_X and the changed count; first: every row counts as changed
cudaError_t launch_lloyd_assign(const Dev& g, const LloydBuf& L, bool first, cudaStream_t st);
// Delta(x, C_j) for every row and center, FP32 (n x k row-major)
cudaError_t launch_lloyd_dist(const Dev& g, const LloydBuf& L, float* out, cudaStream_t st);

// tensor-core passes (BF16, split-BF16 and TF32 forms)
// maps: 512 bytes, 64-byte aligned, holding the four CUtensorMap of the passes
cudaError_t tc_prepare(Dev& s, void* maps);
// one bounded mbarrier wait and one hand-over (the passes' own), limited to limit_ns; out: four ints (k_wait_probe)
cudaError_t launch_wait_probe(uint64_t limit_ns, int arrive, int* out, cudaStream_t st);
// bytes the tcgen05 passes copy per item against a B tile of `cols` rows; with_a: its A tile too
int64_t tc_item_bytes(const Dev& s, int cols, bool with_a);
// partials the distance pass writes per tile of tn support rows (Dev::ppt)
int tc_parts_per_tile(int tn);
// stage_early: the kernel just ahead on `st` (the batch gather, or this pass
// itself) writes neither the tile list nor the pair list and plans, so the
// pass may read them before its grid-dependency wait.
cudaError_t launch_dist_tc(const Dev& s, const void* maps, int rows, cudaStream_t st, bool stage_early = false);
// The window pass reads its pair list and plans before its grid-dependency
// wait: launch it only right after k_move, k_update or a kernel that writes neither.
cudaError_t launch_wgram_tc(const Dev& s, const void* maps, cudaStream_t st, bool norms = false);
// The distance pass on CTA pairs (streamed operands, s.tn 128 or 256).
cudaError_t launch_dist_pair(const Dev& s, const void* maps, int rows, cudaStream_t st);
// A step's distance pass with the window items of the update before it ahead
// of it and their center norms; s.tn 128 or 256.
cudaError_t launch_step_tc(const Dev& s, const void* maps, cudaStream_t st);

}  // namespace kkm
