// tcgen05 / TMA Gram passes of one run: the tensor maps, the launch
// configuration and the entry points of kkm_internal.cuh. The kernels are in
// kkm_gram_tc.cuh.
#include "kkm_gram_tc.cuh"

namespace kkm {
namespace {

// The passes' failure-detection paths, by thread 0. First its bounded wait on an
// mbarrier of one arrival; with arrive = 0 nothing arrives, so the wait runs out
// after limit_ns and out[0] = 1. Then a hand-over through a slot that holds 7
// and, with arrive = 0, is never freed: out[1] = 1 if it was refused, out[2] the
// slot's value, out[3] = 1 if its reader was told.
__global__ void k_wait_probe(uint64_t limit_ns, int arrive, int* out) {
  __shared__ __align__(8) uint64_t bar, empty, full;
  __shared__ int32_t slot;
  if (threadIdx.x != 0) return;
  slot = 7;
  mbar_init(&bar, 1);
  mbar_init(&empty, 1);
  mbar_init(&full, 1);
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  if (arrive) {
    mbar_arrive(&bar);
    mbar_arrive(&empty);
  }
  out[0] = mbar_wait(&bar, 0, limit_ns) ? 0 : 1;
  out[1] = slot_put(&empty, 0, &slot, 3, &full, limit_ns) ? 0 : 1;
  out[2] = slot;
  out[3] = mbar_try_wait(&full, 0) ? 1 : 0;
  mbar_inval(&bar);
  mbar_inval(&empty);
  mbar_inval(&full);
}

}  // namespace

cudaError_t launch_wait_probe(uint64_t limit_ns, int arrive, int* out, cudaStream_t st) {
  k_wait_probe<<<1, 32, 0, st>>>(limit_ns, arrive, out);
  return cudaGetLastError();
}

// Tensor maps of the batch rows and the support store: 2-D tensors of ld
// columns (BF16, or FP32 for the TF32 form), boxes of one 128-byte row of
// columns (64 BF16 or 32 FP32) x 128 (64, 256) rows, 128-byte swizzle.
cudaError_t tc_prepare(Dev& s, void* maps_out) {
  static PFN_cuTensorMapEncodeTiled_v12000 encode = nullptr;
  if (!encode) {
    cudaDriverEntryPointQueryResult q;
    void* fn = nullptr;
    cudaError_t e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000,
                                                     cudaEnableDefault, &q);
    if (e != cudaSuccess || q != cudaDriverEntryPointSuccess || !fn) return cudaErrorNotSupported;
    encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
  }
  CUtensorMap* maps = static_cast<CUtensorMap*>(maps_out);
  const int64_t srows = (int64_t)s.k * s.cap + 256;
  const bool f32 = s.form == FORM_TF32;
  void* xb = f32 ? (void*)s.xb32 : (void*)s.xbh;
  void* yb = f32 ? (void*)s.y32 : (void*)s.ybh;
  const int esz = f32 ? 4 : 2;
  struct { void* base; uint64_t rows; uint32_t box_rows; } ops[4] = {
      {xb, (uint64_t)s.bpad, 128u}, {yb, (uint64_t)srows, 128u}, {yb, (uint64_t)srows, 64u},
      {yb, (uint64_t)srows, 256u}};
  for (int i = 0; i < 4; ++i) {
    cuuint64_t dims[2] = {(cuuint64_t)s.ld, (cuuint64_t)ops[i].rows};
    cuuint64_t strides[1] = {(cuuint64_t)s.ld * esz};
    cuuint32_t box[2] = {(cuuint32_t)(128 / esz), ops[i].box_rows};
    cuuint32_t estr[2] = {1, 1};
    CUresult r = encode(&maps[i], f32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2,
                        ops[i].base, dims, strides, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                        CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return cudaErrorInvalidValue;
  }
  return cudaSuccess;
}

// Whether a launch's batch tile stays in shared memory between items (layout()).
static bool tc_resident(const Dev& s, int cols) {
  const int64_t nsl = s.dp / (s.form == FORM_TF32 ? 32 : KS) * (s.form == FORM_BF16X3 ? 2 : 1);
  return nsl * A_BYTES <= A_RES_MAX && (RING_BYTES - nsl * A_BYTES) / (nsl * cols * KS * 2) >= 2;
}

int64_t tc_item_bytes(const Dev& s, int cols, bool with_a) {
  const int nsl = s.dp / (s.form == FORM_TF32 ? 32 : KS) * (s.form == FORM_BF16X3 ? 2 : 1);
  const int64_t b = (int64_t)nsl * cols * KS * 2, a = (int64_t)nsl * A_BYTES;
  return b + (with_a || !tc_resident(s, cols) ? a : 0);
}

int tc_parts_per_tile(int tn) {
  return tn == 256 ? Geo<256>::GPT : tn == 64 ? Geo<64>::GPT : Geo<128>::GPT;
}

cudaError_t launch_dist_tc(const Dev& s, const void* maps, int rows, cudaStream_t st, bool stage_early) {
  if (rows <= 0) return cudaSuccess;
  // staging before the grid-dependency wait is only safe when the kernel just
  // ahead writes none of what it stages (the gather, or this pass itself)
  Dev d = s;
  d.pre_b = (stage_early && s.pre_b) ? 1 : 0;
  // CTA pairs where the operands stream, an item's MMAs are long (16 or more
  // times a BF16 slice's four) or two items share a row tile's slices
  // (128-column tiles), and the row tiles pair up with little left over: an odd
  // last one costs the pair a whole one. Shorter items are bound by the
  // epilogue, and a pair waits for the slower of its two. Scoring 20000 rows
  // against 64 centers of about 216 rows, pairs and single CTAs: BF16 d = 256 (4
  // slices) 543 and 494 us, d = 784 (13) 914 and 922; split BF16 d = 128 (6 slices'
  // MMAs) 582 and 521, d = 256 (12) 797 and 735, d = 784 (39) 1773 and 1932; TF32
  // d = 128 (4) 538 and 485, d = 784 (25) 1381 and 1463.
  const int R = (rows + TM - 1) / TM;
  const int mmas = d.dp / (d.form == FORM_TF32 ? 32 : KS) * (d.form == FORM_BF16X3 ? 3 : 1);
  if (d.tn >= 128 && !tc_resident(d, d.tn) && (d.tn == 128 || mmas >= 16) && R >= 2 && (R % 2 == 0 || R >= 5))
    return launch_dist_pair(d, maps, rows, st);
  if (d.tn == 64) return launch_mode<0, 64>(d, maps, rows, false, st);
  if (d.tn == 256) return launch_mode<0, 256>(d, maps, rows, false, st);
  return launch_mode<0, 128>(d, maps, rows, false, st);
}

cudaError_t launch_wgram_tc(const Dev& s, const void* maps, cudaStream_t st, bool norms) {
  return launch_mode<1, WPASS_TNV>(s, maps, 0, norms, st);
}

}  // namespace kkm
