// The distance pass on CTA pairs (kkm_gram_tc.cuh), in a translation unit of its
// own so that the sets of kernels compile in parallel.
#include "kkm_gram_tc.cuh"

namespace kkm {

template <int TNV>
static cudaError_t launch_pair(const Dev& s, const void* maps, int rows, cudaStream_t st) {
  const CUtensorMap* m = static_cast<const CUtensorMap*>(maps);
  switch (s.form) {
    case FORM_BF16X3: return launch_pair_kind<OP_X3, TNV>(s, m, rows, st);
    case FORM_TF32: return launch_pair_kind<OP_TF32, TNV>(s, m, rows, st);
    default: return launch_pair_kind<OP_BF16, TNV>(s, m, rows, st);
  }
}

cudaError_t launch_dist_pair(const Dev& s, const void* maps, int rows, cudaStream_t st) {
  return s.tn == 256 ? launch_pair<256>(s, maps, rows, st) : launch_pair<128>(s, maps, rows, st);
}

}  // namespace kkm
