// A step's tcgen05 launch: the window items of the update before and the
// distance items of the batch (mode 2 of kkm_gram_tc.cuh), in a translation
// unit of its own so that the two sets of kernels compile in parallel.
#include "kkm_gram_tc.cuh"

namespace kkm {

cudaError_t launch_step_tc(const Dev& s, const void* maps, cudaStream_t st) {
  if (s.tn == 256) return launch_mode<2, 256>(s, maps, s.b, true, st);
  return launch_mode<2, 128>(s, maps, s.b, true, st);
}

}  // namespace kkm
