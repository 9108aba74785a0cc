// Sliced sweep kernels, reads of any length up to GK_SLICED_MAX_LEN (a test
// per position): the compiled ranges of shift counts, each filtered in one pass.
#include "sliced_kernels.cuh"

namespace gk {

cudaError_t launch_sliced_sweep_m0(int khi, const SlicedArgs &a, cudaStream_t stream) {
  switch (khi) {
    case 5: return launch_sliced_range<0, 5, 0>(a, stream);
    case 7: return launch_sliced_range<6, 7, 0>(a, stream);
    case 8: return launch_sliced_range<6, 8, 0>(a, stream);
    case 10: return launch_sliced_range<6, 10, 0>(a, stream);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace gk
