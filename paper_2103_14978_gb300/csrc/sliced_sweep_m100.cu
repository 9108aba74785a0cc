// Sliced sweep kernels, read length 100 bases: the compiled ranges of shift
// counts, each filtered in one pass.
#include "sliced_kernels.cuh"

namespace gk {

cudaError_t launch_sliced_sweep_m100(int khi, const SlicedArgs &a, cudaStream_t stream) {
  switch (khi) {
    case 5: return launch_sliced_range<0, 5, 100>(a, stream);
    case 7: return launch_sliced_range<6, 7, 100>(a, stream);
    case 8: return launch_sliced_range<6, 8, 100>(a, stream);
    case 10: return launch_sliced_range<6, 10, 100>(a, stream);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace gk
