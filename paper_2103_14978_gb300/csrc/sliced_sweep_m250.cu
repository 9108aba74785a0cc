// Sliced sweep kernels, read length 250 bases: the compiled ranges of shift
// counts, each filtered in one pass.
#include "sliced_kernels.cuh"

namespace gk {

cudaError_t launch_sliced_sweep_m250(int khi, const SlicedArgs &a, cudaStream_t stream) {
  switch (khi) {
    case 5: return launch_sliced_range<0, 5, 250>(a, stream);
    case 7: return launch_sliced_range<6, 7, 250>(a, stream);
    case 8: return launch_sliced_range<6, 8, 250>(a, stream);
    case 10: return launch_sliced_range<6, 10, 250>(a, stream);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace gk
