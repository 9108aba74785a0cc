// Batched filter in sorted tiles, reads of at most 4 words.
#include "batched_tiles.cuh"

namespace gk {

cudaError_t launch_tiles_w4(const BatchArgs &a, cudaStream_t s) { return launch_tiles<4>(a, s); }

}  // namespace gk
