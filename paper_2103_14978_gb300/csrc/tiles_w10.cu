// Batched filter in sorted tiles, reads of at most 10 words.
#include "batched_tiles.cuh"

namespace gk {

cudaError_t launch_tiles_w10(const BatchArgs &a, cudaStream_t s) { return launch_tiles<10>(a, s); }

}  // namespace gk
