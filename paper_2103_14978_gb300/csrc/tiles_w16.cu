// Batched filter in sorted tiles, reads of at most 16 words.
#include "batched_tiles.cuh"

namespace gk {

cudaError_t launch_tiles_w16(const BatchArgs &a, cudaStream_t s) { return launch_tiles<16>(a, s); }

}  // namespace gk
