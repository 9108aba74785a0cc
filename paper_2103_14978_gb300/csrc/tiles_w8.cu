// Batched filter in sorted tiles, reads of at most 8 words.
#include "batched_tiles.cuh"

namespace gk {

cudaError_t launch_tiles_w8(const BatchArgs &a, cudaStream_t s) { return launch_tiles<8>(a, s); }

}  // namespace gk
