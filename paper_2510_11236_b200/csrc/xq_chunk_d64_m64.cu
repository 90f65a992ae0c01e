// Chunk attention kernels for head_dim 64, 64 query rows per CTA.
#include "xq_chunk.cuh"

namespace xq {
template cudaError_t launch_chunk_t<64, 4>(const ChunkParams&, cudaStream_t);
}  // namespace xq
