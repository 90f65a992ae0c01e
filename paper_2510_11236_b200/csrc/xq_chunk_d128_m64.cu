// Chunk attention kernels for head_dim 128, 64 query rows per CTA.
#include "xq_chunk.cuh"

namespace xq {
template cudaError_t launch_chunk_t<128, 4>(const ChunkParams&, cudaStream_t);
}  // namespace xq
