// dressi_tile_ids_many.cu -- per-tile kernel, adjoint from stored layer ids, CTAs of 128 threads (many
// 16 px tiles).
#include "dressi_tile.cuh"

namespace dressi {
template void launch_tile_mode<8>(const Globals &g, cudaStream_t s);
}  // namespace dressi
