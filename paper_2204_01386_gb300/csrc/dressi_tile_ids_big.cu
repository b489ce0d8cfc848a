// dressi_tile_ids_big.cu -- per-tile kernel, adjoint from stored layer ids, for faces of many pixels
// (a warp at one face adds its gradients up first).
#include "dressi_tile.cuh"

namespace dressi {
template void launch_tile_mode<9>(const Globals &g, cudaStream_t s);
}  // namespace dressi
