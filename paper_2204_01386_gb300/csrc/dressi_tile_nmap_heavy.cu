// dressi_tile_nmap_heavy.cu -- dressi_tile_heavy.cu's kernel with the normal map compiled in.
#include "dressi_tile.cuh"

namespace dressi {
template void launch_heavy_mode<6>(const Globals &g, cudaStream_t s);
}  // namespace dressi
