// dressi_tile_heavy.cu -- per-tile kernel of the forward with a cluster of CTAs for each tile that has a
// long face list.
#include "dressi_tile.cuh"

namespace dressi {
template void launch_heavy_mode<0>(const Globals &g, cudaStream_t s);
extern template void launch_heavy_mode<6>(const Globals &g, cudaStream_t s);

void launch_tile_heavy(const Globals &g, cudaStream_t s)
{
    if (g.shade_mode == 3) launch_heavy_mode<6>(g, s);
    else launch_heavy_mode<0>(g, s);
    count_launch(1);
}
}  // namespace dressi
