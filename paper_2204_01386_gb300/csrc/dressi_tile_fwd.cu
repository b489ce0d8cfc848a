// dressi_tile_fwd.cu -- per-tile kernel, forward.
#include "dressi_tile.cuh"

namespace dressi {
template void launch_tile_mode<0>(const Globals &g, cudaStream_t s);
extern template void launch_tile_mode<1>(const Globals &g, cudaStream_t s);
extern template void launch_tile_mode<2>(const Globals &g, cudaStream_t s);
extern template void launch_tile_mode<4>(const Globals &g, cudaStream_t s);
extern template void launch_tile_mode<5>(const Globals &g, cudaStream_t s);
extern template void launch_tile_mode<6>(const Globals &g, cudaStream_t s);
extern template void launch_tile_mode<8>(const Globals &g, cudaStream_t s);
extern template void launch_tile_mode<9>(const Globals &g, cudaStream_t s);

// 16 px tiles past this number: the adjoint from ids takes CTAs of 128 threads, so that more tiles
// are in flight and hide each other's starts (us by 256 / 128 threads: 8,192 tiles 176 / 147, five
// 801 x 1,140 views with K = 1 305 / 228, 3,456 tiles 78 / 70, 1,024 tiles 29.2 / 28.6); with fewer,
// a tile's own time counts (256 tiles: 19 / 24)
constexpr int MANY_TILES = 608;

void launch_tile(const Globals &g, bool backward, cudaStream_t s)
{
    // the adjoint with the light gradient, the inverse UV or the normal map uses the
    // kernels that have them
    const bool extra = (g.glight != nullptr && g.shade_mode >= 2) || g.texgrad_mode == 2 || g.shade_mode == 3;
    if (!backward) g.shade_mode == 3 ? launch_tile_mode<6>(g, s) : launch_tile_mode<0>(g, s);
    else if (g.ids_in && extra) launch_tile_mode<4>(g, s);
    else if (g.ids_in && g.big_faces) launch_tile_mode<9>(g, s);
    else if (g.ids_in && g.tile == 16 && g.total_tiles > MANY_TILES) launch_tile_mode<8>(g, s);
    else if (g.ids_in) launch_tile_mode<2>(g, s);
    else extra ? launch_tile_mode<5>(g, s) : launch_tile_mode<1>(g, s);
    count_launch(1);
}
}  // namespace dressi
