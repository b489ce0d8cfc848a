// dressi_launch.h -- internal launchers shared by the translation units.
#pragma once
#include <cstddef>
#include <cuda_runtime.h>
#include <utility>

namespace dressi {
struct Globals;
// Kernel launches of this library overlap: a kernel may be set up while the one before it in the
// stream ends (programmatic dependent launch), and waits, before it touches memory, until that one
// is complete and its writes are visible.  Every kernel waits, so that completion is transitive.
// The ten short kernels of a textured 256^2 step idled some 2 us at each: without / with, 113 / 91 us;
// inverse UV on one 521 x 337 view 119 / 101, a 1280 x 720 render 128 / 109, a 64^2 step of 320 faces
// 59 / 43.  (Releasing the next kernel at a kernel's start instead of its end made the textured step 5 us
// faster and the other two 4 and 9 us slower.)
// With clusters of `ctas` blocks (1: none).
template <typename... P, typename... A>
inline void launch_clusters(int ctas, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                            A &&...args)
{
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[2] = {};
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = ctas;
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = ctas > 1 ? 2 : 1;
    cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...);
}

template <typename... P, typename... A>
inline void launch(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A &&...args)
{
    launch_clusters(1, kernel, grid, block, smem, s, std::forward<A>(args)...);
}
#ifdef __CUDACC__
// the kernel's first statement: the grids before it in the stream are complete
__device__ __forceinline__ void grid_wait()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
}
#endif
void count_launch(int n);
// words of view and mesh tables that one launch can carry as a parameter
constexpr int TABLE_WORDS = 4000;
template <int N>
struct Tables {
    int n;
    alignas(8) unsigned w[N ? N : 2];
};
// small arrays of 32-bit words set by the vertex transform for the kernels after it
struct Clears {
    static constexpr int MAX = 6;
    int *p[MAX] = {};
    int n[MAX] = {}, v[MAX] = {};
};
// ranges of 32-bit words filled by one launch
struct Fills {
    static constexpr int MAX = 12;
    unsigned *p[MAX] = {};
    long long n[MAX] = {};
    unsigned v[MAX] = {};
};
// exclusive prefix of n_in non-negative ints at src (0 past them) into n_out at dst
struct ScanJob {
    const int *src;
    int *dst;
    int n_in, n_out;
    int *partial;   // scan_partials_needed(n_out) ints; receives the total behind the parts
};
void launch_vertex(const Globals &g, int n_views, int max_nv, const unsigned *tables, int words, const Clears &clr,
                   cudaStream_t s);
void launch_faces(const Globals &g, int n_views, int n_meshes, int max_nf_view, int max_nf, int max_nv, bool lists,
                  bool normals, cudaStream_t s);
void launch_fill(const Fills &f, cudaStream_t s);
void launch_tile(const Globals &g, bool backward, cudaStream_t s);
void launch_tile_shade(const Globals &g, cudaStream_t s);
void launch_tile_heavy(const Globals &g, cudaStream_t s);
void launch_lpt_order(const Globals &g, cudaStream_t s);
size_t texgather_scratch_bytes(long long slots, long long n_texels, size_t align);
void launch_scans(const ScanJob *jobs, int n, cudaStream_t s);   // one or two, in the same launches
int scan_partials_needed(long long n);
void launch_inv_uv_apply(const Globals &g, long long n_texels, cudaStream_t s);
void launch_tex_gather(const Globals &g, long long slots, long long n_texels, int n_meshes, int max_texels,
                       char *scratch, size_t align, cudaStream_t s);
void launch_vertex_bwd(const Globals &g, int n_views, int max_nv, int n_meshes, int max_nf, bool normals,
                       cudaStream_t s);
void launch_l2(const float *out, const float *tgt, long long n, float *grad, float *loss, cudaStream_t s);
}  // namespace dressi
