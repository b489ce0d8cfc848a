// dressi_setup.cu -- per-vertex and per-face stages: double-float vertex transform,
// vertex normals, tile binning (count / scan / fill) and the per-vertex end of
// the adjoint (screen -> clip -> object space, normals -> positions).
#include "dressi_core.cuh"
#include "dressi_launch.h"

#include <algorithm>
#include <cstring>

namespace dressi {

// ---------------------------------------------------------------------------
// vertex transform (render-graph listing: homogeneous position, MVP, face lookup)
// clip = MVP (p, 1), X = (x/w + 1)/2 W, Y = (y/w + 1)/2 H, depth z/w, evaluated in
// double-float arithmetic (an unevaluated sum hi + lo of two FP32 numbers, ~2^-45
// relative accuracy) built from the error-free transformations two-sum (Knuth) and
// two-product with FMA (as in Ogita, Rump and Oishi, "Accurate sum and dot product",
// 2005).  The screen position comes out as the float pair the records keep; products
// of FP32 inputs are exact, so integer geometry with w = 1 stays exact.  GB300's FP64
// rate is low, FP32 is not.
// ---------------------------------------------------------------------------
struct DF {
    float hi, lo;
};

__device__ __forceinline__ DF two_sum(float a, float b)
{
    const float s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    return {s, e};
}

__device__ __forceinline__ DF quick_two_sum(float a, float b)   // |a| >= |b|
{
    const float s = __fadd_rn(a, b);
    return {s, __fsub_rn(b, __fsub_rn(s, a))};
}

__device__ __forceinline__ DF two_prod(float a, float b)
{
    const float p = __fmul_rn(a, b);
    return {p, __fmaf_rn(a, b, -p)};
}

__device__ __forceinline__ DF df_add(DF x, DF y)
{
    const DF s = two_sum(x.hi, y.hi);
    return quick_two_sum(s.hi, __fadd_rn(s.lo, __fadd_rn(x.lo, y.lo)));
}

__device__ __forceinline__ DF df_mul(DF x, DF y)
{
    const DF p = two_prod(x.hi, y.hi);
    return quick_two_sum(p.hi, __fmaf_rn(x.hi, y.lo, __fmaf_rn(x.lo, y.hi, p.lo)));
}

__device__ __forceinline__ DF df_mul_f(DF x, float b)
{
    const DF p = two_prod(x.hi, b);
    return quick_two_sum(p.hi, __fmaf_rn(x.lo, b, p.lo));
}

// 1 / w: the rounded reciprocal and one Newton correction from the exact residual
__device__ __forceinline__ DF df_recip(DF w)
{
    const float r = __frcp_rn(w.hi);
    const float e = __fmaf_rn(-w.lo, r, __fmaf_rn(-w.hi, r, 1.f));   // 1 - w r (w.hi r exact in the FMA)
    return quick_two_sum(r, __fmul_rn(e, r));
}

// The first kernel of a pass also uploads the tables (they travel as its parameter: no host-to-
// device copy, so a pass can be captured into a CUDA graph) and clears the counters of the
// kernels after it: a launch of its own costs a small call as much as its work (a 320-face,
// 64 x 64 step is all launches).  TABLES: words of tables in the parameter (0: already uploaded).
template <int TABLES>
__global__ void k_vertex(Globals g, const __grid_constant__ Tables<TABLES> tab, Clears clr)
{
    grid_wait();
    const ViewK *views = g.views;
    const MeshK *meshes = g.meshes;
    const int nthreads = gridDim.x * gridDim.y * blockDim.x;
    const int gtid = (blockIdx.y * gridDim.x + blockIdx.x) * blockDim.x + threadIdx.x;
    if (TABLES) {
        unsigned *dst = reinterpret_cast<unsigned *>(const_cast<ViewK *>(g.views));
        for (int i = gtid; i < tab.n; i += nthreads) dst[i] = tab.w[i];
        // this kernel's own reads come from the parameter
        views = reinterpret_cast<const ViewK *>(tab.w);
        meshes = reinterpret_cast<const MeshK *>(tab.w + (reinterpret_cast<const unsigned *>(g.meshes) - dst));
    }
#pragma unroll
    for (int q = 0; q < Clears::MAX; ++q)
        for (int i = gtid; i < clr.n[q]; i += nthreads) clr.p[q][i] = clr.v[q];
    const ViewK &V = views[blockIdx.y];
    const MeshK &M = meshes[V.mesh];
    VRec *out = g.vrec + V.vrec_off;
    const long long nvt = g.n_verts_total;
    bool bad = false;
    // this view's tiles: the tile -> view table, and cleared bin counters when the face table
    // will count into them
    const int nt = V.tiles_x * V.tiles_y;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < nt; i += gridDim.x * blockDim.x) {
        g.tile_view[V.tile_base + i] = blockIdx.y;
        if (g.zero_bins) {
            g.tile_count[V.tile_base + i] = 0;
            g.tile_cursor[V.tile_base + i] = 0;
        }
    }
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < M.nV; i += gridDim.x * blockDim.x) {
        const long long gi = M.vert_off + i;
        const float p0 = __ldg(g.pos + gi), p1 = __ldg(g.pos + nvt + gi), p2 = __ldg(g.pos + 2 * nvt + gi);
        DF c[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const float *m = V.mvp + 4 * r;
            c[r] = df_add(df_add(df_add(two_prod(m[0], p0), two_prod(m[1], p1)), two_prod(m[2], p2)), DF{m[3], 0.f});
        }
        const DF iw = df_recip(c[3]);
        const DF X = df_mul_f(df_add(df_mul(c[0], iw), DF{1.f, 0.f}), 0.5f * (float)V.W);
        const DF Y = df_mul_f(df_add(df_mul(c[1], iw), DF{1.f, 0.f}), 0.5f * (float)V.H);
        const DF Z = df_mul(c[2], iw);
        VRec r;
        r.xh = X.hi;
        r.xl = X.lo;
        r.yh = Y.hi;
        r.yl = Y.lo;
        r.z = Z.hi;
        r.iw = iw.hi;
        const bool fin = isfinite(X.hi) && isfinite(Y.hi) && isfinite(Z.hi) && isfinite(X.lo) && isfinite(Y.lo);
        // the signs of w - 1e-6, Z and 1 - Z from the pairs (hi carries the sign unless it is 0)
        const bool w_pos = c[3].hi > 1e-6f || (c[3].hi == 1e-6f && c[3].lo > 0.f);
        const bool z_ge0 = Z.hi > 0.f || (Z.hi == 0.f && Z.lo >= 0.f);
        const bool z_le1 = Z.hi < 1.f || (Z.hi == 1.f && Z.lo <= 0.f);
        r.valid = w_pos && z_ge0 && z_le1 && fin && fabsf(X.hi) < 1e30f && fabsf(Y.hi) < 1e30f;
        r.pad = 0;
        if (!(isfinite(p0) && isfinite(p1) && isfinite(p2))) bad = true;
        out[i] = r;
    }
    if (bad) atomicOr(g.status, DRESSI_DEV_NONFINITE);
}

// ---------------------------------------------------------------------------
// area-weighted vertex normals (listing BuildNormalCompute): m_v = sum of
// (P1 - P0) x (P2 - P0) over the faces holding v, n_v = m_v / |m_v|.
// The sum runs over a vertex -> face adjacency in increasing face order, so the
// normals (and everything shaded with them) are bitwise reproducible.
// ---------------------------------------------------------------------------
__device__ __forceinline__ bool face_vertices(const Globals &g, const MeshK &M, int f, int v[3])
{
    const int *fv = g.faces + 3 * (M.face_off + f);
    v[0] = __ldg(fv); v[1] = __ldg(fv + 1); v[2] = __ldg(fv + 2);
    return (unsigned)v[0] < (unsigned)M.nV && (unsigned)v[1] < (unsigned)M.nV && (unsigned)v[2] < (unsigned)M.nV;
}

// the vertex -> face adjacency of mesh m: PASS 0 counts, PASS 1 fills.  Runs in the extra grid rows
// (one per mesh) of the face table and list fill kernels, which it does not depend on.
template <int PASS>
__device__ __forceinline__ void adjacency(const Globals &g, int m)
{
    const MeshK &M = g.meshes[m];
    for (int f = blockIdx.x * blockDim.x + threadIdx.x; f < M.nF; f += gridDim.x * blockDim.x) {
        int v[3];
        if (!face_vertices(g, M, f, v)) continue;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const long long gv = M.vert_off + v[j];
            if (PASS == 0) atomicAdd(g.adj_off + gv, 1);
            else g.adj[g.adj_off[gv] + atomicAdd(g.adj_cur + gv, 1)] = f;
        }
    }
}

template <int PASS>
__global__ void k_adjacency(Globals g)
{
    grid_wait();
    adjacency<PASS>(g, blockIdx.y);
}

__global__ void k_normal_csr(Globals g)
{
    grid_wait();
    const MeshK &M = g.meshes[blockIdx.y];
    const long long nvt = g.n_verts_total;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < M.nV; i += gridDim.x * blockDim.x) {
        const long long gv = M.vert_off + i;
        const int b = g.adj_off[gv], e = g.adj_off[gv + 1];
        float m0 = 0.f, m1 = 0.f, m2 = 0.f;
        // incident faces in increasing id order (the lists are short: pick the next
        // larger id each round)
        int last = -1;
        for (int round = b; round < e; ++round) {
            int f = 0x7fffffff;
            for (int q = b; q < e; ++q) {
                const int c = g.adj[q];
                if (c > last && c < f) f = c;
            }
            if (f == 0x7fffffff) break;
            last = f;
            int v[3];
            face_vertices(g, M, f, v);
            float P[3][3];
#pragma unroll
            for (int j = 0; j < 3; ++j)
#pragma unroll
                for (int c = 0; c < 3; ++c) P[j][c] = __ldg(g.pos + c * nvt + M.vert_off + v[j]);
            const float u[3] = {P[1][0] - P[0][0], P[1][1] - P[0][1], P[1][2] - P[0][2]};
            const float w[3] = {P[2][0] - P[0][0], P[2][1] - P[0][1], P[2][2] - P[0][2]};
            m0 += u[1] * w[2] - u[2] * w[1];
            m1 += u[2] * w[0] - u[0] * w[2];
            m2 += u[0] * w[1] - u[1] * w[0];
        }
        const float l = sqrtf(m0 * m0 + m1 * m1 + m2 * m2);
        const float s = l > 0.f ? 1.f / l : 0.f;
        g.nrm[gv] = make_float4(m0 * s, m1 * s, m2 * s, l);
    }
}

// ---------------------------------------------------------------------------
// tile binning: every live face goes into the list of each tile that its
// bounding box, grown by bin_R pixels (r plus the edge-mask halo plus a guard),
// touches.  The face table kernel counts, k_bin fills.  Order inside a list is
// irrelevant: the peel keeps the K smallest (key, id) pairs.
// ---------------------------------------------------------------------------
// the tiles [tx0, tx1] x [ty0, ty1] that the grown box of the face's screen corners
// touches; false when it misses the view
__device__ __forceinline__ bool bin_rect(const Globals &g, const ViewK &V, const FaceGeo &R, int &tx0, int &tx1,
                                         int &ty0, int &ty1)
{
    const float Tinv = 1.f / (float)g.tile;
    const float x0 = fminf(R.c[0].xh, fminf(R.c[1].xh, R.c[2].xh)) - V.bin_R;
    const float x1 = fmaxf(R.c[0].xh, fmaxf(R.c[1].xh, R.c[2].xh)) + V.bin_R;
    const float y0 = fminf(R.c[0].yh, fminf(R.c[1].yh, R.c[2].yh)) - V.bin_R;
    const float y1 = fmaxf(R.c[0].yh, fmaxf(R.c[1].yh, R.c[2].yh)) + V.bin_R;
    if (x1 < 0.f || y1 < 0.f || x0 > (float)V.W || y0 > (float)V.H) return false;
    tx0 = max(0, (int)floorf(x0 * Tinv));
    tx1 = min(V.tiles_x - 1, (int)floorf(x1 * Tinv));
    ty0 = max(0, (int)floorf(y0 * Tinv));
    ty1 = min(V.tiles_y - 1, (int)floorf(y1 * Tinv));
    return tx0 <= tx1 && ty0 <= ty1;
}

// A face's tile rect [tx0, tx1] x [ty0, ty1], packed into one word for the list fill:
// tx0 | ty0 << 11 | (tx1 - tx0) << 22 | (ty1 - ty0) << 27.  Tile coordinates are below
// 2048 (views of at most 32,768 pixels at 16 px tiles); a rect more than 32 tiles wide or
// high is BRECT_WIDE, and the list fill takes it from the face record.  Neither marker
// is a valid packing (both would put tx0 + (tx1 - tx0) past 2047).
constexpr unsigned BRECT_NONE = 0xffffffffu;   // no tile: culled, or off the view
constexpr unsigned BRECT_WIDE = 0xfffffffeu;

__device__ __forceinline__ unsigned pack_brect(bool any, int tx0, int tx1, int ty0, int ty1)
{
    if (!any) return BRECT_NONE;
    if (tx1 - tx0 > 31 || ty1 - ty0 > 31) return BRECT_WIDE;
    return (unsigned)tx0 | ((unsigned)ty0 << 11) | ((unsigned)(tx1 - tx0) << 22) | ((unsigned)(ty1 - ty0) << 27);
}

// the (face, tile) pairs of a warp's faces, one step per tile of each lane's box: the
// lanes at the same tile in a step share one atomic (consecutive faces of a mesh are
// mostly neighbours), and PASS 1 gives them consecutive list slots.  All 32 lanes call it.
template <int PASS>
__device__ __forceinline__ void bin_walk(const Globals &g, const ViewK &V, int f, bool any, int tx0, int tx1,
                                         int ty0, int ty1)
{
    const int lane = threadIdx.x & 31;
    int tx = tx0, ty = ty0;
    bool more = any;
    while (__any_sync(0xffffffffu, more)) {
        const int t = more ? V.tile_base + ty * V.tiles_x + tx : -1;
        const unsigned grp = __match_any_sync(0xffffffffu, t);
        if (more) {
            const int leader = __ffs(grp) - 1;
            if (PASS == 0) {
                if (lane == leader) atomicAdd(g.tile_count + t, __popc(grp));
            } else {
                // the list's start loads under the reservation.  (Read after it, as the compiler has to where
                // the kernel writes other integers too, k_bin took 14.4 instead of 13.3 us for 15,000 faces
                // at 1024^2 and 1278 instead of 1211 us for two faces over 4,096 tiles.)
                const int off = __ldg(g.tile_off + t);
                int base = 0;
                if (lane == leader) base = atomicAdd(g.tile_cursor + t, __popc(grp));
                base = __shfl_sync(grp, base, leader) + __popc(grp & ((1u << lane) - 1u));
                const long long idx = (long long)off + base;
                if (idx < g.list_cap) g.lists[idx] = f;
            }
            if (++tx > tx1) {
                tx = tx0;
                if (++ty > ty1) more = false;
            }
        }
    }
}

// ---------------------------------------------------------------------------
// front words: the front hard (key, id) of every pixel, by 64-bit atomicMin in the order of the
// faces, for passes that need more layers only inside the edge mask.  A small face covers a few
// pixels; visiting them from the face (a dozen pixel tests, the record at hand) replaces its
// staging, bounding boxes and shared-memory lists in each of the tiles that its grown box touches
// (measured on both sides of the line that chooses it: FRONT_MIN_FACES, dressi_api.cu).  A lane
// visits a face's rows, cut to the covered interval: two 2048^2 views of 1.31 M faces 165 us with
// the table, which alone takes 106; a warp-wide list of all box pixels took 198, and on 21-pixel
// faces 84 instead of 44 us (its batches look up face, record and pixel for each pair).  Larger faces
// are k_front_big's.
// ---------------------------------------------------------------------------
// Pixels of a bounding box that its face's lane visits alone; past them it is left to k_front_big, whose
// warps share such faces out over the GPU.  A few hundred mid-sized faces among many small ones follow
// one another in the mesh: while up to 4,096 pixels went through a list of their own warp's pixels, ten
// warps had 300 of them.  Forward, us, with such lists / 96 / 128 / 192 / 256, without front words:
//   81,920 small faces, 1280 x 720                102 / 101 / 101 / 100 / 100, 175
//   ... and 300 of some 1,500 px                  436 / 125 / 127 / 136 / 144, 200
//   ... and 3,000 of some 700 px                  286 / 157 / 150 / 157 / 168, 212
//   ... and 2,000 of some 3,000 px                644 / 252 / 250 / 250 / 252, 321
//   the small ones from close by, 1024^2          159 / 152 / 129 / 116 / 116, 197
//   step of four 768^2 views of 32,000 faces      512 / 520 / 513 / 511 / 510, 874
constexpr int FRONT_LANE = 192;

// the pixel centres inside the face's bounding box (grown by a margin over the corners' low parts)
__device__ __forceinline__ bool front_rect(const ViewK &V, const FaceGeo &R, int &x0, int &y0, int &w, int &h)
{
    const float M = 0.01f;
    x0 = max(0, (int)ceilf(fminf(R.c[0].xh, fminf(R.c[1].xh, R.c[2].xh)) - 0.5f - M));
    y0 = max(0, (int)ceilf(fminf(R.c[0].yh, fminf(R.c[1].yh, R.c[2].yh)) - 0.5f - M));
    w = min(V.W - 1, (int)floorf(fmaxf(R.c[0].xh, fmaxf(R.c[1].xh, R.c[2].xh)) - 0.5f + M)) - x0 + 1;
    h = min(V.H - 1, (int)floorf(fmaxf(R.c[0].yh, fmaxf(R.c[1].yh, R.c[2].yh)) - 0.5f + M)) - y0 + 1;
    return w > 0 && h > 0;
}

__device__ __forceinline__ void front_pixel(const ViewK &V, const FaceGeo &R, int f, int x, int y, unsigned long long *words)
{
    Frag fr;
    if (eval_face<false>(R, (float)x + 0.5f, (float)y + 0.5f, 0.f, V.half_inv_S, fr, true)) {
        // a key of 1/2 or more (the far plane; the noise of a sliver's depth) is stored as 1/2: the pixel is
        // covered (word_hard) and its tile decided from all layers (word_tie), whatever the value
        const unsigned long long v = pack_frag(fr.key, f), tie = pack_frag(0.5f, f);
        atomicMin(words + (long long)y * V.W + x, v < tie ? v : tie);
    }
}

// a face's pixels by its own lane: each row of the box cut to where the three cross products, linear
// along the row, are above -FRONT_SLACK px (a division-free half-plane per edge), and the pixels
// left tested exactly.  Where the crosses' rounding could reach the slack (corners far outside
// the box, or an edge far shorter than the face), the whole rows are tested.  With u = 2^-24 and no corner
// farther than e from a pixel of the box along either axis, eval_face's cross is within 11 u e^2 of the exact
// one (differences good to 2 u, two products, a sum), the row start's within 12 u e^2, the slope times a
// column within 6 u e^2, and the bound's division moves it by up to 14 u e^2: together 43 u e^2 or
// 2.6e-6 e^2 / (the edge's length) px.  (10 million accepted pixels of needles, slivers and cut faces,
// emulated in FP32 with the limit ten times as far: none came closer than 0.91 slacks to being cut.)
constexpr float FRONT_SLACK = 2e-3f, FRONT_CUT_ERR = 3e-6f;

__device__ __forceinline__ void front_lane(const ViewK &V, const FaceGeo &R, int f, int x0, int y0, int w, int h,
                                           unsigned long long *words)
{
    float dx[3], slope[3], inv[3], eps[3], sgn[3];
    float ext = 0.f, sharp = 0.f;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        dx[i] = ((float)x0 + 0.5f - R.c[i].xh) - R.c[i].xl;
        const float ddy = (float)y0 + 0.5f - R.c[i].yh;
        ext = fmaxf(ext, fmaxf(fmaxf(fabsf(dx[i]), fabsf(dx[i] + (float)(w - 1))), fmaxf(fabsf(ddy), fabsf(ddy + (float)(h - 1)))));
        sharp = fmaxf(sharp, fabsf(R.invL[i]));
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const int P = i == 2 ? 0 : i, Q = i == 2 ? 2 : i + 1;
        sgn[i] = R.invL[i] > 0.f ? 1.f : -1.f;
        // d cross / d x = dy_Q - dy_P; a level edge keeps or drops a whole row
        const float sl = sgn[i] * ((R.c[P].yh - R.c[Q].yh) + (R.c[P].yl - R.c[Q].yl));
        slope[i] = fabsf(sl) < 1e-9f ? 1e-9f : sl;
        inv[i] = __fdividef(1.f, slope[i]);
        eps[i] = __fdividef(FRONT_SLACK, fabsf(R.invL[i]));
    }
    const bool cut = FRONT_CUT_ERR * ext * ext * sharp <= FRONT_SLACK;
    for (int y = y0; y < y0 + h; ++y) {
        float lo = 0.f, hi = (float)(w - 1);
        if (cut) {
            float dy[3];
#pragma unroll
            for (int i = 0; i < 3; ++i) dy[i] = ((float)y + 0.5f - R.c[i].yh) - R.c[i].yl;
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                const int P = i == 2 ? 0 : i, Q = i == 2 ? 2 : i + 1;
                const float c = sgn[i] * (dx[P] * dy[Q] - dy[P] * dx[Q]);
                const float t = -(c + eps[i]) * inv[i];
                if (slope[i] > 0.f) lo = fmaxf(lo, t);
                else hi = fminf(hi, t);
            }
        }
        if (!(lo <= hi)) continue;
        const int k1 = (int)floorf(hi);
        for (int k = (int)ceilf(lo); k <= k1; ++k) front_pixel(V, R, f, x0 + k, y, words);
    }
}

// a band of the rows of a face's box, by a warp
__device__ __forceinline__ void front_band(const Globals &g, const ViewK &V, const FaceGeo &R, int f, int band, int bands)
{
    const int lane = threadIdx.x & 31;
    int x0, y0, w, h;
    if (!front_rect(V, R, x0, y0, w, h)) return;
    const int r0 = (int)((long long)h * band / bands), r1 = (int)((long long)h * (band + 1) / bands);
    for (int y = y0 + r0; y < y0 + r1; ++y)
        for (int x = x0 + lane; x < x0 + w; x += 32) front_pixel(V, R, f, x, y, g.kth + V.slot_base);
}

// the faces with larger boxes, from the list that k_face left: a warp takes a band of a face's rows.  Where
// the list had no room for all (a capacity of the tile lists far too small for the scene), they are
// looked for in the whole table instead, a warp taking a band of those among 32 faces: four faces that
// fill 1280 x 720 among 81,920 small ones, capacity 2: forward 74 ms while their own lanes visited
// them, 10.6 now, 11.5 without front words (all tiles take all faces).
__global__ void __launch_bounds__(256) k_front_big(Globals g)
{
    grid_wait();
    const int n = *g.big_n;
    if (n == 0) return;
    const int warps = gridDim.x * (blockDim.x >> 5), lane = threadIdx.x & 31;
    const int warp = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (n <= g.big_cap) {
        const int bands = max(1, min(64, warps / n));
        for (long long it = warp; it < (long long)n * bands; it += warps) {
            const int2 e = g.big[it / bands];
            const ViewK &V = g.views[e.x];
            front_band(g, V, g.frec[V.frec_off + e.y], e.y, (int)(it % bands), bands);
        }
        return;
    }
    for (int v = 0; v < g.n_views; ++v) {
        const ViewK &V = g.views[v];
        const int nF = g.meshes[V.mesh].nF, groups = (nF + 31) / 32;
        const int bands = max(1, min(64, warps / max(groups, 1)));
        // (each view's first group at another warp)
        for (long long it = (warp + v * 97ll) % warps; it < (long long)groups * bands; it += warps) {
            const int f0 = (int)(it / bands) * 32;
            bool big = false;
            if (f0 + lane < nF) {
                const FaceGeo &R = g.frec[V.frec_off + f0 + lane];
                int x0, y0, w, h;
                big = (R.flags & FLAG_LIVE) && front_rect(V, R, x0, y0, w, h) && (long long)w * h > FRONT_LANE;
            }
            for (unsigned todo = __ballot_sync(0xffffffffu, big); todo; todo &= todo - 1u) {
                const int f = f0 + __ffs(todo) - 1;
                front_band(g, V, g.frec[V.frec_off + f], f, (int)(it % bands), bands);
            }
        }
    }
}

// ---------------------------------------------------------------------------
// face table: the record of every (view, face) -- screen corners, canonical edges,
// lengths, area, flags -- built once per call and read by binning, staging,
// shading and the adjoint (112 bytes each).  COUNT: also the tile counts of the
// binning (the lists' lengths).
// ---------------------------------------------------------------------------
// FRONT: also the front words of the faces' pixels.
template <bool COUNT, bool FRONT>
__global__ void __launch_bounds__(256, FRONT ? 3 : 4) k_face(Globals g)
{
    grid_wait();
    // each warp's 32 records (7 float4 each) go through shared memory so that the warp
    // writes its 3,584 contiguous bytes with full-line stores
    __shared__ float4 stage[256 / 32][32 * 7];
    if (blockIdx.y >= g.n_views) {
        adjacency<0>(g, blockIdx.y - g.n_views);
        return;
    }
    const ViewK V = g.views[blockIdx.y];   // copies: the fields stay in registers across the stores
    const MeshK M = g.meshes[V.mesh];
    const VRec *vr = g.vrec + V.vrec_off;
    const int lane = threadIdx.x & 31;
    float4 *ws = stage[threadIdx.x >> 5];
    bool bad = false;
    // block-uniform trip count: every lane of a warp takes part in the binning steps
    for (int f0 = blockIdx.x * blockDim.x; f0 < M.nF; f0 += gridDim.x * blockDim.x) {
        const int f = f0 + threadIdx.x;
        bool live = false;
        FaceRec R;
        if (f < M.nF) {
            face_load(g, M, vr, f, R);
            if (R.flags & FLAG_RANGE) {
                // out of range: nothing else of the record is meaningful
                bad = true;
#pragma unroll
                for (int i = 0; i < 3; ++i) { R.vi[i] = 0; R.c[i].xh = R.c[i].xl = R.c[i].yh = R.c[i].yl = 0.f; }
            }
            live = (R.flags & FLAG_LIVE) != 0;
            float4 *d = ws + lane * 7;   // 112-byte lane stride: no bank conflict within 8 lanes
#pragma unroll
            for (int i = 0; i < 3; ++i) d[i] = make_float4(R.c[i].xh, R.c[i].xl, R.c[i].yh, R.c[i].yl);
            d[3] = make_float4(R.invL[0], R.invL[1], R.invL[2], R.z[0]);
            d[4] = make_float4(R.z[1], R.z[2], R.invA, __int_as_float(R.flags));
            d[5] = make_float4(__int_as_float(R.id), __int_as_float(R.vi[0]), __int_as_float(R.vi[1]),
                               __int_as_float(R.vi[2]));
            d[6] = make_float4(R.iw[0], R.iw[1], R.iw[2], 0.f);
        }
        __syncwarp();
        {
            const int wf0 = f0 + (threadIdx.x & ~31);   // the warp's first face
            const int nrec = max(0, min(32, M.nF - wf0));
            float4 *dst = reinterpret_cast<float4 *>(g.frec + V.frec_off + wf0);
            for (int i = lane; i < nrec * 7; i += 32) dst[i] = ws[i];
        }
        int x0, y0, w, h;
        if (FRONT && live && front_rect(V, R, x0, y0, w, h)) {
            if ((long long)w * h <= FRONT_LANE) {
                front_lane(V, R, f, x0, y0, w, h, g.kth + V.slot_base);
            } else {
                const int q = atomicAdd(g.big_n, 1);
                if (q < g.big_cap) g.big[q] = make_int2(blockIdx.y, f);   // else: see k_front_big
            }
        }
        __syncwarp();   // the staged records are read before the next iteration writes them
        if (COUNT) {
            int tx0 = 0, tx1 = -1, ty0 = 0, ty1 = -1;
            const bool any = live && bin_rect(g, V, R, tx0, tx1, ty0, ty1);
            if (f < M.nF) g.brect[V.frec_off + f] = pack_brect(any, tx0, tx1, ty0, ty1);
            bin_walk<0>(g, V, f, any, tx0, tx1, ty0, ty1);
        }
    }
    if (bad) atomicOr(g.status, DRESSI_DEV_FACE_RANGE);
}

// the list entries of every (face, tile) pair, into the slots the counts' prefix gives;
// each face's tile rect comes packed from the face table kernel
__global__ void k_bin(Globals g)
{
    grid_wait();
    if (blockIdx.y >= g.n_views) {
        adjacency<1>(g, blockIdx.y - g.n_views);
        return;
    }
    if (g.heavy) {
        const int nthreads = gridDim.x * g.n_views * blockDim.x;
        for (int t = (blockIdx.y * gridDim.x + blockIdx.x) * blockDim.x + threadIdx.x; t < g.total_tiles; t += nthreads)
            if (long_list(g, t)) {
                const int q = atomicAdd(g.heavy, 1);
                if (q < g.heavy_cap) g.heavy[1 + q] = t;
            }
    }
    const ViewK V = g.views[blockIdx.y];   // copies: the fields stay in registers across the stores
    const MeshK M = g.meshes[V.mesh];
    for (int f0 = blockIdx.x * blockDim.x; f0 < M.nF; f0 += gridDim.x * blockDim.x) {
        const int f = f0 + threadIdx.x;
        int tx0 = 0, tx1 = -1, ty0 = 0, ty1 = -1;
        const unsigned b = f < M.nF ? __ldg(g.brect + V.frec_off + f) : BRECT_NONE;
        bool any = false;
        if (b == BRECT_WIDE) {
            FaceRec R;
            any = face_get(g, V, M, f, R) && bin_rect(g, V, R, tx0, tx1, ty0, ty1);
        } else if (b != BRECT_NONE) {
            tx0 = b & 2047;
            ty0 = (b >> 11) & 2047;
            tx1 = tx0 + ((b >> 22) & 31);
            ty1 = ty0 + (b >> 27);
            any = true;
        }
        bin_walk<1>(g, V, f, any, tx0, tx1, ty0, ty1);
    }
}

// ---------------------------------------------------------------------------
// longest-first tile order for the persistent tile kernel: a counting sort of the
// tiles by descending face-list length (lengths bucketed, ties in any order)
// ---------------------------------------------------------------------------
__device__ __forceinline__ int lpt_bin(int count) { return LPT_BINS - 1 - min(count, LPT_BINS - 1); }

__global__ void k_lpt_hist(Globals g)
{
    grid_wait();
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < g.total_tiles; t += gridDim.x * blockDim.x)
        atomicAdd(g.lpt_hist + lpt_bin(g.tile_count[t]), 1);
}

__global__ void __launch_bounds__(LPT_BINS) k_lpt_scan(Globals g)
{
    grid_wait();
    __shared__ int warp_sums[LPT_BINS / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int v = g.lpt_hist[tid];
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) warp_sums[warp] = x;
    __syncthreads();
    if (warp == 0) {
        int w = warp_sums[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += y;
        }
        warp_sums[lane] = w;
    }
    __syncthreads();
    g.lpt_hist[tid] = x - v + (warp > 0 ? warp_sums[warp - 1] : 0);   // exclusive offsets
}

__global__ void k_lpt_scatter(Globals g)
{
    grid_wait();
    int *order = const_cast<int *>(g.tile_order);
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < g.total_tiles; t += gridDim.x * blockDim.x)
        order[atomicAdd(g.lpt_hist + lpt_bin(g.tile_count[t]), 1)] = t;
}

// the same order in one block (a launch instead of three): the histogram in shared memory
__global__ void __launch_bounds__(LPT_BINS) k_lpt_single(Globals g)
{
    grid_wait();
    __shared__ int hist[LPT_BINS];
    __shared__ int warp_sums[LPT_BINS / 32];
    int *order = const_cast<int *>(g.tile_order);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    hist[tid] = 0;
    __syncthreads();
    for (int t = tid; t < g.total_tiles; t += LPT_BINS) atomicAdd(hist + lpt_bin(g.tile_count[t]), 1);
    __syncthreads();
    const int v = hist[tid];
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) warp_sums[warp] = x;
    __syncthreads();
    int before = 0;
    for (int w = 0; w < warp; ++w) before += warp_sums[w];
    hist[tid] = before + x - v;
    __syncthreads();
    for (int t = tid; t < g.total_tiles; t += LPT_BINS) order[atomicAdd(hist + lpt_bin(g.tile_count[t]), 1)] = t;
}

// ---------------------------------------------------------------------------
// adjoint, per (view, vertex): (dX, dY, d(1/w)) -> clip -> object space
// ---------------------------------------------------------------------------
__device__ __forceinline__ void normal_bwd(const Globals &g, int m);

// dL/dcolour from its float4 accumulator (ngrad) to the planes
__device__ __forceinline__ void color_bwd(const Globals &g)
{
    const long long nvt = g.n_verts_total;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < nvt; i += (long long)gridDim.x * blockDim.x) {
        const float4 c = g.ngrad[i];
        g.gcol[i] = c.x;
        g.gcol[nvt + i] = c.y;
        g.gcol[2 * nvt + i] = c.z;
    }
}

// grid rows: one per view, then (normals) one per mesh for the normals' share of the positions, or
// (vertex colours) one for their planes
__global__ void k_vertex_bwd(Globals g)
{
    grid_wait();
    if (blockIdx.y >= g.n_views) {
        if (g.gcol) color_bwd(g);
        else normal_bwd(g, blockIdx.y - g.n_views);
        return;
    }
    const ViewK &V = g.views[blockIdx.y];
    const MeshK &M = g.meshes[V.mesh];
    const float4 *sg = g.sgrad + V.vrec_off;
    const long long nvt = g.n_verts_total;
    // dL/dMVP of this view: dL/dclip_r (p, 1)_c for the x, y and w rows (depth only
    // orders the layers and has no gradient)
    float am[12];
#pragma unroll
    for (int q = 0; q < 12; ++q) am[q] = 0.f;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < M.nV; i += gridDim.x * blockDim.x) {
        float4 s = sg[i];
        if (s.x == 0.f && s.y == 0.f && s.z == 0.f) continue;
        const long long gi = M.vert_off + i;
        const float p[3] = {__ldg(g.pos + gi), __ldg(g.pos + nvt + gi), __ldg(g.pos + 2 * nvt + gi)};
        float c[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const float *m = V.mvp + 4 * r;
            c[r] = m[0] * p[0] + m[1] * p[1] + m[2] * p[2] + m[3];
        }
        const float iw = 1.f / c[3];
        const float hx = 0.5f * (float)V.W * iw, hy = 0.5f * (float)V.H * iw;
        const float gcx = s.x * hx, gcy = s.y * hy;
        const float gcw = -(s.x * hx * c[0] + s.y * hy * c[1]) * iw - s.z * iw * iw;
#pragma unroll
        for (int col = 0; col < 3; ++col) {
            float gp = V.mvp[col] * gcx + V.mvp[4 + col] * gcy + V.mvp[12 + col] * gcw;
            atomicAdd(g.gpos + col * nvt + gi, gp);
        }
        if (g.gmvp) {
            const float ph[4] = {p[0], p[1], p[2], 1.f};
#pragma unroll
            for (int col = 0; col < 4; ++col) {
                am[col] = fmaf(gcx, ph[col], am[col]);
                am[4 + col] = fmaf(gcy, ph[col], am[4 + col]);
                am[8 + col] = fmaf(gcw, ph[col], am[8 + col]);
            }
        }
    }
    if (g.gmvp) {
        float *out = g.gmvp + 16 * (long long)blockIdx.y;
#pragma unroll
        for (int q = 0; q < 12; ++q) {
            float v = am[q];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if ((threadIdx.x & 31) == 0 && v != 0.f) atomicAdd(out + (q < 8 ? q : q + 4), v);
        }
    }
}

// normals -> positions: dm_v = (dn_v - n_v (n_v . dn_v)) / |m_v|; per face
// da = sum of dm over its corners; a = u x w gives du = w x da, dw = da x u
__device__ __forceinline__ void normal_bwd(const Globals &g, int m)
{
    const MeshK &M = g.meshes[m];
    const long long nvt = g.n_verts_total;
    for (int f = blockIdx.x * blockDim.x + threadIdx.x; f < M.nF; f += gridDim.x * blockDim.x) {
        const int *fv = g.faces + 3 * (M.face_off + f);
        int v[3] = {__ldg(fv), __ldg(fv + 1), __ldg(fv + 2)};
        if ((unsigned)v[0] >= (unsigned)M.nV || (unsigned)v[1] >= (unsigned)M.nV || (unsigned)v[2] >= (unsigned)M.nV)
            continue;
        float ga[3] = {0.f, 0.f, 0.f};
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const long long gi = M.vert_off + v[j];
            float4 n = g.nrm[gi];
            float4 dn = g.ngrad[gi];
            if (!(n.w > 0.f)) continue;
            float nd = n.x * dn.x + n.y * dn.y + n.z * dn.z;
            float il = 1.f / n.w;
            ga[0] += (dn.x - n.x * nd) * il;
            ga[1] += (dn.y - n.y * nd) * il;
            ga[2] += (dn.z - n.z * nd) * il;
        }
        if (ga[0] == 0.f && ga[1] == 0.f && ga[2] == 0.f) continue;
        float P[3][3];
#pragma unroll
        for (int j = 0; j < 3; ++j)
#pragma unroll
            for (int c = 0; c < 3; ++c) P[j][c] = __ldg(g.pos + c * nvt + M.vert_off + v[j]);
        float u[3] = {P[1][0] - P[0][0], P[1][1] - P[0][1], P[1][2] - P[0][2]};
        float w[3] = {P[2][0] - P[0][0], P[2][1] - P[0][1], P[2][2] - P[0][2]};
        float gu[3] = {w[1] * ga[2] - w[2] * ga[1], w[2] * ga[0] - w[0] * ga[2], w[0] * ga[1] - w[1] * ga[0]};
        float gw[3] = {ga[1] * u[2] - ga[2] * u[1], ga[2] * u[0] - ga[0] * u[2], ga[0] * u[1] - ga[1] * u[0]};
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            atomicAdd(g.gpos + c * nvt + M.vert_off + v[1], gu[c]);
            atomicAdd(g.gpos + c * nvt + M.vert_off + v[2], gw[c]);
            atomicAdd(g.gpos + c * nvt + M.vert_off + v[0], -(gu[c] + gw[c]));
        }
    }
}

__global__ void k_normal_bwd(Globals g) { grid_wait(); normal_bwd(g, blockIdx.y); }
__global__ void k_color_bwd(Globals g) { grid_wait(); color_bwd(g); }

// fills up to Fills::MAX ranges of 32-bit words in one launch (the adjoint's outputs and accumulators)
__global__ void __launch_bounds__(256) k_fill(Fills f)
{
    grid_wait();
    const long long t0 = blockIdx.x * (long long)blockDim.x + threadIdx.x, stride = (long long)gridDim.x * blockDim.x;
#pragma unroll
    for (int q = 0; q < Fills::MAX; ++q) {
        const unsigned v = f.v[q];
        unsigned *p = f.p[q];
        const long long n = f.n[q];
        long long done = 0;
        if ((reinterpret_cast<uintptr_t>(p) & 15) == 0) {
            const long long n4 = n >> 2;
            for (long long i = t0; i < n4; i += stride) reinterpret_cast<uint4 *>(p)[i] = make_uint4(v, v, v, v);
            done = n4 << 2;
        }
        for (long long i = done + t0; i < n; i += stride) p[i] = v;
    }
}

// L2 loss helper
__global__ void k_l2(const float *out, const float *tgt, long long n, float *grad, float *loss)
{
    grid_wait();
    float acc = 0.f;
    const long long i0 = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    const long long stride = (long long)gridDim.x * blockDim.x;
    long long done = 0;
    if (((reinterpret_cast<uintptr_t>(out) | reinterpret_cast<uintptr_t>(tgt) | reinterpret_cast<uintptr_t>(grad)) &
         15) == 0) {
        // 16-byte accesses over the whole float4s, then the scalar tail
        const long long n4 = n >> 2;
        const float4 *o4 = reinterpret_cast<const float4 *>(out), *t4 = reinterpret_cast<const float4 *>(tgt);
        float4 *g4 = reinterpret_cast<float4 *>(grad);
        for (long long i = i0; i < n4; i += stride) {
            const float4 a = __ldg(o4 + i), b = __ldg(t4 + i);
            const float dx = a.x - b.x, dy = a.y - b.y, dz = a.z - b.z, dw = a.w - b.w;
            g4[i] = make_float4(2.f * dx, 2.f * dy, 2.f * dz, 2.f * dw);
            acc += dx * dx + dy * dy + dz * dz + dw * dw;
        }
        done = n4 << 2;
    }
    for (long long i = done + i0; i < n; i += stride) {
        const float d = out[i] - tgt[i];
        grad[i] = 2.f * d;
        acc += d * d;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0 && loss) atomicAdd(loss, acc);
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
static int grid_x(long long n, int block, int cap)
{
    long long b = (n + block - 1) / block;
    if (b < 1) b = 1;
    if (b > cap) b = cap;
    return (int)b;
}

constexpr int MAX_GRID_Y = 65535;

constexpr long long GRID_BLOCKS = 8192;

// blocks along x for `rows` grid rows whose longest takes n: the rows of a ragged batch are mostly far
// shorter, and past some thousands of blocks those without work cost more than a second round of
// the others (32 meshes of 1,000 to 200,000 faces, us without / at 8,192 / at 4,096 blocks: face table
// 85 / 53 / 60, list fill 52 / 32 / 38, end of the adjoint 60 / 35 / 50).  But a thread of the longest row
// takes eight items at most: one long row among many short ones would keep a few blocks busy alone
// (63 meshes of 320 faces and one of 1.31 M, at most 80 / 16 / 8 / 4 items: face table 427 / 157 / 141 / 141,
// list fill 398 / 195 / 183 / 183, end of the adjoint 405 / 203 / 141 / 141; 255 and one of 327,680: face table
// 151 / 105 / 108 / 171).
constexpr int GRID_ITEMS = 8;

static int grid_rows(long long n, int block, int cap, int rows)
{
    int x = grid_x(n, block, cap);
    const long long least = std::max<long long>(64, n / ((long long)block * GRID_ITEMS));
    while (x > least && (long long)x * rows > GRID_BLOCKS) x = (x + 1) / 2;
    return x;
}

template <int TABLES>
static void launch_vertex_t(const Globals &g, dim3 grid, const unsigned *tables, int words, const Clears &clr,
                            cudaStream_t s)
{
    Tables<TABLES> t;
    t.n = words;
    if (TABLES) std::memcpy(t.w, tables, sizeof(unsigned) * words);
    launch(k_vertex<TABLES>, grid, 256, 0, s, g, t, clr);
    count_launch(1);
}

// the vertex transform; uploads the tables (words of them at tables) unless they are already there
// (words 0), from a parameter as small as they allow: the launch copies all of it
void launch_vertex(const Globals &g, int n_views, int max_nv, const unsigned *tables, int words, const Clears &clr,
                   cudaStream_t s)
{
    dim3 grid(grid_rows(max_nv, 256, 1024, n_views), n_views);
    if (words == 0) launch_vertex_t<0>(g, grid, tables, words, clr, s);
    else if (words <= 128) launch_vertex_t<128>(g, grid, tables, words, clr, s);
    else launch_vertex_t<TABLE_WORDS>(g, grid, tables, words, clr, s);
}

// The per-face setup after the vertex transform: face table; with lists, the tile counts, their
// prefix and the lists; with normals, the vertex -> face adjacency (counted beside the face
// table, filled beside the lists) and the normals.  adj_off and adj_cur are cleared.
void launch_faces(const Globals &g, int n_views, int n_meshes, int max_nf_view, int max_nf, int max_nv, bool lists,
                  bool normals, cudaStream_t s)
{
    // (a launch holds 65,535 grid rows; views and meshes may be more together)
    const bool merge = normals && n_views + n_meshes <= MAX_GRID_Y;
    const int rows = n_views + (merge ? n_meshes : 0);
    const dim3 grid(grid_rows(std::max(max_nf_view, merge ? max_nf : 0), 256, 2048, rows), rows);
    const dim3 grid_m(grid_x(max_nf, 256, 2048), n_meshes);
    if (lists && g.fronts == 2) launch(k_face<true, true>, grid, 256, 0, s, g);
    else if (lists) launch(k_face<true, false>, grid, 256, 0, s, g);
    else launch(k_face<false, false>, grid, 256, 0, s, g);
    count_launch(1);
    if (lists && g.fronts == 2) {
        launch(k_front_big, 152 * 4, 256, 0, s, g);   // before the tile lists are written
        count_launch(1);
    }
    if (normals && !merge) {
        launch(k_adjacency<0>, grid_m, 256, 0, s, g);
        count_launch(1);
    }
    // exclusive prefixes: tile_off[n] = total list entries
    ScanJob jobs[2];
    int nj = 0;
    if (lists) jobs[nj++] = {g.tile_count, g.tile_off, g.total_tiles, g.total_tiles + 1, g.scan_partial};
    if (normals) {
        const int n = (int)(g.n_verts_total + 1);
        jobs[nj++] = {g.adj_off, g.adj_off, n, n, g.scan_partial2};
    }
    if (nj) launch_scans(jobs, nj, s);
    if (lists) {
        launch(k_bin, grid, 256, 0, s, g);
        count_launch(1);
    }
    if (normals && !(lists && merge)) {
        launch(k_adjacency<1>, grid_m, 256, 0, s, g);
        count_launch(1);
    }
    if (normals) {
        launch(k_normal_csr, dim3(grid_rows(max_nv, 256, 2048, n_meshes), n_meshes), 256, 0, s, g);
        count_launch(1);
    }
}

void launch_fill(const Fills &f, cudaStream_t s)
{
    long long words = 0;
    for (int q = 0; q < Fills::MAX; ++q) words = std::max(words, f.n[q]);
    if (words == 0) return;
    launch(k_fill, grid_x(words / 4 + 1, 256, 152 * 16), 256, 0, s, f);
    count_launch(1);
}

// one block up to LPT_SINGLE tiles: 16 rounds of its threads, against three launches of 2 to 7 us
constexpr int LPT_SINGLE = 16 * LPT_BINS;

void launch_lpt_order(const Globals &g, cudaStream_t s)
{
    if (g.total_tiles <= LPT_SINGLE) {
        launch(k_lpt_single, 1, LPT_BINS, 0, s, g);
        count_launch(1);
        return;
    }
    const int grid = grid_x(g.total_tiles, 256, 1024);
    launch(k_lpt_hist, grid, 256, 0, s, g);
    launch(k_lpt_scan, 1, LPT_BINS, 0, s, g);
    launch(k_lpt_scatter, grid, 256, 0, s, g);
    count_launch(3);
}

void launch_vertex_bwd(const Globals &g, int n_views, int max_nv, int n_meshes, int max_nf, bool normals,
                       cudaStream_t s)
{
    const int rows = normals ? n_meshes : g.gcol ? 1 : 0;
    const bool merge = rows > 0 && n_views + rows <= MAX_GRID_Y;
    const long long wide = !merge ? 0 : normals ? max_nf : g.n_verts_total;
    const int all = n_views + (merge ? rows : 0);
    const dim3 grid(grid_rows(std::max<long long>(max_nv, wide), 256, 2048, all), all);
    launch(k_vertex_bwd, grid, 256, 0, s, g);
    count_launch(1);
    if (g.gcol && !merge) {
        launch(k_color_bwd, grid_x(g.n_verts_total, 256, 2048), 256, 0, s, g);
        count_launch(1);
    }
    if (normals && !merge) {
        launch(k_normal_bwd, dim3(grid_x(max_nf, 256, 2048), n_meshes), 256, 0, s, g);
        count_launch(1);
    }
}

void launch_l2(const float *out, const float *tgt, long long n, float *grad, float *loss, cudaStream_t s)
{
    launch(k_l2, grid_x(n, 256, 152 * 8), 256, 0, s, out, tgt, n, grad, loss);
    count_launch(1);
}

}  // namespace dressi
