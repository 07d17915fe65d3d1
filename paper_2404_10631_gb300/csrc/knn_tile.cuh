// The tiled KNN walk's arguments and geometry (k_knn_tile.cu).
#pragma once

#include <cuda_runtime.h>

#include "hsc_internal.cuh"

namespace hsc {

constexpr int kKnnTileRows = 2;      // pixel rows per lane
constexpr int kKnnTileMaxWarps = 8;  // warps per CTA at most
constexpr int kTileShell = 8;        // entries of a shell at most (s <= 20)

// One frame's maps.
struct TileFrame {
    const float *I;
    const float *P;    // planes (used when P4 is null)
    const float4 *P4;  // pixel-interleaved, (k + 3) / 4 float4 per pixel
    float *O;          // nullable
    int32_t *labels;
    Control *ctl;
    long N;
    int H, W;
};

// (K <= 64: the K nearest offsets lie within s = dr^2 + dc^2 <= 20)
struct TileArgs {
    TileFrame frame;           // frames == null: this frame
    const BatchFrame *frames;  // a stage-major batch (frames[i].knn_cta0: CTA ranges)
    int n_frames, cta_base;
    int2 *redo_list;
    unsigned redo_cap;
    int K, R;
    float lam;
    int sK, disk, shell;  // K-th smallest s, entries below it, entries of it
    int prev, next;       // the largest s with entries below sK, the smallest above
    int rad;              // reach of s <= sK
    unsigned shell_r, shell_c;  // the shell's entries by index, 4 bits each: dr + 4, dc + 4
    int cut;              // the window cuts the disk: every pixel by itself
};

// A frame's CTAs: first the border pixels, one per thread (the pixels whose
// disk leaves the image, or every pixel), then the warps' tiles, 32 columns x
// kKnnTileRows rows each, rows fastest, over rows rad .. H - rad - 1.
struct TileGeom {
    long border_px;
    int border_ctas, row_groups, tiles;
};

__host__ __device__ inline TileGeom tile_geom(int H, int W, int rad, int cut, int warps)
{
    TileGeom g;
    const int ih = H - 2 * rad, iw = W - 2 * rad;
    if (cut || ih < kKnnTileRows || iw < 1) {
        g.border_px = (long)H * W;
        g.row_groups = 1;
        g.tiles = 0;
    } else {
        g.border_px = (long)H * W - (long)ih * iw;
        g.row_groups = (ih + kKnnTileRows - 1) / kKnnTileRows;
        g.tiles = g.row_groups * ((W + 31) / 32);
    }
    g.border_ctas = (int)((g.border_px + 32 * warps - 1) / (32 * warps));
    return g;
}

// The i-th border pixel: the rows above, the rows below, then the columns at
// both sides of the rows between (every pixel in order when there are no tiles).
__device__ __forceinline__ void border_pixel(const TileGeom &g, int H, int W, int rad, long i,
                                             int &r, int &c)
{
    const long top = g.tiles ? (long)rad * W : (long)H * W;
    if (i < top) {
        r = (int)(i / W);
        c = (int)(i - (long)r * W);
        return;
    }
    i -= top;
    if (i < top) {
        r = (int)(i / W);
        c = (int)(i - (long)r * W);
        r += H - rad;
        return;
    }
    i -= top;
    r = (int)(i / (2 * rad));
    c = (int)(i - (long)r * (2 * rad));
    if (c >= rad) c += W - 2 * rad;
    r += rad;
}

// The instantiations, probabilities from the interleaved copy or the planes (a
// translation unit each): the upload of its copy of the offset table, and the
// launch.
cudaError_t knn_tile_init_p4(const char2 *tab, int n);
cudaError_t knn_tile_init_planes(const char2 *tab, int n);
cudaError_t launch_knn_tile_p4(int k, const TileArgs &a, int ctas, int warps, cudaStream_t st);
cudaError_t launch_knn_tile_planes(int k, const TileArgs &a, int ctas, int warps, cudaStream_t st);

// The pruned search (lambda > 0) of one frame (frames null), or of a batch's
// frames over n_ctas CTAs numbered from cta_base; then the redo pass is due.
cudaError_t launch_knn_tile(const TileFrame &f, const BatchFrame *frames, int n_frames, int n_ctas,
                            int cta_base, int k, int K, int R, float lam, int2 *redo_list,
                            unsigned redo_cap, int warps, cudaStream_t st);

}  // namespace hsc
