// Host side of the tiled KNN walk (knn_tile_kernel.cuh).
#include <cuda_runtime.h>

#include "knn_key.cuh"
#include "knn_tile.cuh"

namespace hsc {
namespace {

int isqrt(int x)
{
    int r = 0;
    while ((r + 1) * (r + 1) <= x) ++r;
    return r;
}

// offsets (dr, dc) with dr^2 + dc^2 == s
int shell_size(int s)
{
    int n = 0;
    for (int a = -isqrt(s); a <= isqrt(s); ++a) {
        const int b = isqrt(s - a * a);
        if (a * a + b * b == s) n += b ? 2 : 1;
    }
    return n;
}

void fill_args(TileArgs &a, int K, int R)
{
    a.K = K;
    a.R = R;
    // the K nearest offsets of an unbounded window
    a.disk = 0;
    a.prev = 0;
    for (a.sK = 0;; ++a.sK) {
        a.shell = shell_size(a.sK);
        if (a.disk + a.shell >= K) break;
        a.disk += a.shell;
        if (a.shell) a.prev = a.sK;
    }
    a.next = a.sK + 1;
    while (!shell_size(a.next)) ++a.next;
    a.rad = isqrt(a.sK);
    a.shell_r = a.shell_c = 0u;
    for (int dr = -a.rad, i = 0; dr <= a.rad; ++dr)
        for (int dc = -a.rad; dc <= a.rad; ++dc)
            if (dr * dr + dc * dc == a.sK) {
                a.shell_r |= (unsigned)(dr + 4) << (4 * i);
                a.shell_c |= (unsigned)(dc + 4) << (4 * i);
                ++i;
            }
    // a window that cuts the disk leaves every pixel to box_pixel
    a.cut = a.rad > R / 2 || a.rad > (R + 1) / 2 - 1;
}

}  // namespace

cudaError_t knn_tile_init(const char2 *tab, int n)
{
    const cudaError_t e = knn_tile_init_p4(tab, n);
    return e == cudaSuccess ? knn_tile_init_planes(tab, n) : e;
}

int knn_tile_ctas(int H, int W, int K, int R, int warps)
{
    TileArgs a{};
    fill_args(a, K, R);
    const TileGeom g = tile_geom(H, W, a.rad, a.cut, warps);
    return g.border_ctas + (g.tiles + warps - 1) / warps;
}

cudaError_t launch_knn_tile(const TileFrame &f, const BatchFrame *frames, int n_frames, int n_ctas,
                            int cta_base, int k, int K, int R, float lam, int2 *redo_list,
                            unsigned redo_cap, int warps, cudaStream_t st)
{
    TileArgs a{};
    a.frame = f;
    a.frames = frames;
    a.n_frames = n_frames;
    a.cta_base = cta_base;
    a.redo_list = redo_list;
    a.redo_cap = redo_cap;
    a.lam = lam;
    fill_args(a, K, R);
    if (!frames) n_ctas = knn_tile_ctas(f.H, f.W, K, R, warps);
    return frames || f.P4 ? launch_knn_tile_p4(k, a, n_ctas, warps, st)
                          : launch_knn_tile_planes(k, a, n_ctas, warps, st);
}

}  // namespace hsc
