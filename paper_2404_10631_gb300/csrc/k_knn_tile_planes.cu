// The tiled KNN walk (knn_tile_kernel.cuh) with the probabilities from the
// planes.
#include "knn_tile_kernel.cuh"

namespace hsc {

cudaError_t knn_tile_init_planes(const char2 *tab, int n) { return upload_knn_tab(tab, n); }

cudaError_t launch_knn_tile_planes(int k, const TileArgs &a, int ctas, int warps, cudaStream_t st)
{
    switch (k) {
    case 1: return launch_tile_kc<1, false>(a, ctas, warps, st);
    case 2: return launch_tile_kc<2, false>(a, ctas, warps, st);
    case 3: return launch_tile_kc<3, false>(a, ctas, warps, st);
    case 4: return launch_tile_kc<4, false>(a, ctas, warps, st);
    case 5: return launch_tile_kc<5, false>(a, ctas, warps, st);
    case 6: return launch_tile_kc<6, false>(a, ctas, warps, st);
    case 7: return launch_tile_kc<7, false>(a, ctas, warps, st);
    case 8: return launch_tile_kc<8, false>(a, ctas, warps, st);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace hsc
