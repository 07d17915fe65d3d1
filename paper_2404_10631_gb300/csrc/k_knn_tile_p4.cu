// The tiled KNN walk (knn_tile_kernel.cuh) with the probabilities from the
// pixel-interleaved copy.
#include "knn_tile_kernel.cuh"

namespace hsc {

cudaError_t knn_tile_init_p4(const char2 *tab, int n) { return upload_knn_tab(tab, n); }

cudaError_t launch_knn_tile_p4(int k, const TileArgs &a, int ctas, int warps, cudaStream_t st)
{
    switch (k) {
    case 2: return launch_tile_kc<2, true>(a, ctas, warps, st);
    case 3: return launch_tile_kc<3, true>(a, ctas, warps, st);
    case 4: return launch_tile_kc<4, true>(a, ctas, warps, st);
    case 5: return launch_tile_kc<5, true>(a, ctas, warps, st);
    case 6: return launch_tile_kc<6, true>(a, ctas, warps, st);
    case 7: return launch_tile_kc<7, true>(a, ctas, warps, st);
    case 8: return launch_tile_kc<8, true>(a, ctas, warps, st);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace hsc
