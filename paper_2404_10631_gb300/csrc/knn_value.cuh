// The KNN filter without a spatial term (k_knn_value.cu).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "hsc_internal.cuh"

namespace hsc {

// The largest window (candidates) it sorts: 128 KB of shared memory. Larger
// ones take the full scan.
constexpr long kKnnValueMax = 16384;

bool knn_value_applies(int H, int W, int R, float lam);
cudaError_t launch_knn_value(const float *I, const float *P, int k, int H, int W, int K, int R,
                             float *O, int32_t *labels, int32_t *nbr, Control *ctl, cudaStream_t st);

}  // namespace hsc
