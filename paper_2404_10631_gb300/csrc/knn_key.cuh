// The exact distance key of the KNN filter (Eq. 1) and the offset table that
// orders candidates by spatial distance, shared by the KNN's translation
// units.
#pragma once

#include <cuda_runtime.h>
#include <math.h>

#include "hsc_internal.cuh"

namespace hsc {

// Offsets (dr, dc) with dr^2 + dc^2 <= 400 and |dr| <= 16, sorted by
// s = dr^2 + dc^2 (then dr, dc), built on the host once per device.
constexpr int kTabR2 = 400;            // table: dr^2 + dc^2 <= 400
constexpr int kTabDr = 16;             // |dr| <= 16: windows of up to 32 rows
constexpr int kTabDc = 20;             // |dc| <= 20 follows from kTabR2
constexpr int kTabCap = 1200;

// Labels of a pixel left to the redo pass: box_pixel with its larger buffer may
// finish it, or (kRedoFarLabel) only the unbounded walk can. The batch's list
// holds the latter's frame as ~frame.
constexpr int kRedoLabel = -2147483647 - 1;
constexpr int kRedoFarLabel = kRedoLabel + 1;
constexpr int kRedoCap = 32;  // undecided keys per lane in the redo pass's box_pixel

struct Key {
    float hi, lo;
    int q;
};

__device__ __forceinline__ bool key_le(const Key &a, const Key &b)
{
    return a.hi < b.hi || (a.hi == b.hi && (a.lo < b.lo || (a.lo == b.lo && a.q <= b.q)));
}
__device__ __forceinline__ bool key_lt(const Key &a, const Key &b)
{
    return a.hi < b.hi || (a.hi == b.hi && (a.lo < b.lo || (a.lo == b.lo && a.q < b.q)));
}

// Exact distance as (hi, lo) = s + e (Knuth's TwoSum, round-to-nearest ops).
__device__ __forceinline__ Key make_key(float Ip, float Iq, int dr, int dc, float l2, int q)
{
    float dI = __fsub_rn(Ip, Iq);
    float e = __fmul_rn(dI, dI);
    float s = __fmul_rn(l2, (float)(dr * dr + dc * dc));
    Key k;
    k.hi = __fadd_rn(s, e);
    float bb = __fsub_rn(k.hi, s);
    k.lo = __fadd_rn(__fsub_rn(s, __fsub_rn(k.hi, bb)), __fsub_rn(e, bb));
    k.q = q;
    return k;
}

__device__ __forceinline__ bool below_L(const Key &a, float L)
{
    return a.hi < L || (a.hi == L && a.lo < 0.f);
}

// O = acc / K per class and the label (the smaller class on ties).
template <int KC>
__device__ __forceinline__ void write_pixel(const float (&acc)[KC], int K, long N, long p,
                                            float *__restrict__ O, int32_t *__restrict__ labels)
{
    const float invK = 1.f / (float)K;
    int best = 0;
    float bestv = -INFINITY;
#pragma unroll
    for (int cl = 0; cl < KC; ++cl) {
        const float o = acc[cl] * invK;
        if (O) O[(size_t)cl * (size_t)N + p] = o;
        if (o > bestv) {
            bestv = o;
            best = cl;
        }
    }
    labels[p] = best;
}

// Host side of the tiled walk (k_knn_tile.cu).
// Uploads its copy of the offset table to the current device.
cudaError_t knn_tile_init(const char2 *tab, int n);
// CTAs (of `warps` warps) of one H x W frame.
int knn_tile_ctas(int H, int W, int K, int R, int warps);

}  // namespace hsc
