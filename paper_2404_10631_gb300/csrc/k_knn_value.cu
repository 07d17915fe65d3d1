// KNN filter without a spatial term (lambda^2 == 0): the K nearest in value
// over a pixel's whole row window.
//
// All pixels of a row share the window, and every key is e = fl((I_p - I_q)^2)
// with ties to the smaller index. So a CTA takes one row, sorts the window's
// values once (with their indices, a bitonic network in shared memory) and
// finds each pixel's K nearest by walking outwards from its place in the
// order, a lane per pixel: e does not decrease on either side (a rounded
// difference and its rounded square are monotone), so the next nearest is
// always one of two. Entries of equal e (equal values, values on both sides,
// or values whose rounded distances agree) are one group, listed by index; a
// group of many values (distances that underflow or overflow to one e) is
// taken from the window in index order, which stops at the K-th.
// O(n log^2 n) per row and O(K) per pixel, where the full scan
// (knn_kernel) forms n keys per pixel and, without a spatial term to bound
// them, keeps replacing its candidates. Measured: 208 x 256, K = 16, 7 rows
// 28 ms -> 47 us; 416 x 512, K = 40, 14 rows 179 ms -> 0.34 ms; 16 x 16, K = 8,
// 7 rows 1.8 ms -> 16 us: the sort is the better one at every size it takes.
//
// Bound: the sort's passes over shared memory (66 of 2048 entries for that
// map), then the gathers of the neighbours' probabilities.
#include <cuda_runtime.h>
#include <math.h>

#include "hsc_internal.cuh"
#include "knn_key.cuh"
#include "knn_value.cuh"

namespace hsc {
namespace {

constexpr int kThreads = 512;
// Runs of a group that give the full list nothing before the group is taken in
// index order instead. Two runs, one on either side, are a group of ordinary
// values; hundreds are one where the squared distances underflow or overflow
// (1 x 4096, values of 1e-24, K = 16: 39 ms run by run, 0.53 ms this way).
constexpr int kPastRuns = 16;

// Entries are (ordered value key << 32 | index).
__device__ __forceinline__ float value_of(unsigned long long x)
{
    return key_to_float((unsigned)(x >> 32));
}

// First entry of the sorted s[0..n) whose value key is >= v.
__device__ __forceinline__ int lower_bound(const unsigned long long *s, int n, unsigned v)
{
    int lo = 0, hi = n;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if ((unsigned)(s[mid] >> 32) < v) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

template <int KC>
__global__ void __launch_bounds__(kThreads)
knn_value_kernel(const float *__restrict__ I, const float *__restrict__ P, int H, int W, int K, int R,
                 int n2, float *__restrict__ O, int32_t *__restrict__ labels,
                 int32_t *__restrict__ nbr, Control *ctl)
{
    extern __shared__ unsigned long long s[];  // n2, a power of two >= the window
    const int r = blockIdx.x, tid = threadIdx.x;
    const int lo_r = max(0, r - R / 2);
    const int hi_r = min(H - 1, r + (R + 1) / 2 - 1);
    const int n = (hi_r - lo_r + 1) * W, q0 = lo_r * W;
    const long N = (long)H * W;
    bool bad = false;
    for (int i = tid; i < n2; i += kThreads) {
        unsigned long long e = ~0ull;  // after every entry
        if (i < n && HSC_IN_BOUNDS(q0 + i >= 0 && q0 + i < N, ctl)) {
            const float v = I[q0 + i];
            bad |= !isfinite(v);
            e = (unsigned long long)float_to_key(v == 0.f ? 0.f : v) << 32 | (unsigned)(q0 + i);
        }
        s[i] = e;
    }
    if (__syncthreads_or(bad) && tid == 0) atomicOr(&ctl->status, ST_NONFINITE_MAP);
    for (int k = 2; k <= n2; k <<= 1)
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int t = tid; t < n2 / 2; t += kThreads) {
                const int a = 2 * t - (t & (j - 1)), b = a + j;
                const unsigned long long x = s[a], y = s[b];
                if ((x > y) == ((a & k) == 0)) {
                    s[a] = y;
                    s[b] = x;
                }
            }
            __syncthreads();
        }

    for (int c = tid; c < W; c += kThreads) {
        const int p = r * W + c;
        const float Ip = I[p];
        auto dist = [&](int i) {
            const float d = __fsub_rn(Ip, value_of(s[i]));
            return __fmul_rn(d, d);
        };
        int sel[HSC_MAX_K];  // by (e, index)
        int m = 0, m0 = 0;   // listed, listed before this group
        // an entry of the group: sel[m0 ..] by index, the K - m0 smallest;
        // false when it and all larger indices are out
        auto put = [&](int q) {
            if (m == K && q > sel[K - 1]) return false;
            int at = m < K ? m++ : K - 1;
            for (; at > m0 && sel[at - 1] > q; --at) sel[at] = sel[at - 1];
            sel[at] = q;
            return true;
        };
        int rt = lower_bound(s, n, float_to_key(Ip == 0.f ? 0.f : Ip)), lf = rt - 1;
        while (m < K && (lf >= 0 || rt < n)) {
            const float el = lf >= 0 ? dist(lf) : INFINITY, er = rt < n ? dist(rt) : INFINITY;
            const float e = (lf >= 0 && !(el > er)) || rt >= n ? el : er;
            m0 = m;
            bool moved = false;
            int past = 0;  // runs all of whose indices are out
            // runs of one value, the indices of each ascending
            while (lf >= 0 && dist(lf) == e) {
                const unsigned v = (unsigned)(s[lf] >> 32);
                int i = lf;
                if (i > 0 && (unsigned)(s[i - 1] >> 32) == v) i = lower_bound(s, lf, v);
                const int first = i;
                while (i <= lf && put((int)(unsigned)s[i])) ++i;
                lf = first - 1;
                moved = true;
                if (i == first && ++past > kPastRuns) break;
            }
            while (rt < n && dist(rt) == e) {
                const unsigned v = (unsigned)(s[rt] >> 32);
                bool in = true;
                while (rt < n && (unsigned)(s[rt] >> 32) == v && (in = put((int)(unsigned)s[rt]))) ++rt;
                if (!in) rt = v == 0xffffffffu ? n : lower_bound(s, n, v + 1u);
                moved = true;
                if (!in && ++past > kPastRuns) break;
            }
            if (past > kPastRuns) {  // the group fills the list: its first by a scan in index order
                m = m0;
                for (int q = q0; m < K && q < q0 + n; ++q) {
                    const float v = __ldg(I + q);
                    const float d = __fsub_rn(Ip, v == 0.f ? 0.f : v);
                    if (__fmul_rn(d, d) == e) sel[m++] = q;
                }
                break;
            }
            if (!moved) {  // NaN: no e equals itself; any entry will do
                put((int)(unsigned)s[lf >= 0 ? lf : rt]);
                if (lf >= 0) --lf;
                else ++rt;
            }
        }
        if (m < K) atomicOr(&ctl->status, ST_KNN_SHORT);
        float acc[KC];
#pragma unroll
        for (int cl = 0; cl < KC; ++cl) acc[cl] = 0.f;
        for (int a = 0; a < m; ++a) {
            if (!HSC_IN_BOUNDS(sel[a] >= 0 && sel[a] < N, ctl)) continue;
            const float *Pq = P + sel[a];
#pragma unroll
            for (int cl = 0; cl < KC; ++cl) acc[cl] += __ldg(Pq + (size_t)cl * (size_t)N);
        }
        if (nbr) {
            for (int a = 0; a < m; ++a) nbr[(long)p * K + a] = sel[a];
            for (int a = m; a < K; ++a) nbr[(long)p * K + a] = -1;
        }
        write_pixel(acc, K, N, (long)p, O, labels);
    }
}

template <int KC>
cudaError_t launch(const float *I, const float *P, int H, int W, int K, int R, int n2, float *O,
                   int32_t *labels, int32_t *nbr, Control *ctl, cudaStream_t st)
{
    const size_t smem = sizeof(unsigned long long) * (size_t)n2;
    if (smem > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(
            knn_value_kernel<KC>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    knn_value_kernel<KC><<<H, kThreads, smem, st>>>(I, P, H, W, K, R, n2, O, labels, nbr, ctl);
    return cudaGetLastError();
}

// the network's size for a frame's largest window, 0: too large
int sort_size(int H, int W, int R)
{
    const long n = (long)(R < H ? R : H) * W;
    if (n > kKnnValueMax) return 0;
    int n2 = 2;
    while (n2 < n) n2 <<= 1;
    return n2;
}

}  // namespace

bool knn_value_applies(int H, int W, int R, float lam)
{
    return lam * lam == 0.f && sort_size(H, W, R) > 0;
}

cudaError_t launch_knn_value(const float *I, const float *P, int k, int H, int W, int K, int R,
                             float *O, int32_t *labels, int32_t *nbr, Control *ctl, cudaStream_t st)
{
    const int n2 = sort_size(H, W, R);
    if (n2 == 0) return cudaErrorInvalidValue;
    switch (k) {
#define HSC_VALUE_K(KC) \
    case KC: return launch<KC>(I, P, H, W, K, R, n2, O, labels, nbr, ctl, st);
        HSC_VALUE_K(1)
        HSC_VALUE_K(2)
        HSC_VALUE_K(3)
        HSC_VALUE_K(4)
        HSC_VALUE_K(5)
        HSC_VALUE_K(6)
        HSC_VALUE_K(7)
        HSC_VALUE_K(8)
#undef HSC_VALUE_K
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace hsc
