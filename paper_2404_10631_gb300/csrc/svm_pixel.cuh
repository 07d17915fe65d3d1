// The per-pixel arithmetic of the projection/SVM pass (Section II.C.2 step
// (iv) and Section II.C.1 / III.A.1), shared by its own kernels and by the
// stage-major batch's fused projection/SVM + KNN kernel: the pairwise
// coupling solve, one pixel's finish (I, decision values, Platt, coupling,
// probabilities), the band loop over groups of pixels, the staging of the
// weights and the block min/max of I.
#pragma once

#include <cuda_runtime.h>
#include <math.h>

#include "hsc_internal.cuh"
#include "dfloat.cuh"

namespace hsc {
namespace {

// Threads of the batch's projection/SVM CTAs (the strided load form's pixel
// stride).
constexpr int kSvmThreads = 256;

// Floats per band of the staged weights (w_0 .. w_{M-1}, v1, mu), padded to
// 16-byte loads.
__host__ __device__ constexpr int svm_stride(int k)
{
    return (k * (k - 1) / 2 + 2 + 3) & ~3;
}

// The coupling of one pixel: (Q + e e^T) y = e, p = y / sum y, by LDL^T in
// FP32. kRefine (HSC_SVM_COUPLE_F64): two steps of iterative refinement to
// better than FP64's accuracy, in double-float on the FP32 pipe. Solved is Q y
// = c e, c = 1 - e^T y kept as an unknown of its own: in c - (Q y)_i the terms
// of a class that loses every pair are all as small as its y_i, where 1 -
// ((Q + e e^T) y)_i would cancel against the winner's y = 1 and lose them (one
// correction in that form: relative errors up to 1e-6 for p = 1e-8). The
// products r_ij r_ji and squares r_ji^2 are FP32 pairs (1 - r is exact as one,
// products are split by an FMA), the correction d comes from the FP32 factors
// of Q + e e^T (condition number below 25: each step gains six digits), then
// y += d and c -= e^T d as pairs; sum and quotient in pairs. Against exact
// rational arithmetic (consistent, cyclic and clipped r, 2 to 8 classes) p is
// the correctly rounded FP32 value in 99.5% of the cases, the FP64 LDL^T's in
// 99.3%, and never more than 1.00 half-units off.
// 509 x 401 x 100, 6 classes: 46 us with one correction, 47 us with these two,
// 112 us in FP64 arithmetic throughout (250 operations and 7 divisions at under
// two per clock and SM).
template <int KC, bool kRefine>
__device__ __forceinline__ void couple_solve(const float *r /* M, pair order */, float *p)
{
    float R[KC][KC];
    {
        int m = 0;
#pragma unroll
        for (int i = 0; i < KC; ++i)
#pragma unroll
            for (int j = i + 1; j < KC; ++j, ++m) {
                R[i][j] = r[m];
                R[j][i] = 1.f - r[m];
            }
    }
    // A = Q + e e^T (symmetric), stored lower part in L with D separate
    float L[KC][KC], D[KC], invD[KC];
#pragma unroll
    for (int i = 0; i < KC; ++i) {
        float d = 1.f;
#pragma unroll
        for (int j = 0; j < KC; ++j)
            if (j != i) d += R[j][i] * R[j][i];
        L[i][i] = d;
#pragma unroll
        for (int j = 0; j < i; ++j) L[i][j] = 1.f - R[j][i] * R[i][j];
    }
    // LDL^T in place
#pragma unroll
    for (int j = 0; j < KC; ++j) {
        float d = L[j][j];
#pragma unroll
        for (int m = 0; m < j; ++m) d -= L[j][m] * L[j][m] * D[m];
        D[j] = d;
        invD[j] = 1.f / d;
#pragma unroll
        for (int i = j + 1; i < KC; ++i) {
            float t = L[i][j];
#pragma unroll
            for (int m = 0; m < j; ++m) t -= L[i][m] * L[j][m] * D[m];
            L[i][j] = t * invD[j];
        }
    }
    auto solve = [&](float (&y)[KC]) {  // L D L^T y = y
#pragma unroll
        for (int i = 0; i < KC; ++i) {
            float t = y[i];
#pragma unroll
            for (int m = 0; m < i; ++m) t -= L[i][m] * y[m];
            y[i] = t;
        }
#pragma unroll
        for (int i = 0; i < KC; ++i) y[i] *= invD[i];
#pragma unroll
        for (int i = KC - 1; i >= 0; --i) {
            float t = y[i];
#pragma unroll
            for (int m = i + 1; m < KC; ++m) t -= L[m][i] * y[m];
            y[i] = t;
        }
    };
    float y[KC];
#pragma unroll
    for (int i = 0; i < KC; ++i) y[i] = 1.f;
    solve(y);
    if constexpr (!kRefine) {
        float s = 0.f;
#pragma unroll
        for (int i = 0; i < KC; ++i) s += y[i];
        const float inv = 1.f / s;
#pragma unroll
        for (int i = 0; i < KC; ++i) p[i] = y[i] * inv;
    } else {
        // Q's entries as pairs: r_ij r_ji per class pair, sum_j r_ji^2 per class
        constexpr int M = KC * (KC - 1) / 2;
        float qh[M], ql[M], ds[KC], dl[KC];
#pragma unroll
        for (int i = 0; i < KC; ++i) ds[i] = dl[i] = 0.f;
        auto add_sq = [&](int i, float h, float l) {  // diagonal i += (h + l)^2
            const float q = __fmul_rn(h, h);
            const float qe = __fmaf_rn(__fmul_rn(2.f, h), l, __fmaf_rn(h, h, -q));
            float e;
            two_sum(ds[i], q, ds[i], e);
            dl[i] = __fadd_rn(dl[i], __fadd_rn(e, qe));
        };
        {
            int m = 0;
#pragma unroll
            for (int i = 0; i < KC; ++i)
#pragma unroll
                for (int j = i + 1; j < KC; ++j, ++m) {
                    float h, l;  // 1 - r_ij = r_ji
                    two_sum(1.f, -r[m], h, l);
                    add_sq(i, h, l);
                    add_sq(j, r[m], 0.f);
                    qh[m] = __fmul_rn(r[m], h);
                    ql[m] = __fmaf_rn(r[m], l, __fmaf_rn(r[m], h, -qh[m]));
                }
        }
        float yl[KC], ch = 1.f, cl = 0.f;  // y = y + yl, c = ch + cl
#pragma unroll
        for (int i = 0; i < KC; ++i) {
            const dfl a = fast_two_sum(ds[i], dl[i]);
            ds[i] = a.h;
            dl[i] = a.l;
            yl[i] = 0.f;
            ch -= y[i];
        }
#pragma unroll 1
        for (int it = 0; it < 2; ++it) {
            float rs[KC], rl[KC];  // c - (Q y)_i
#pragma unroll
            for (int i = 0; i < KC; ++i) {
                rs[i] = ch;
                rl[i] = cl;
            }
            auto add = [&](int i, float ah, float al, int j) {  // res_i += (ah + al) y_j
                const float q = __fmul_rn(ah, y[j]);
                float t = __fmaf_rn(ah, y[j], -q);
                t = __fmaf_rn(al, y[j], t);
                t = __fmaf_rn(ah, yl[j], t);
                float e;
                two_sum(rs[i], q, rs[i], e);
                rl[i] = __fadd_rn(rl[i], __fadd_rn(e, t));
            };
            int m = 0;
#pragma unroll
            for (int i = 0; i < KC; ++i)
#pragma unroll
                for (int j = i + 1; j < KC; ++j, ++m) {
                    add(i, qh[m], ql[m], j);
                    add(j, qh[m], ql[m], i);
                }
            float d[KC], g = 0.f;
#pragma unroll
            for (int i = 0; i < KC; ++i) {
                add(i, -ds[i], -dl[i], i);
                d[i] = __fadd_rn(rs[i], rl[i]);
            }
            solve(d);
            float e;
#pragma unroll
            for (int i = 0; i < KC; ++i) {
                g += d[i];
                float t;
                two_sum(y[i], d[i], t, e);
                const dfl n = fast_two_sum(t, __fadd_rn(yl[i], e));
                y[i] = n.h;
                yl[i] = n.l;
            }
            float t;
            two_sum(ch, -g, t, e);
            const dfl n = fast_two_sum(t, __fadd_rn(cl, e));
            ch = n.h;
            cl = n.l;
        }
        float s = 0.f, sl = 0.f;
#pragma unroll
        for (int i = 0; i < KC; ++i) {
            float e;
            two_sum(s, y[i], s, e);
            sl = __fadd_rn(sl, __fadd_rn(e, yl[i]));
        }
        const dfl sum = fast_two_sum(s, sl);
        const float inv = 1.f / sum.h;
#pragma unroll
        for (int i = 0; i < KC; ++i) {
            const float q = __fmul_rn(y[i], inv);
            const float rem = __fadd_rn(__fmaf_rn(-q, sum.h, y[i]), __fmaf_rn(-q, sum.l, yl[i]));
            p[i] = __fmaf_rn(rem, inv, q);
        }
    }
}

// The end of one pixel's work, common to every form of the pass: I (and its
// running min/max), the M decision values f = acc + bias, Platt, coupling, the
// k probabilities, the label and the pixel-interleaved copy.
template <int KC, bool kF64>
__device__ __forceinline__ void finish_svm_pixel(const float (&acc)[KC * (KC - 1) / 2 > 0 ? KC * (KC - 1) / 2 : 1],
                                             float accI, long p, long N, bool do_pca,
                                             const float *sbias, const float *sa, const float *sb,
                                             float *__restrict__ I_raw, float *__restrict__ probs,
                                             int32_t *__restrict__ labels,
                                             float &lmin, float &lmax, bool &bad,
                                             float4 *__restrict__ P4)
{
    constexpr int M = KC * (KC - 1) / 2;
    constexpr int MA = M > 0 ? M : 1;
    if (do_pca) {
        const float I = accI;
        bad |= !isfinite(I);
        I_raw[p] = I;
        lmin = fminf(lmin, I);
        lmax = fmaxf(lmax, I);
    }
    if constexpr (M > 0) {
        float r[MA];
#pragma unroll
        for (int m = 0; m < M; ++m) {
            float f = acc[m] + sbias[m];
            bad |= !isfinite(f);
            float rr = 1.f / (1.f + expf(fmaf(sa[m], f, sb[m])));
            r[m] = fminf(fmaxf(rr, 1e-7f), 1.f - 1e-7f);
        }
        float pr[KC > 0 ? KC : 1];
        couple_solve<KC, kF64>(r, pr);
        int best = 0;
        float bv = pr[0];
#pragma unroll
        for (int c = 0; c < KC; ++c) {
            probs[(size_t)c * (size_t)N + p] = pr[c];
            if (pr[c] > bv) {
                bv = pr[c];
                best = c;
            }
        }
        if (labels) labels[p] = best;
        if (P4) {  // pixel-interleaved copy for the KNN's gathers
            constexpr int NQ = (KC + 3) / 4;
#pragma unroll
            for (int i = 0; i < NQ; ++i) {
                float v[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) v[e] = 4 * i + e < KC ? pr[4 * i + e] : 0.f;
                P4[(size_t)p * NQ + i] = make_float4(v[0], v[1], v[2], v[3]);
            }
        }
    }
}

// The per-pixel work of the pass for groups g_begin, g_begin + g_step, ...
// below g_end of PX pixels: group g holds pixels g * PX + u (one 16-byte
// load per band when kVec, else PX 4-byte loads), or, kStrided, pixels
// p_base + g + u * kSvmThreads (4-byte loads, each coalesced across the warp).
// ws holds svm_stride(KC) floats per band (16-byte aligned): w_0..w_{M-1}, v1,
// mu. The arithmetic of a pixel does not
// depend on the grouping or the loads.
// The loads run kAhead bands ahead: a band's register is reloaded as soon as
// its values are used, so a thread always has that many loads in flight. (In
// blocks of 16 bands, loaded and then used, all warps of the one wave waited
// out the memory's latency once per block. Measured: the projection alone on
// 416 x 512 x 128 30.4 -> 19.0 us, on 300 x 400 x 200 45 -> 26 us; 256 snapshot
// frames' projection + SVM 54 + 87 -> 43 + 75 us; with 4 classes on 416 x 512 x
// 128 the coupling solves after the last band are the rest, 27 us both ways.)
// Loads in flight per thread in the single-frame launches (kAhead PX registers
// beside (M + 1) PX accumulators); the batch's kernels, three CTAs of 256
// threads per SM at 80 registers, take 4.
// (24 with the refined coupling of 4 classes: 128 registers, four CTAs per SM.)
constexpr int svm_ahead(int k, int px, bool f64)
{
    return px == 4 ? 8 : px == 2 ? 16 : k >= 5 ? 16 : k == 4 && f64 ? 24 : 32;
}

template <int KC, int PX, bool kVec, bool kF64, bool kStrided = false,
          int kAhead = svm_ahead(KC, PX, kF64)>
__device__ __forceinline__ void project_svm_groups(
    const float *__restrict__ cube, int B, long N, const float *ws, const float *sbias,
    const float *sa, const float *sb, bool do_pca, long g_begin, long g_end, long g_step,
    float *__restrict__ I_raw, float *__restrict__ probs, int32_t *__restrict__ labels,
    float &lmin, float &lmax, bool &bad, long p_base = 0,
    float4 *__restrict__ P4 = nullptr)
{
    constexpr int M = KC * (KC - 1) / 2;
    constexpr int MA = M > 0 ? M : 1;
    constexpr int S = svm_stride(KC);
    constexpr long kPs = kStrided ? kSvmThreads : 1;  // pixel stride within a group
    for (long g = g_begin; g < g_end; g += g_step) {
        const long p0 = kStrided ? p_base + g : g * PX;
        float acc[MA][PX];
        float accI[PX];
#pragma unroll
        for (int u = 0; u < PX; ++u) {
            accI[u] = 0.f;
#pragma unroll
            for (int m = 0; m < MA; ++m) acc[m][u] = 0.f;
        }
        float x[kAhead][PX];
        auto load = [&](float (&v)[PX], int b) {
            const float *src = cube + (size_t)b * (size_t)N + p0;
            if constexpr (PX == 4 && kVec) {
                const float4 q = __ldcs(reinterpret_cast<const float4 *>(src));
                v[0] = q.x;
                v[1] = q.y;
                v[2] = q.z;
                v[3] = q.w;
            } else if constexpr (PX == 2 && kVec) {
                const float2 q = __ldcs(reinterpret_cast<const float2 *>(src));
                v[0] = q.x;
                v[1] = q.y;
            } else {
#pragma unroll
                for (int u = 0; u < PX; ++u)
                    v[u] = (p0 + u * kPs < N) ? __ldcs(src + u * kPs) : 0.f;
            }
        };
        auto use = [&](const float (&v)[PX], int b) {
            float wr[S];
            const float4 *w4 = reinterpret_cast<const float4 *>(ws + b * S);
#pragma unroll
            for (int i = 0; i < S / 4; ++i) {
                const float4 q = w4[i];
                wr[4 * i] = q.x;
                wr[4 * i + 1] = q.y;
                wr[4 * i + 2] = q.z;
                wr[4 * i + 3] = q.w;
            }
#pragma unroll
            for (int m = 0; m < M; ++m)
#pragma unroll
                for (int u = 0; u < PX; ++u) acc[m][u] = fmaf(wr[m], v[u], acc[m][u]);
#pragma unroll
            for (int u = 0; u < PX; ++u) accI[u] = fmaf(wr[M], v[u] - wr[M + 1], accI[u]);
        };
#pragma unroll
        for (int i = 0; i < kAhead; ++i)
            if (i < B) load(x[i], i);
        int b = 0;
#pragma unroll 1
        for (; b + 2 * kAhead <= B; b += kAhead) {
#pragma unroll
            for (int i = 0; i < kAhead; ++i) {
                use(x[i], b + i);
                load(x[i], b + i + kAhead);
            }
        }
        // the last bands: fewer than kAhead still to load
#pragma unroll
        for (int i = 0; i < kAhead; ++i) {
            if (b + i >= B) break;
            use(x[i], b + i);
            if (b + i + kAhead < B) load(x[i], b + i + kAhead);
        }
        b += kAhead;
#pragma unroll
        for (int i = 0; i < kAhead; ++i) {
            if (b + i >= B) break;
            use(x[i], b + i);
        }
#pragma unroll
        for (int u = 0; u < PX; ++u) {
            const long p = p0 + u * kPs;
            if (p >= N) break;
            float a[MA];
#pragma unroll
            for (int m = 0; m < MA; ++m) a[m] = acc[m][u];
            finish_svm_pixel<KC, kF64>(a, accI[u], p, N, do_pca, sbias, sa, sb, I_raw, probs, labels,
                                       lmin, lmax, bad, P4);
        }
    }
}

// Stages per band w_0..w_{M-1}, v1, mu and the Platt constants in shared memory.
template <int KC>
__device__ __forceinline__ void stage_weights(int B, const float *__restrict__ v1f,
                                              const float *__restrict__ muf,
                                              const float *__restrict__ w,
                                              const float *__restrict__ bias,
                                              const float *__restrict__ pa,
                                              const float *__restrict__ pb, float *ws,
                                              float *sbias, float *sa, float *sb)
{
    constexpr int M = KC * (KC - 1) / 2;
    constexpr int S = svm_stride(KC);
    const bool do_pca = (v1f != nullptr);
    // a band per thread: its rows' loads go together, each coalesced over bands
    for (int b = threadIdx.x; b < B; b += blockDim.x) {
        float v[S];
#pragma unroll
        for (int m = 0; m < S; ++m)
            v[m] = m < M ? w[(size_t)m * B + b] : 0.f;
        if (do_pca) {
            v[M] = v1f[b];
            v[M + 1] = muf[b];
        }
        float4 *dst = reinterpret_cast<float4 *>(ws + b * S);
#pragma unroll
        for (int i = 0; i < S / 4; ++i)
            dst[i] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
    }
    if constexpr (M > 0)
        for (int m = threadIdx.x; m < M; m += blockDim.x) {
            sbias[m] = bias[m];
            sa[m] = pa[m];
            sb[m] = pb[m];
        }
}

// Block min/max of I into the ordered-int keys, the non-finite flag.
__device__ __forceinline__ void finish_block(bool do_pca, float lmin, float lmax, bool bad,
                                             Control *ctl)
{
    if (do_pca) {
        for (int o = 16; o > 0; o >>= 1) {
            lmin = fminf(lmin, __shfl_xor_sync(0xffffffffu, lmin, o));
            lmax = fmaxf(lmax, __shfl_xor_sync(0xffffffffu, lmax, o));
        }
        if ((threadIdx.x & 31) == 0 && lmin <= lmax) {
            atomicMin(&ctl->imin_key, float_to_key(lmin));
            atomicMax(&ctl->imax_key, float_to_key(lmax));
        }
    }
    if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(&ctl->status, ST_NONFINITE_CUBE);
}

}  // namespace
}  // namespace hsc
