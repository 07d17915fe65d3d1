// Step (iii) of the PCA (Section II.C.2, III.A.2.c), the default form for one
// eigenvector and up to 256 bands: the leading eigenpair of the covariance
// from a Krylov space, refined in double-float.
//
//  1. Up to kSteps steps of Lanczos in FP32 on A = C / 2^e, each new vector made
//     orthogonal to all before it by classical Gram-Schmidt applied twice: a
//     basis Q and the tridiagonal T = Q^T A Q. The start vector is A's column
//     of the largest diagonal entry plus 1% of a fixed pseudo-random vector
//     (a start inside an invariant subspace would never leave it). Pixel
//     spectra have a few strong directions over a flat noise floor, so the
//     space holds the leading eigenvector to FP32 accuracy after as many
//     steps as there are such directions plus two or three.
//  2. T's largest eigenvalue by 33-section (a warp's 32 trial shifts at a
//     time, the signs of the pivots of T - x I), its vector s by inverse
//     iteration; v = Q s.
//  3. Refinement against C in double-float, as k_jacobi.cu's: with r = C v -
//     rho v and g = Q^T r,
//        v <- v + Q y + (r - Q g) / (rho - theta_c),  (sigma I - T) y = g,
//     sigma = theta_1 (1 + 1e-4) fixed, so that T's factors are formed once
//     (the shift only slows the convergence by 1e-4 / the relative gap), and
//     theta_c the mean of the eigenvalues outside the space, from the traces;
//     until ||r|| <= 1e-13 max(rho, max C_ii) ||v||. On the workloads' frames
//     two corrections.
//  4. Where a correction divides ||r|| by less than 4 (a spectrum that decays
//     with no floor: what is left of r lies outside the space), the space is
//     built again, from v and the double-float r; T's leading vector without
//     its first entry is the next correction, and each restart gains a
//     Chebyshev polynomial of degree 9 on the gap: 100-fold for a gap of 8%.
//  5. The sign rule; v / ||v||.
// A frame this cannot finish (a zero C, two restarts that gained less than 4:
// a leading eigenvalue hardly separated) is flagged (Control::jac_redo) for
// the full Jacobi kernel launched behind it.
//
// Layout: a thread holds 32 (16) of C's (hi, lo) pairs of one row in
// registers for the whole run, so a matrix-vector product reads only the
// vector, by broadcast. Up to 128 bands one CTA of 16 warps holds C; up to
// 256 bands a cluster of 8 CTAs, 32 rows each, which exchanges the product's
// 32 entries by distributed shared memory and one cluster barrier per step;
// everything after the exchange is done by every CTA alike, so they take the
// same decisions. A batch runs the one-CTA form with the same arithmetic, a
// CTA per frame.
//
// Bound: latency (a chain of about 50 block-wide phases: 2100 cycles a step,
// 4400 a correction, 9000 before the first step). The eigensolver stage, this
// kernel and the guarded one behind it, measured: 416 x 512 x 128 29 us (a
// block power step, Gram-Schmidt of 16 columns, Rayleigh-Ritz by Jacobi and 5
// corrections in one CTA: 87 us; always 10 steps here: 34 us); 1024 x 1024 x 256
// 29 us (one Jacobi sweep on a 16-CTA cluster, then 10-25 corrections on one
// CTA: 498 us); 300 x 400 x 200 29 us (450 us, and 3.5 ms for frames whose
// one-sweep basis did not converge). Eigenvalues e^(-j/8) and e^(-j/12), 200 x
// 200 pixels: 70 and 84 us with 128 bands, 88 and 126 us with 200 (corrections
// in the first space only, then the full kernel: 350 and 3200, 1150 and 12500
// us; the block power basis: 147 and 203, 12200 and 12260 us).
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "hsc_internal.cuh"
#include "pdl.cuh"
#include "dfloat.cuh"

namespace hsc {
namespace {

constexpr int kThreads = 512;
constexpr int kSteps = 10;
constexpr int kMaxRounds = 32;   // restarts at most
constexpr float kSlow = 16.f;    // a step that divides ||r||^2 by less is slow
constexpr float kShift = 1e-4f;
constexpr float kMargin = 4e-6f;

template <int CL>  // CTAs per cluster
struct Shape {
    static constexpr int kPad = CL == 1 ? 128 : 256;  // bands at most
    static constexpr int kRows = kPad / CL;           // rows per CTA
    static constexpr int kR = kRows / 32;             // row chunks of a warp
    static constexpr int kSlices = 16 / kR;           // column slices
    static constexpr int kNJ = kPad / kSlices;        // columns per thread
    static_assert(kSlices * kR * 32 == kThreads && kNJ % 16 == 0, "16 warps");
};

struct EigFrame {
    const float2 *C2;
    const double *mu;
    double *v1, *lambda1;
    float *v1f, *muf;
    Control *ctl;
};

template <int CL>
struct Smem {
    static constexpr int kPad = Shape<CL>::kPad;
    float Q[kSteps][kPad];
    float vh[kPad], vl[kPad];
    float y[2][kPad], r[kPad];  // y: Lanczos, two steps' buffers
    float2 part[Shape<CL>::kSlices][Shape<CL>::kRows];
    float2 x[2][kPad];  // the exchanged product, two steps' buffers
    float al[kSteps], be[kSteps];
    float ca[16], cb[16], n2[2];
    float4 red4[8];
    float red2[8];
    unsigned long long key[8];
    int arg[8];
    double scale;
};

__device__ __forceinline__ float warp_sum(float v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ dfl df_xor_sum(dfl x, int width)
{
    for (int o = width >> 1; o > 0; o >>= 1) {
        const dfl y = {__shfl_xor_sync(0xffffffffu, x.h, o), __shfl_xor_sync(0xffffffffu, x.l, o)};
        x = df_add(x, y);
    }
    return x;
}

// the dot product of two kPad-long vectors in shared memory, by a warp
template <int kPad>
__device__ __forceinline__ float dot(const float *a, const float *b, int lane)
{
    float s[kPad / 32];
#pragma unroll
    for (int i = 0; i < kPad / 32; ++i) s[i] = a[lane + 32 * i] * b[lane + 32 * i];
#pragma unroll
    for (int w = kPad / 64; w > 0; w >>= 1)
#pragma unroll
        for (int i = 0; i < w; ++i) s[i] += s[i + w];
    return warp_sum(s[0]);
}

__device__ __forceinline__ uint32_t cta_rank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

__device__ __forceinline__ void cluster_barrier()
{
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__device__ __forceinline__ uint32_t peer_addr(const void *local, uint32_t rank)
{
    const uint32_t a = (uint32_t)__cvta_generic_to_shared(local);
    uint32_t p;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(p) : "r"(a), "r"(rank));
    return p;
}
__device__ __forceinline__ void store_peer(const void *local, uint32_t rank, float v)
{
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(peer_addr(local, rank)), "f"(v) : "memory");
}
__device__ __forceinline__ void store_peer(const void *local, uint32_t rank, float2 v)
{
    const uint32_t p = peer_addr(local, rank);
    asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(p), "f"(v.x), "f"(v.y) : "memory");
}

// (x I - T) = L D L^T: f_c = beta_c / D_c and 1 / D_c. x exceeds T's largest
// eigenvalue by kMargin of it or more, a few dozen FP32 roundings, so every
// pivot is positive and 1 / D_c at most 1 / (kMargin x). (At the eigenvalue
// itself a pivot can come out as zero or negative before the last one; kept
// above 1e-7 x it made the next ones negative too, and their quotients
// overflowed: three frames of some 1200 were lost so.)
__device__ __forceinline__ void tri_factor(const float (&al)[kSteps], const float (&be)[kSteps],
                                           float x, float (&f)[kSteps], float (&inv)[kSteps])
{
    float d = x - al[0];
#pragma unroll
    for (int c = 0; c < kSteps; ++c) {
        inv[c] = __fdividef(1.f, d);
        f[c] = be[c] * inv[c];
        if (c + 1 < kSteps) d = (x - al[c + 1]) - be[c] * f[c];
    }
}
__device__ __forceinline__ void tri_solve(const float (&f)[kSteps], const float (&inv)[kSteps],
                                          float (&b)[kSteps])
{
#pragma unroll
    for (int c = 1; c < kSteps; ++c) b[c] = fmaf(f[c - 1], b[c - 1], b[c]);
    b[kSteps - 1] *= inv[kSteps - 1];
#pragma unroll
    for (int c = kSteps - 2; c >= 0; --c) b[c] = fmaf(f[c], b[c + 1], b[c] * inv[c]);
}

template <int CL, bool kBatch>
__global__ void __launch_bounds__(kThreads, 1)
krylov_kernel(int B, EigFrame fr, const BatchFrame *__restrict__ frames)
{
    typedef Shape<CL> Sh;
    constexpr int kPad = Sh::kPad, kRows = Sh::kRows, kSlices = Sh::kSlices, kNJ = Sh::kNJ;
    constexpr int kVW = kPad / 32;  // warps that hold a vector
    __shared__ __align__(16) Smem<CL> sm;
    pdl_wait();
    if (kBatch) {
        const BatchFrame &b = frames[blockIdx.x];
        fr = {b.C2, b.mu, b.v1, b.lambda1, b.v1f, b.muf, b.ctl};
    }
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t rank = CL > 1 ? cta_rank() : 0u;
    const float2 *__restrict__ C2 = fr.C2;
    const long long t0 = clock64();

    // ---- this thread's part of C: row `row`, columns j0 .. j0 + kNJ - 1 (its
    // loads are in flight while the diagonal is looked at)
    const int rl = (warp % Sh::kR) * 32 + lane, row = (int)rank * kRows + rl;
    const int sl = warp / Sh::kR, j0 = sl * kNJ;
    float ch[kNJ], cl[kNJ];
#pragma unroll
    for (int u = 0; u < kNJ; ++u) {
        const int j = j0 + u;
        const float2 c = row < B && j < B ? C2[(size_t)j * B + row] : make_float2(0.f, 0.f);
        ch[u] = c.x;
        cl[u] = c.y;
    }
    // ---- the diagonal: its maximum (the smaller band on ties) and its sum,
    // by every warp alike; A = C / 2^e (exact)
    float dmax, trace;
    int jmax, e2 = 0;
    {
        unsigned key = 0u;
        int at = 0;
        float s = 0.f;
#pragma unroll
        for (int i = 0; i < kVW; ++i) {
            const int b = lane + 32 * i;
            const float d = b < B ? C2[(size_t)b * B + b].x : 0.f;
            s += d;
            const unsigned k = __float_as_uint(fmaxf(d, 0.f));
            if (k > key) {
                key = k;
                at = b;
            }
        }
        trace = warp_sum(s);
        const unsigned top = __reduce_max_sync(0xffffffffu, key);
        jmax = __reduce_min_sync(0xffffffffu, key == top ? at : kPad);
        dmax = __uint_as_float(top);
    }
    if (!(dmax > 0.f) || !isfinite(dmax) || !isfinite(trace)) {  // uniform over the cluster
        if (rank == 0 && tid == 0) fr.ctl->jac_redo = 1u;
        return;
    }
    frexpf(dmax, &e2);
    e2 = e2 < -100 ? -100 : (e2 > 100 ? 100 : e2);
    const float inv_p2 = ldexpf(1.f, -e2);
    const float dmax_s = dmax * inv_p2;
    trace *= inv_p2;

#pragma unroll
    for (int u = 0; u < kNJ; ++u) {
        ch[u] *= inv_p2;
        cl[u] *= inv_p2;
    }
    // ---- the start vector
    if (tid < kPad) {
        const float g = (float)(((unsigned)tid * 2654435761u >> 16) & 1023u) * (1.f / 512.f) - 1.f;
        sm.y[1][tid] = tid < B ? fmaf(0.01f * dmax_s, g, C2[(size_t)jmax * B + tid].x * inv_p2) : 0.f;
    }
    __syncthreads();
    {
        const float n2 = dot<kPad>(sm.y[1], sm.y[1], lane);
        if (tid < kPad) sm.Q[0][tid] = sm.y[1][tid] * rsqrtf(n2);
    }
    __syncthreads();
    if constexpr (CL > 1) cluster_barrier();  // every CTA runs before its memory is written
    int par = 0;
    // the slices of a product's rows summed and given to every CTA; df: pairs
    auto exchange = [&](bool df) {
        if (CL > 1 ? warp < CL : tid < kPad) {
            const int rr = CL > 1 ? lane : tid;
            float s = 0.f, lo = 0.f;
#pragma unroll
            for (int k = 0; k < kSlices; ++k) {
                const float2 q = sm.part[k][rr];
                if (df) {
                    float e;
                    two_sum(s, q.x, s, e);
                    lo = __fadd_rn(lo, __fadd_rn(e, q.y));
                } else {
                    s += q.x;
                }
            }
            const int at = (int)rank * kRows + rr;
            if (!HSC_IN_BOUNDS(rr < kRows && at < kPad, fr.ctl)) {
                // (nothing is written; the barrier below is every thread's)
            } else if (df) {
                const dfl w = fast_two_sum(s, lo);
                if constexpr (CL > 1) store_peer(&sm.x[par][at], (uint32_t)warp, make_float2(w.h, w.l));
                else sm.x[par][at] = make_float2(w.h, w.l);
            } else {
                if constexpr (CL > 1) store_peer(&sm.y[par][at], (uint32_t)warp, s);
                else sm.y[par][at] = s;
            }
        }
        if constexpr (CL > 1) cluster_barrier();
        else __syncthreads();
    };

    const int m = B < kSteps ? B : kSteps;
    int k = 0, it = 0, stalled = 0;
    dfl rho = {0.f, 0.f}, vv = {0.f, 0.f};
    float e_last = INFINITY, e_round = INFINITY;  // ||r||^2 / ||v||^2 a step and a round ago
    bool converged = false;
    long long t1 = 0;
#pragma unroll 1
    for (int round = 0;; ++round) {
        // ---- Lanczos (a restart's first column and its row of T are there)
        float top = rho.h, prod = 1.f;
#pragma unroll 1
        for (int j = round ? 1 : 0;; ++j) {
            {
                float a0 = 0.f, a1 = 0.f;
                const float4 *q = reinterpret_cast<const float4 *>(sm.Q[j] + j0);
#pragma unroll
                for (int u = 0; u < kNJ; u += 4) {
                    const float4 v = q[u / 4];
                    a0 = fmaf(ch[u], v.x, a0);
                    a1 = fmaf(ch[u + 1], v.y, a1);
                    a0 = fmaf(ch[u + 2], v.z, a0);
                    a1 = fmaf(ch[u + 3], v.w, a1);
                }
                sm.part[sl][rl].x = a0 + a1;
            }
            __syncthreads();
            exchange(false);
            float *y = sm.y[par];
            par ^= 1;
            // two passes: the dot products with the columns so far (warp c) and
            // the vector's own square (warp j + 1), then the subtraction
#pragma unroll 1
            for (int pass = 0; pass < 2; ++pass) {
                if (warp <= j + 1) {
                    const float d = dot<kPad>(warp <= j ? sm.Q[warp] : y, y, lane);
                    if (lane == 0) {
                        if (warp <= j) (pass ? sm.cb : sm.ca)[warp] = d;
                        else sm.n2[pass] = d;
                    }
                }
                __syncthreads();
                if (pass == 0) {
                    if (tid < kPad) {
                        float v = y[tid];
#pragma unroll 4
                        for (int c = 0; c <= j; ++c) v = fmaf(-sm.ca[c], sm.Q[c][tid], v);
                        y[tid] = v;
                    }
                    __syncthreads();
                }
            }
            float b2 = sm.n2[1], v = tid < kPad ? y[tid] : 0.f;
#pragma unroll 4
            for (int c = 0; c <= j; ++c) {
                const float d = sm.cb[c];
                b2 = fmaf(-d, d, b2);
                if (tid < kPad) v = fmaf(-d, sm.Q[c][tid], v);
            }
            // The space is exhausted when what is left of the product is rounding,
            // and large enough when the product of beta / theta (theta by the
            // largest alpha so far) is: it bounds the leading Ritz vector's last
            // component, its share of the residual, up to the gaps.
            const float alpha = sm.ca[j] + sm.cb[j];
            top = fmaxf(top, alpha);
            prod *= fminf(1.f, b2 * __fdividef(1.f, top * top));  // squares
            const bool last = j == m - 1 || !(b2 > 1e-12f * sm.n2[0]) || prod < 1e-24f;
            const float ib = last ? 0.f : rsqrtf(b2);
            if (tid == 0) {
                sm.al[j] = alpha;
                sm.be[j] = last ? 0.f : b2 * ib;
            }
            if (last) {
                k = j + 1;
                break;
            }
            if (!HSC_IN_BOUNDS(j + 1 < kSteps, fr.ctl)) break;  // uniform
            if (tid < kPad) sm.Q[j + 1][tid] = v * ib;
            __syncthreads();
        }
        __syncthreads();

        // ---- T's largest eigenvalue and its vector (a restart: the new part of
        // it, (theta I - T') t = beta_0 ||v|| e_1 without the first row and column,
        // which keeps its digits when beta_0 is small), by every thread alike
        float f[kSteps], inv[kSteps], s[kSteps];
        float theta, rest;
        {
            float al[kSteps], be[kSteps];
            float lo = -INFINITY, hi = -INFINITY, sum = 0.f, bp = 0.f;
#pragma unroll
            for (int c = 0; c < kSteps; ++c) {
                // past the space: a pivot of 1e30, which leaves its component zero
                al[c] = c < k ? sm.al[c] : -1e30f;
                be[c] = c < k ? sm.be[c] : 0.f;
                sum += c < k ? al[c] : 0.f;
                lo = fmaxf(lo, al[c]);
                hi = fmaxf(hi, al[c] + bp + be[c]);
                bp = be[c];
            }
            rest = trace - sum;
            hi = hi * (1.f + 1e-6f);
#pragma unroll 1
            for (int round = 0; round < 4; ++round) {
                const float x = lo + (hi - lo) * ((float)(lane + 1) * (1.f / 32.f));
                float d = al[0] - x;
                bool above = d < 0.f;
#pragma unroll
                for (int c = 1; c < kSteps; ++c) {
                    d = (al[c] - x) - __fdividef(be[c - 1] * be[c - 1], d);
                    above = above && d < 0.f;
                }
                const unsigned mask = __ballot_sync(0xffffffffu, above) | 0x80000000u;
                const int first = __ffs(mask) - 1;
                const float nh = __shfl_sync(0xffffffffu, x, first);
                const float nl = __shfl_sync(0xffffffffu, x, first > 0 ? first - 1 : 0);
                lo = first > 0 ? nl : lo;
                hi = nh;
            }
            theta = hi;
            const float a0 = al[0], b0 = be[0], xs = theta * (1.f + kMargin);
            if (round) {
                al[0] = -1e30f;
                be[0] = 0.f;
            }
            tri_factor(al, be, xs, f, inv);
            if (round) {
#pragma unroll
                for (int c = 0; c < kSteps; ++c) s[c] = 0.f;
                s[1] = b0 * sqrtf(vv.h);
                tri_solve(f, inv, s);
                al[0] = a0;
                be[0] = b0;
            } else {
#pragma unroll
                for (int c = 0; c < kSteps; ++c) s[c] = 1.f;
#pragma unroll 1
                for (int i = 0; i < 2; ++i) {
                    tri_solve(f, inv, s);
                    float n2 = 0.f;
#pragma unroll
                    for (int c = 0; c < kSteps; ++c) {
                        s[c] *= 1e-4f;  // (the squares of 1e7 stay far inside FP32's range)
                        n2 = fmaf(s[c], s[c], n2);
                    }
                    const float sc = rsqrtf(n2);
#pragma unroll
                    for (int c = 0; c < kSteps; ++c) s[c] *= sc;
                }
            }
            tri_factor(al, be, theta * (1.f + kShift), f, inv);
        }
        if (tid < kPad) {
            float v = 0.f;
#pragma unroll
            for (int c = 0; c < kSteps; ++c)
                if (c < k) v = fmaf(s[c], sm.Q[c][tid], v);
            if (round) {  // v += Q t
                float sum, e;
                two_sum(sm.vh[tid], v, sum, e);
                const dfl nv = fast_two_sum(sum, __fadd_rn(sm.vl[tid], e));
                sm.vh[tid] = nv.h;
                sm.vl[tid] = nv.l;
            } else {
                sm.vh[tid] = v;
                sm.vl[tid] = 0.f;
            }
        }
        __syncthreads();
        if (round == 0) t1 = clock64();

        // ---- refinement (double-float; v is not renormalised between steps)
        const bool deflate = B > k;
        const float theta_c = deflate ? rest / (float)(B - k) : 0.f;
        float e_now = 0.f, rn = 0.f;
#pragma unroll 1
        for (;; ++it) {
            // w = A v: the products split exactly by an FMA, summed by TwoSum,
            // the small terms in FP32, at most 16 per chain
            {
                constexpr int kCh = kNJ / 16;
                float sum[kCh], lo[kCh];
#pragma unroll
                for (int h = 0; h < kCh; ++h) sum[h] = lo[h] = 0.f;
#pragma unroll
                for (int u = 0; u < 16; ++u)
#pragma unroll
                    for (int h = 0; h < kCh; ++h) {
                        const int j = u + 16 * h;
                        const float vh = sm.vh[j0 + j], vl = sm.vl[j0 + j];
                        const float p = __fmul_rn(ch[j], vh);
                        const float pe = __fmaf_rn(ch[j], vh, -p);
                        float e;
                        two_sum(sum[h], p, sum[h], e);
                        lo[h] = __fadd_rn(lo[h], e);
                        lo[h] = __fadd_rn(lo[h], pe);
                        lo[h] = __fmaf_rn(ch[j], vl, lo[h]);
                        lo[h] = __fmaf_rn(cl[j], vh, lo[h]);
                    }
                if constexpr (kCh > 1) {
                    float e;
                    two_sum(sum[0], sum[1], sum[0], e);
                    lo[0] = __fadd_rn(__fadd_rn(lo[0], lo[1]), e);
                }
                sm.part[sl][rl] = make_float2(sum[0], lo[0]);
            }
            __syncthreads();
            exchange(true);
            const float2 *w = sm.x[par];
            par ^= 1;
            if (warp < kVW) {
                const dfl v = {sm.vh[tid], sm.vl[tid]}, wi = {w[tid].x, w[tid].y};
                const dfl tvv = df_xor_sum(df_mul(v, v), 32), tvw = df_xor_sum(df_mul(v, wi), 32);
                if (lane == 0) sm.red4[warp] = make_float4(tvv.h, tvv.l, tvw.h, tvw.l);
            }
            __syncthreads();
            {  // every warp forms the same rho from the same partials
                const float4 q = sm.red4[lane % kVW];
                vv = df_xor_sum({q.x, q.y}, kVW);
                rho = df_div(df_xor_sum({q.z, q.w}, kVW), vv);
            }
            if (warp < kVW) {
                const dfl pv = df_mul(rho, {sm.vh[tid], sm.vl[tid]});
                const dfl r = df_add({w[tid].x, w[tid].y}, {-pv.h, -pv.l});
                const float ri = __fadd_rn(r.h, r.l);
                sm.r[tid] = ri;
                const float r2 = warp_sum(ri * ri);
                if (lane == 0) sm.red2[warp] = r2;
            }
            __syncthreads();
            float rr = 0.f;
#pragma unroll
            for (int i = 0; i < kVW; ++i) rr += sm.red2[i];
            const float tol = 1e-13f * fmaxf(fabsf(rho.h), dmax_s);
            converged = rr <= tol * tol * vv.h;
            rn = sqrtf(rr);
            e_now = rr / vv.h;
            // one restart after another once the first space has given what it
            // has (NaN counts as slow)
            if (converged || round || !(e_now * kSlow < e_last)) break;
            e_last = e_now;
            if (warp < k) {
                const float g = dot<kPad>(sm.Q[warp], sm.r, lane);
                if (lane == 0) sm.ca[warp] = g;
            }
            __syncthreads();
            if (tid < kPad) {
                const float den = rho.h - theta_c;
                const float idc = deflate && fabsf(den) > 1e-3f * fabsf(rho.h) ? 1.f / den : 0.f;
                float g[kSteps], y[kSteps];
#pragma unroll
                for (int c = 0; c < kSteps; ++c) y[c] = g[c] = c < k ? sm.ca[c] : 0.f;
                tri_solve(f, inv, y);
                float acc = sm.r[tid] * idc;
#pragma unroll
                for (int c = 0; c < kSteps; ++c)
                    if (c < k) acc = fmaf(fmaf(-g[c], idc, y[c]), sm.Q[c][tid], acc);
                float sum, e;
                two_sum(sm.vh[tid], acc, sum, e);
                const dfl nv = fast_two_sum(sum, __fadd_rn(sm.vl[tid], e));
                sm.vh[tid] = nv.h;
                sm.vl[tid] = nv.l;
            }
            __syncthreads();
        }
        if (converged) break;
        if (round && !(e_now * kSlow < e_round)) ++stalled;
        if (stalled == 2 || round == kMaxRounds || B < 2) break;
        e_round = e_now;
        ++it;
        // ---- restart: the columns v / ||v|| and r / ||r|| (from the double-float
        // residual: FP32's product would not know it), T's first row
        if (tid < kPad) sm.Q[0][tid] = sm.vh[tid] * rsqrtf(vv.h);
        __syncthreads();
        {
            const float g = dot<kPad>(sm.Q[0], sm.r, lane);
            if (tid < kPad) sm.Q[1][tid] = fmaf(-g, sm.Q[0][tid], sm.r[tid]);
        }
        __syncthreads();
        {
            const float n2 = dot<kPad>(sm.Q[1], sm.Q[1], lane);
            __syncthreads();
            if (tid < kPad) sm.Q[1][tid] *= rsqrtf(n2);
            if (tid == 0) {
                sm.al[0] = rho.h;
                sm.be[0] = rn * rsqrtf(vv.h);
            }
        }
        __syncthreads();
    }
    if (rank != 0) return;  // no CTA reads a peer's memory after the last barrier
    if (!converged) {
        if (tid == 0) fr.ctl->jac_redo = 1u;
        return;
    }

    // ---- outputs: v / ||v||, the largest |v_i| positive (the smaller band on
    // a tie; |v_i| ordered by the integer value of its bits), lambda = rho 2^e.
    // 1 / ||v|| by one cubic correction of the FP32 value in FP64 (its
    // operations have a 64-cycle latency: no FP64 square root or division).
    double x = 0.0;
    if (warp < kVW) {
        x = (double)sm.vh[tid] + (double)sm.vl[tid];
        unsigned long long key = (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffull;
        int arg = tid;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long k2 = __shfl_xor_sync(0xffffffffu, key, o);
            const int a2 = __shfl_xor_sync(0xffffffffu, arg, o);
            if (k2 > key || (k2 == key && a2 < arg)) {
                key = k2;
                arg = a2;
            }
        }
        if (lane == 0) {
            sm.key[warp] = key;
            sm.arg[warp] = arg;
        }
    } else if (tid == kPad) {
        const double n2 = (double)vv.h + (double)vv.l;
        const double q = (double)rsqrtf(vv.h);
        const double e = fma(-n2 * q, q, 1.0);
        sm.scale = fma(q * e, fma(0.375, e, 0.5), q);
        *fr.lambda1 = ldexp((double)rho.h + (double)rho.l, e2);
    }
    __syncthreads();
    if (tid < B) {
        unsigned long long key = sm.key[0];
        int arg = sm.arg[0];
#pragma unroll
        for (int i = 1; i < kVW; ++i)
            if (sm.key[i] > key) {  // equal: the smaller band is in the earlier warp
                key = sm.key[i];
                arg = sm.arg[i];
            }
        const float bh = sm.vh[arg], bl = sm.vl[arg];
        const bool neg = bh < 0.f || (bh == 0.f && bl < 0.f);
        const double v = (neg ? -sm.scale : sm.scale) * x;
        fr.v1[tid] = v;
        fr.v1f[tid] = (float)v;
        fr.muf[tid] = (float)fr.mu[tid];
    }
    if (tid == 0) {
        Control *ctl = fr.ctl;
        ctl->jacobi_sweeps = CL > 1 ? 1u : 0u;  // the cluster's basis counts as one
        ctl->refine_iters = (unsigned)it;
        ctl->jacobi_sweep_cycles = (unsigned long long)(t1 - t0);
        ctl->jacobi_refine_cycles = (unsigned long long)(clock64() - t1);
        ctl->jac_redo = 0u;
        ctl->svm_done = 0u;
        ctl->imin_key = float_to_key(INFINITY);
        ctl->imax_key = float_to_key(-INFINITY);
    }
}

}  // namespace

bool krylov_applies(int B) { return B >= 1 && B <= Shape<8>::kPad; }

cudaError_t launch_krylov(int B, const PcaScratch &s, cudaStream_t st)
{
    const EigFrame fr = {s.C2, s.mu, s.v1, s.lambda1, s.v1f, s.muf, s.ctl};
    if (B <= Shape<1>::kPad) {
        return launch_pdl(krylov_kernel<1, false>, dim3(1), dim3(kThreads), 0, st, B, fr, nullptr);
    }
    if (!krylov_applies(B)) return cudaErrorInvalidValue;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 8;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // as launch_pdl
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = dim3(8, 1, 1);
    cfg.blockDim = dim3(kThreads, 1, 1);
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    const BatchFrame *none = nullptr;
    return cudaLaunchKernelEx(&cfg, krylov_kernel<8, false>, B, fr, none);
}

cudaError_t launch_batch_krylov(const BatchFrame *frames, int n_frames, int B, cudaStream_t st)
{
    if (n_frames < 1 || B < 1 || B > Shape<1>::kPad) return cudaErrorInvalidValue;
    krylov_kernel<1, true><<<n_frames, kThreads, 0, st>>>(B, EigFrame{}, frames);
    return cudaGetLastError();
}

}  // namespace hsc
