// The exact K nearest of any pixels (KNN filter, pruned search), a lane each:
// the tiled walk's border pixels (knn_tile_kernel.cuh) and the second pass
// over what the tiles left (k_knn.cu).
#pragma once

#include <cuda_runtime.h>
#include <math.h>

#include <algorithm>
#include <type_traits>
#include <vector>

#include "hsc_internal.cuh"
#include "knn_key.cuh"
#include "knn_tile.cuh"

namespace hsc {
namespace {

// The offset table (each translation unit holds a copy: upload_knn_tab).
// Entries from c_knn_tab_n on are outside every window (dr = 127).
__constant__ __align__(16) char2 c_knn_tab[kTabCap];
__constant__ int c_knn_tab_n;
static_assert(kTabCap % 8 == 0, "read 8 entries at a time");

inline cudaError_t upload_knn_tab(const char2 *tab, int n)
{
    std::vector<char2> all((size_t)kTabCap, make_char2(127, 0));
    std::copy(tab, tab + n, all.begin());
    cudaError_t e = cudaMemcpyToSymbol(c_knn_tab, all.data(), sizeof(char2) * all.size());
    if (e == cudaSuccess) e = cudaMemcpyToSymbol(c_knn_tab_n, &n, sizeof(int));
    return e;
}


// The probabilities of one pixel, loaded and added per class: pairs of
// classes in one 64-bit register (packed FP32 additions, each rounded as the
// scalar one) from the pixel-interleaved copy, or scalars from the planes.
template <int KC, bool kP4>
struct Acc;

template <int KC>
struct Acc<KC, true> {
    static constexpr int NP = (KC + 1) / 2, NQ = (KC + 3) / 4;
    unsigned long long v[NP];
    typedef const float4 *Ptr;  // a pixel's place; neighbours of its row at fixed offsets
    static __device__ __forceinline__ Ptr at(const TileFrame &f, int q)
    {
        return f.P4 + (size_t)(unsigned)q * NQ;
    }
    __device__ __forceinline__ void zero()
    {
#pragma unroll
        for (int i = 0; i < NP; ++i) v[i] = 0ull;
    }
    __device__ __forceinline__ void load(Ptr p, int d)
    {
#pragma unroll
        for (int i = 0; i < NQ; ++i) {
            if (2 * i + 1 < NP) {
                asm("ld.global.nc.v2.u64 {%0, %1}, [%2];"
                    : "=l"(v[2 * i]), "=l"(v[2 * i + 1])
                    : "l"(p + d * NQ + i));
            } else {
                asm("ld.global.nc.u64 %0, [%1];" : "=l"(v[2 * i]) : "l"(p + d * NQ + i));
            }
        }
    }
    __device__ __forceinline__ void add(const Acc &o)
    {
#pragma unroll
        for (int i = 0; i < NP; ++i) asm("add.rn.f32x2 %0, %0, %1;" : "+l"(v[i]) : "l"(o.v[i]));
    }
    __device__ __forceinline__ void get(float (&out)[KC]) const
    {
#pragma unroll
        for (int i = 0; i < KC; ++i)
            out[i] = __uint_as_float((unsigned)(i & 1 ? v[i / 2] >> 32 : v[i / 2] & 0xffffffffull));
    }
};

template <int KC>
struct Acc<KC, false> {
    float v[KC];
    struct Ptr {
        const float *c[KC];
    };
    static __device__ __forceinline__ Ptr at(const TileFrame &f, int q)
    {
        Ptr p;
#pragma unroll
        for (int i = 0; i < KC; ++i) p.c[i] = f.P + ((size_t)i * (size_t)f.N + (unsigned)q);
        return p;
    }
    __device__ __forceinline__ void zero()
    {
#pragma unroll
        for (int i = 0; i < KC; ++i) v[i] = 0.f;
    }
    __device__ __forceinline__ void load(const Ptr &p, int d)
    {
#pragma unroll
        for (int i = 0; i < KC; ++i) v[i] = __ldg(p.c[i] + d);
    }
    __device__ __forceinline__ void add(const Acc &o)
    {
#pragma unroll
        for (int i = 0; i < KC; ++i) v[i] += o.v[i];
    }
    __device__ __forceinline__ void get(float (&out)[KC]) const
    {
#pragma unroll
        for (int i = 0; i < KC; ++i) out[i] = v[i];
    }
};

// The undecided keys of one lane in shared memory: entry i's hi, lo and q are
// the words 3 i, 3 i + 1 and 3 i + 2 of the lane's column (128 bytes apart) at
// the 32-bit shared address a.
struct Buf {
    uint32_t a;
    __device__ __forceinline__ Key get(int i) const
    {
        Key k;
        const uint32_t p = a + 384u * (uint32_t)i;
        asm volatile("ld.shared.f32 %0, [%1];" : "=f"(k.hi) : "r"(p));
        asm volatile("ld.shared.f32 %0, [%1+128];" : "=f"(k.lo) : "r"(p));
        asm volatile("ld.shared.s32 %0, [%1+256];" : "=r"(k.q) : "r"(p));
        return k;
    }
    __device__ __forceinline__ void put(int i, const Key &k) const
    {
        const uint32_t p = a + 384u * (uint32_t)i;
        asm volatile("st.shared.f32 [%0], %1;" ::"r"(p), "f"(k.hi));
        asm volatile("st.shared.f32 [%0+128], %1;" ::"r"(p), "f"(k.lo));
        asm volatile("st.shared.s32 [%0+256], %1;" ::"r"(p), "r"(k.q));
    }
};
constexpr size_t buf_bytes(int cap) { return (size_t)cap * 384; }  // per warp

// floor(sqrt(x)), 0 <= x < 2^20
__device__ __forceinline__ int isqrt_d(int x)
{
    int r = (int)sqrtf((float)x);  // exact, or one off
    r -= r * r > x ? 1 : 0;
    r += (r + 1) * (r + 1) <= x ? 1 : 0;
    return r;
}

// The pixels of a warp one by one, a lane each, any 32 pixels (all 32 lanes
// call; p < 0: none). sK comes from counting valid offsets in increasing s.
// The warp walks the rows of the box that holds every lane's disk s <= s_K
// together, four columns' loads at a time; a lane adds the candidates of
// s < s_K whose key is below L as they come (canonical order) and lists the
// others. tau = L + e_max over the candidates seen bounds the K-th key; where
// it reaches past s_K the ring up to it is walked the same way. The K - m
// smallest of the list complete the set. Returns the keys kept, or that the
// pixel is not finished: kLeftKeys (more than cap undecided keys, kRedoCap
// hold them) or kLeftFar (more still, or a disk beyond the table's).
constexpr unsigned kLeftFar = ~0u, kLeftKeys = ~0u - 1u;
template <int KC, bool kP4>
__device__ __forceinline__ unsigned box_pixel(const TileFrame &f, int p, int K, int R, float l2,
                                              Buf buf, int cap)
{
    const unsigned kAll = 0xffffffffu;
    const int W = f.W;
    const bool on = p >= 0;
    if (!on) p = 0;
    const int r = p / W, c = p - r * W;
    const int up = min(r, R / 2), dn = min(f.H - 1 - r, (R + 1) / 2 - 1);
    const float *__restrict__ Ic = f.I + p;
    const float Ip = __ldg(Ic);
    if (on && !isfinite(Ip)) atomicOr(&f.ctl->status, ST_NONFINITE_MAP);
    int sK = on ? -1 : 0;
    {
        const int ntab = c_knn_tab_n;
        int cnt = 0;
#pragma unroll 1
        for (int t = 0; on && t < ntab; t += 8) {  // 8 entries per 16-byte load
            if (!HSC_IN_BOUNDS(t + 8 <= kTabCap, f.ctl)) break;
            const uint4 w4 = *reinterpret_cast<const uint4 *>(c_knn_tab + t);
            const unsigned w[4] = {w4.x, w4.y, w4.z, w4.w};
            unsigned mask = 0u;
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int dr = (int)(w[u / 2] << (u & 1 ? 8 : 24)) >> 24;
                const int dc = (int)(w[u / 2] << (u & 1 ? 0 : 16)) >> 24;
                const bool v = (unsigned)(dr + up) <= (unsigned)(up + dn) &&
                               (unsigned)(c + dc) < (unsigned)W;
                mask |= v ? 1u << u : 0u;
            }
            const int n8 = __popc(mask);
            if (cnt + n8 >= K) {  // the K-th is the (K - cnt)-th of these
                for (int i = 1; i < K - cnt; ++i) mask &= mask - 1u;
                const char2 o = c_knn_tab[t + __ffs(mask) - 1];
                sK = o.x * o.x + o.y * o.y;
                break;
            }
            cnt += n8;
        }
        __syncwarp();
    }
    bool ok = on && sK >= 0;
    const float L = __fmul_rn(l2, (float)sK);
    Acc<KC, kP4> acc;
    acc.zero();
    int m = 0, n = 0;
    float dmax = 0.f, tau = INFINITY;
    // candidates whose loads go together (by the registers of their P)
    constexpr int kU = KC <= 4 ? 4 : 2;
    // the candidates s0 < s <= s1 of this lane (s1 < 0: none), s1w the
    // largest s1 of the warp; ring: only list, and only keys <= tau
    auto walk = [&](auto ring_tag, int s0, int s1, int s1w) {
        constexpr bool kRing = decltype(ring_tag)::value;
        typedef Acc<KC, kP4> A;
        const int reach = isqrt_d(s1w);
        const int d0 = -__reduce_max_sync(kAll, s1 < 0 ? 0 : min(up, reach));
        const int d1 = __reduce_max_sync(kAll, s1 < 0 ? 0 : min(dn, reach));
#pragma unroll 1
        for (int dr = d0; dr <= d1; ++dr) {
            const int w = isqrt_d(s1w - dr * dr), dr2 = dr * dr;
            const bool row = dr >= -up && dr <= dn;
            // this lane's part of the row: |dc| <= wl, columns 0 .. W-1
            const int wl = row && s1 >= dr2 ? isqrt_d(s1 - dr2) : -1;
            const int c0 = max(-wl, -c), c1 = min(wl, W - 1 - c);
            const int q = row ? p + dr * W : p;
            const float *__restrict__ Ir = f.I + q;
            typename A::Ptr Pr;
            if constexpr (!kRing) Pr = A::at(f, q);
#pragma unroll 1
            for (int dc = -w; dc <= w; dc += kU) {
                float x[kU];
                A pv[kU];
                bool in[kU];
#pragma unroll
                for (int u = 0; u < kU; ++u) {
                    const int d = dc + u;
                    in[u] = d >= c0 && d <= c1;
                    if constexpr (kRing) in[u] = in[u] && dr2 + d * d > s0;
                    in[u] = in[u] && HSC_IN_BOUNDS(q + d >= 0 && q + d < f.N, f.ctl);
                    x[u] = in[u] ? __ldg(Ir + d) : Ip;
                    if constexpr (!kRing)
                        if (in[u]) pv[u].load(Pr, d);
                }
#pragma unroll
                for (int u = 0; u < kU; ++u) {
                    const float st = __fmul_rn(l2, (float)(dr2 + (dc + u) * (dc + u)));
                    const float d = __fsub_rn(Ip, x[u]);
                    const float e = __fmul_rn(d, d);
                    const float h = __fadd_rn(st, e);
                    if constexpr (!kRing) {
                        dmax = fmaxf(dmax, fabsf(d));
                        if (in[u] && h < L) {  // (only s < s_K)
                            ++m;
                            acc.add(pv[u]);
                            continue;
                        }
                    }
                    if (in[u] && !(kRing && h > tau)) {
                        const float bb = __fsub_rn(h, st);
                        const Key kk = {h, __fadd_rn(__fsub_rn(st, __fsub_rn(h, bb)), __fsub_rn(e, bb)),
                                        q + dc + u};
                        if (!kRing && below_L(kk, L)) {
                            ++m;
                            acc.add(pv[u]);
                        } else {
                            if (n < cap) buf.put(n, kk);
                            ++n;
                        }
                    }
                }
            }
        }
    };
    walk(std::false_type(), -1, ok ? sK : -1, __reduce_max_sync(kAll, ok ? sK : 0));
    // every key of the K nearest is <= L + e_max; candidates of s_term > tau
    // are farther (s1: the largest s to look at, at least sK)
    int s1 = -1;
    if (ok) {
        tau = __fadd_ru(L, __fmul_ru(dmax, dmax));
        const float q = __fdiv_ru(tau * (1.f + 1.f / 1048576.f), l2);
        if (!(q < (float)(kTabR2 + 1))) ok = false;  // the ring leaves the table's disk
        else if (__fmul_rn(l2, (float)(sK + 1)) <= tau) s1 = (int)q;
    }
    const int s1w = __reduce_max_sync(kAll, s1);
    if (s1w >= 0) walk(std::true_type(), sK, s1, s1w);
    const int need = K - m;
    if (!ok || n > cap || n < need) {  // (n < need: NaN in the map)
        if (!on) return 0u;
        return ok && n > cap && n <= kRedoCap ? kLeftKeys : kLeftFar;
    }
#pragma unroll 1
    for (int a = 0; a < need; ++a) {  // the smallest of entries a .. n-1 to place a
        const Key first = buf.get(a);
        Key best = first;
        int im = a;
#pragma unroll 4
        for (int b = a + 1; b < n; ++b) {
            const Key kb = buf.get(b);
            const bool less = key_lt(kb, best);
            best.hi = less ? kb.hi : best.hi;
            best.lo = less ? kb.lo : best.lo;
            best.q = less ? kb.q : best.q;
            im = less ? b : im;
        }
        buf.put(im, first);
        if (!HSC_IN_BOUNDS(im < cap && best.q >= 0 && best.q < f.N, f.ctl)) continue;
        Acc<KC, kP4> x;
        x.load(Acc<KC, kP4>::at(f, best.q), 0);
        acc.add(x);
    }
    float out[KC];
    acc.get(out);
    write_pixel(out, K, f.N, (long)p, f.O, f.labels);
    return (unsigned)(m + n);
}

}  // namespace
}  // namespace hsc
