// KNN filter, pruned search (lambda > 0), tiled: a warp takes 32 columns x 2
// rows of pixels, a lane one column.
//
// Every key is s_term + e with s_term = fl(lambda^2 (dr^2 + dc^2)) and
// e = fl((I_p - I_q)^2). With s_K the K-th smallest dr^2 + dc^2 of a pixel's
// valid candidates and L = fl(lambda^2 s_K), the K-th smallest key lies in
// [L, L + e_max], e_max the largest e of the K spatially nearest. For a pixel
// whose whole disk dr^2 + dc^2 <= s_K lies inside the window and the image,
// s_K depends on K alone; and when e_max, taken over the warp's (or the lane's)
// neighbourhood, is smaller than the step from the shell before s_K to it and
// from it to the next one (with lambda >= 1 and a map in [0, 1] this is nearly
// always so), the K nearest are known without a search: the whole disk
// dr^2 + dc^2 < s_K, plus the K - |disk| entries of the shell
// dr^2 + dc^2 == s_K with the smallest (e, index). So the tile path forms no
// keys for the disk: it adds P over one of the 12 patterns that s_K takes for
// K <= 64, in the canonical order (the rounding of O does not depend on the
// path), then picks from the shell in registers.
//
// The other pixels take box_pixel: the image's border, whose disks are cut, in
// CTAs of their own, numbered first; lanes with too large an e_max in their
// own warp, a row at a time (left to a second kernel they came to it in
// clusters, a few warps with several rows each: 509 x 401, K = 24, lambda 0.5
// 60 us). Pixels with too many undecided keys there are left to the second
// pass (labels kRedoLabel, kRedoFarLabel).
//
// Measured, walk and second pass together, against one pixel per lane with
// every candidate of the disk keyed and P gathered by dependent loads:
// 416 x 512, K = 40, 14 rows, lambda 1, 4 classes: 66 -> 23 us; 1024 x 1024:
// 183 -> 39 us; 509 x 401, K = 24, 9 rows, lambda 0.5, 3 classes: 275 -> 36 us.
//
// What bounds it: instruction issue (1024 x 1024: 50% of the slots, L1 at 72%)
// and, on frames of a few hundred thousand
// pixels, how fast the code itself arrives (each warp runs the pattern once).
// Four rows per lane with the shell unrolled per row were 2500 instructions
// and waited 11.8 of 14 cycles for instructions; the same loops rolled up
// with run-time widths issued twice as many. Two rows, the pattern unrolled
// and the shell rolled, keep both small.
#pragma once

#include <cuda_runtime.h>
#include <math.h>

#include "hsc_internal.cuh"
#include "knn_generic.cuh"
#include "pdl.cuh"

namespace hsc {
namespace {

constexpr int kV = kKnnTileRows;  // rows per lane
constexpr int kTileCap = 16;      // undecided keys per border pixel

__host__ __device__ constexpr int isqrt_c(int x)
{
    int r = 0;
    while ((r + 1) * (r + 1) <= x) ++r;
    return r;
}

// Adds the disk dr^2 + dc^2 < SK of the pixels (r0 .. r0 + kV - 1, c), q0 the
// first one's index: straight-line code, each entry loaded once for the rows
// that share it, a pixel's entries by increasing index.
template <int KC, bool kP4, int SK>
__device__ __forceinline__ void add_disk(const TileFrame &f, int q0, Acc<KC, kP4> (&acc)[kV])
{
    if constexpr (SK > 0) {
        constexpr int RD = isqrt_c(SK - 1);
        const int W = f.W;
#pragma unroll
        for (int rho = -RD; rho <= kV - 1 + RD; ++rho) {
            const auto row = Acc<KC, kP4>::at(f, q0 + rho * W);
#pragma unroll
            for (int dc = -RD; dc <= RD; ++dc) {
                bool any = false;
#pragma unroll
                for (int v = 0; v < kV; ++v) any |= (rho - v) * (rho - v) + dc * dc < SK;
                if (!any) continue;
                Acc<KC, kP4> x;
                x.load(row, dc);
#pragma unroll
                for (int v = 0; v < kV; ++v)
                    if ((rho - v) * (rho - v) + dc * dc < SK) acc[v].add(x);
            }
        }
    }
}

// Orders the shell's e by (e, entry): word of the entries' numbers, nearest
// first, 4 bits each. e's bits with the entry in the lowest 3 are sorted as
// integers (19 compare-exchanges); where two share the other 29 bits the
// order is taken from the e themselves, one minimum after another.
__device__ __forceinline__ unsigned shell_order(const float (&e)[kTileShell], int shell, int need)
{
    static_assert(kTileShell == 8, "an 8-input network");
    unsigned k[8];
#pragma unroll
    for (int i = 0; i < 8; ++i)
        k[i] = i < shell ? (__float_as_uint(e[i]) & ~7u) | (unsigned)i : 0xffffff00u + 9u * i;
    auto cx = [&](int a, int b) {
        const unsigned lo = min(k[a], k[b]), hi = max(k[a], k[b]);
        k[a] = lo;
        k[b] = hi;
    };
    cx(0, 1), cx(2, 3), cx(4, 5), cx(6, 7);
    cx(0, 2), cx(1, 3), cx(4, 6), cx(5, 7);
    cx(1, 2), cx(5, 6);
    cx(0, 4), cx(1, 5), cx(2, 6), cx(3, 7);
    cx(2, 4), cx(3, 5);
    cx(1, 2), cx(3, 4), cx(5, 6);
    bool tie = false;
    unsigned ord = 0u;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        if (i < 7) tie |= (k[i] ^ k[i + 1]) < 8u;
        ord |= (k[i] & 7u) << (4 * i);
    }
    if (tie) {
        ord = 0u;
        unsigned used = 0u;
#pragma unroll 1
        for (int n = 0; n < need; ++n) {
            float be = 0.f;
            int bi = -1;
#pragma unroll
            for (int i = 0; i < 8; ++i)
                if (i < shell && !(used >> i & 1u) && (bi < 0 || e[i] < be)) {
                    be = e[i];
                    bi = i;
                }
            used |= 1u << bi;
            ord |= (unsigned)bi << (4 * n);
        }
    }
    return ord;
}

// The tile path: rows r0 .. r0 + kV - 1, this lane's column c0 + lane.
// Returns whether this lane's pixels are done: not when its e_max leaves more
// than the shell undecided (nothing is written then). on: the lane's disks lie
// inside the image; vfirst: rows before it belong to another warp.
template <int KC, bool kP4>
__device__ __forceinline__ bool tile_fast(const TileFrame &f, const TileArgs &a, int r0, int c0,
                                          int lane, bool on, int vfirst, float l2)
{
    const int W = f.W, rad = a.rad;
    // (every access below is within rad of rows r0 .. r0 + kV - 1 and of a
    // column clamped to rad .. W - 1 - rad)
    if (!HSC_IN_BOUNDS(r0 >= rad && r0 + kV - 1 + rad < f.H && W > 2 * rad, f.ctl)) return false;
    const int c = c0 + lane;
    // an off lane computes a neighbour's pixel (its loads stay in bounds)
    const int ca = min(max(c, rad), W - 1 - rad);
    const int q0 = r0 * W + ca;
    bool ok;
    {
        // region column i is image column c0 - rad + i: lane l reads columns l
        // and (l < 2 rad) 32 + l, rows r0 - rad .. r0 + kV - 1 + rad
        float alo = INFINITY, ahi = -INFINITY, blo = INFINITY, bhi = -INFINITY;
        const int x1 = min(max(c0 - rad + lane, 0), W - 1);
        const int x2 = lane < 2 * rad ? min(c0 - rad + 32 + lane, W - 1) : x1;
        const float *Ir = f.I + (long)(r0 - rad) * W;
#pragma unroll 4
        for (int i = 0; i < kV + 2 * rad; ++i) {
            const float v = __ldg(Ir + i * W + x1);
            const float w = __ldg(Ir + i * W + x2);
            alo = fminf(alo, v);
            ahi = fmaxf(ahi, v);
            blo = fminf(blo, w);
            bhi = fmaxf(bhi, w);
        }
        const float L = __fmul_rn(l2, (float)a.sK);
        const float Lp = __fmul_rn(l2, (float)a.prev), Ln = __fmul_rn(l2, (float)a.next);
        // (false with an infinite value; a NaN neighbour counts as absent, its
        // own pixel reports it)
        auto decided = [&](float dI) {
            const float em = __fmul_ru(dI, dI);
            return Ln > __fadd_ru(L, em) && (a.sK == 0 || __fadd_ru(Lp, em) < L);
        };
        float vmin = fminf(alo, blo), vmax = fmaxf(ahi, bhi);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            vmin = fminf(vmin, __shfl_xor_sync(0xffffffffu, vmin, o));
            vmax = fmaxf(vmax, __shfl_xor_sync(0xffffffffu, vmax, o));
        }
        ok = decided(__fsub_ru(vmax, vmin));
        if (!ok) {  // warp-uniform: each lane over its own columns, from its own values
            vmin = INFINITY;
            vmax = -INFINITY;
#pragma unroll 1
            for (int d = 0; d <= 2 * rad; ++d) {
                const int src = lane + d;
                const float a0 = __shfl_sync(0xffffffffu, alo, src & 31);
                const float a1 = __shfl_sync(0xffffffffu, ahi, src & 31);
                const float b0 = __shfl_sync(0xffffffffu, blo, src & 31);
                const float b1 = __shfl_sync(0xffffffffu, bhi, src & 31);
                vmin = fminf(vmin, src < 32 ? a0 : b0);
                vmax = fmaxf(vmax, src < 32 ? a1 : b1);
            }
            float dI = 0.f;
#pragma unroll
            for (int v = 0; v < kV; ++v) {
                const float Ip = __ldg(f.I + q0 + v * W);
                dI = fmaxf(dI, fmaxf(__fsub_ru(Ip, vmin), __fsub_ru(vmax, Ip)));
            }
            ok = decided(dI);
            if (__ballot_sync(0xffffffffu, ok && on) == 0u) return false;
        }
    }
    Acc<KC, kP4> acc[kV];
#pragma unroll
    for (int v = 0; v < kV; ++v) acc[v].zero();
    switch (a.sK) {
#define HSC_TILE_DISK(SK) \
    case SK: add_disk<KC, kP4, SK>(f, q0, acc); break;
        HSC_TILE_DISK(1)
        HSC_TILE_DISK(2)
        HSC_TILE_DISK(4)
        HSC_TILE_DISK(5)
        HSC_TILE_DISK(8)
        HSC_TILE_DISK(9)
        HSC_TILE_DISK(10)
        HSC_TILE_DISK(13)
        HSC_TILE_DISK(16)
        HSC_TILE_DISK(17)
        HSC_TILE_DISK(18)
        HSC_TILE_DISK(20)
#undef HSC_TILE_DISK
    default: break;  // 0: no disk
    }
    // the shell: per row the K - |disk| smallest (e, index); the table lists
    // its entries by increasing index, so the first of equal e is the smaller
    const int need = a.K - a.disk;
    int o[kTileShell];
#pragma unroll
    for (int i = 0; i < kTileShell; ++i) {
        const char2 d = c_knn_tab[a.disk + min(i, a.shell - 1)];
        o[i] = HSC_IN_BOUNDS(abs(d.x) <= rad && abs(d.y) <= rad, f.ctl) ? d.x * W + d.y : 0;
    }
    bool bad = false;
    unsigned ord[kV];
#pragma unroll
    for (int v = 0; v < kV; ++v) {
        const float *__restrict__ Ic = f.I + (q0 + v * W);
        const float Ip = __ldg(Ic);
        bad |= !isfinite(Ip);
        float e[kTileShell];
#pragma unroll
        for (int i = 0; i < kTileShell; ++i) {
            const float d = __fsub_rn(Ip, __ldg(Ic + o[i]));
            e[i] = __fmul_rn(d, d);
        }
        ord[v] = shell_order(e, a.shell, need);
    }
    if (bad) atomicOr(&f.ctl->status, ST_NONFINITE_MAP);
#pragma unroll 1
    for (int n = 0; n < need; ++n) {  // nearest first
        Acc<KC, kP4> x[kV];
#pragma unroll
        for (int v = 0; v < kV; ++v) {
            const unsigned i = (ord[v] >> (4 * n)) & 15u;
            const int dr = (int)((a.shell_r >> (4 * i)) & 15u) - 4;
            const int dc = (int)((a.shell_c >> (4 * i)) & 15u) - 4;
            if (!HSC_IN_BOUNDS(i < (unsigned)a.shell && abs(dr) <= rad && abs(dc) <= rad, f.ctl)) {
                x[v].zero();
                continue;
            }
            x[v].load(Acc<KC, kP4>::at(f, q0 + (v + dr) * W + dc), 0);
        }
#pragma unroll
        for (int v = 0; v < kV; ++v) acc[v].add(x[v]);
    }
    if (on && ok) {
#pragma unroll
        for (int v = 0; v < kV; ++v) {
            if (v < vfirst) continue;
            float out[KC];
            acc[v].get(out);
            write_pixel(out, a.K, f.N, (long)(r0 + v) * W + c, f.O, f.labels);
        }
    }
    return ok;
}

template <int KC, bool kP4>
__global__ void __launch_bounds__(32 * kKnnTileMaxWarps)
knn_tile_kernel(const __grid_constant__ TileArgs a)
{
    extern __shared__ float sm[];
    pdl_wait();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    TileFrame f = a.frame;
    int cta = blockIdx.x, frame = 0;
    if (a.frames) {  // a stage-major batch: the frame whose CTA range holds this CTA
        cta += a.cta_base;
        int lo = 0, hi = a.n_frames - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (a.frames[mid].knn_cta0 <= cta) lo = mid;
            else hi = mid - 1;
        }
        frame = lo;
        const BatchFrame &fr = a.frames[lo];
        f.I = fr.I;
        f.P = fr.P;
        f.P4 = fr.P4;
        f.O = fr.O;
        f.labels = fr.labels;
        f.ctl = fr.ctl;
        f.H = fr.H;
        f.W = fr.W;
        f.N = fr.N;
        cta -= fr.knn_cta0;
    }
    const Buf buf = {(uint32_t)__cvta_generic_to_shared(sm) + warp * (uint32_t)buf_bytes(kTileCap) +
                     4u * lane};
    const float l2 = a.lam * a.lam;
    const int K = a.K, W = f.W;
    const TileGeom g = tile_geom(f.H, f.W, a.rad, a.cut, nw);
    unsigned evals = 0, redo = 0;
    auto leave = [&](int p, bool far) {  // to the second pass
        ++redo;
        f.labels[p] = far ? kRedoFarLabel : kRedoLabel;
        if (a.frames) {
            const unsigned i = atomicAdd(&a.frames[0].ctl->knn_redo_list, 1u);
            if (i < a.redo_cap) a.redo_list[i] = make_int2(far ? ~frame : frame, p);
        }
    };
    // the pixels that box_pixel takes: this lane's border pixel, or the rows
    // the tile path left (rows first .. first + passes - 1 below p0)
    int p0 = -1, passes = 0;
    if (cta < g.border_ctas) {
        const long i = (long)cta * blockDim.x + threadIdx.x;
        if (i < g.border_px) {
            int r, c;
            border_pixel(g, f.H, W, a.rad, i, r, c);
            if (HSC_IN_BOUNDS(r >= 0 && r < f.H && c >= 0 && c < W, f.ctl)) p0 = r * W + c;
        }
        passes = 1;
    } else {
        const int t = (cta - g.border_ctas) * nw + warp;
        if (t < g.tiles) {  // warp-uniform
            const int tc = t / g.row_groups, gr = t - tc * g.row_groups;
            int r0 = a.rad + gr * kV;
            const int last = f.H - a.rad - kV;
            const int vfirst = r0 > last ? r0 - last : 0;
            r0 -= vfirst;
            const int c0 = tc * 32, c = c0 + lane;
            const bool on = c >= a.rad && c < W - a.rad;
            const bool fast = tile_fast<KC, kP4>(f, a, r0, c0, lane, on, vfirst, l2);
            if (on && fast) evals += (unsigned)((kV - vfirst) * a.shell);
            if (on && !fast) p0 = (r0 + vfirst) * W + c;
            passes = __any_sync(0xffffffffu, p0 >= 0) ? kV - vfirst : 0;
        }
    }
#pragma unroll 1
    for (int v = 0; v < passes; ++v) {
        const int p = p0 >= 0 ? p0 + v * W : -1;
        const unsigned ev = box_pixel<KC, kP4>(f, p, K, a.R, l2, buf, kTileCap);
        if (ev < kLeftKeys) evals += ev;
        else leave(p, ev == kLeftFar);
    }
    // the counters: keys formed, pixels left to the second pass
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        evals += __shfl_xor_sync(0xffffffffu, evals, o);
        redo += __shfl_xor_sync(0xffffffffu, redo, o);
    }
    if (lane == 0 && evals) atomicAdd(&f.ctl->knn_evals, (unsigned long long)evals);
    if (lane == 0 && redo && !a.frames) atomicAdd(&f.ctl->knn_redo, redo);
}

template <int KC, bool kP4>
cudaError_t launch_tile_kc(const TileArgs &a, int ctas, int warps, cudaStream_t st)
{
    auto kern = knn_tile_kernel<KC, kP4>;
    const size_t smem = buf_bytes(kTileCap) * (size_t)warps;
    if (smem > 48 * 1024)
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    return launch_pdl(kern, dim3((unsigned)ctas), dim3(32 * warps), smem, st, a);
}

}  // namespace
}  // namespace hsc
