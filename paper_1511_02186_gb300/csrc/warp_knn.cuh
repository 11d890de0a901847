// The one-warp-per-query phase-1 scans (FP32 in f32_device.cuh, FP64 in kernels_f64.cu): the walk
// over the dataset's box hierarchy and the warp's candidate buffer.
//
// The dataset's curve-ordered points are grouped three ways, each with a bounding box: 32-tile
// super-tiles (16,384 points), 512-point tiles and 64-point sub-tiles. A warp first descends to
// the sub-tile nearest its query (smallest bound, then nearest centre), takes the k-th of its 64
// distances as an upper bound T of the query's k-th distance, and then visits every other
// sub-tile whose box comes within T, super-tiles and tiles nearest first. A visited point within T
// goes into a small buffer in shared memory; nothing is kept sorted while points arrive. Only
// when the buffer would overflow, after a tile that brought many, and at the end, is it cut to the
// k nearest, which also lowers T.
//
// The scan is latency bound when a call has few queries (one chain of dependent loads per
// level) and issue bound when it has many. Before, a list was kept sorted across the lanes with
// every arriving candidate, every next box was picked by a 64-bit minimum across the lanes, and
// FP64 formed and compared every distance on the FP64 pipe. Phase 1 before / now, us (the points
// along a Hilbert curve since): FP32 1,024 x 1,024 62 / 11, 257 x 300,007 209 / 15, 8,192 x 1M
// 304 / 27, 32,768 x 1M 860 / 78; FP64 1,024 x 1,024 51 / 18, 8,191 x 131,072 393 / 49, 16,384 x
// 262,144 797 / 80.
#pragma once

#include <math_constants.h>

#include "aidw_internal.cuh"

namespace aidw {

constexpr unsigned kFullMask = 0xffffffffu;
constexpr int kWarpBuffer = 64;  // candidates a warp's buffer holds (at least k + 32)
constexpr int kWarpSettle = 16;  // candidates beyond k at which a finished tile cuts the buffer
static_assert(kWarpBuffer >= AIDW_MAX_K + 32, "a cut buffer takes a whole step's candidates");

constexpr float kBoundShrink = 1.0f - 9.5367431640625e-07f;  // 1 - 2^-20, box bounds

// Squared-distance lower bound from (qx, qy) to a box (xmin, ymin, xmax, ymax), shrunk by 2^-20
// for rounding; +inf for an empty box.
__device__ __forceinline__ float box_bound(float qx, float qy, float4 b)
{
    const float dx = fmaxf(0.0f, fmaxf(b.x - qx, qx - b.z));
    const float dy = fmaxf(0.0f, fmaxf(b.y - qy, qy - b.w));
    return __fmul_rn(__fmaf_rn(dx, dx, __fmul_rn(dy, dy)), kBoundShrink);
}

// Squared distance to a box's centre (orders boxes of equal bound only).
__device__ __forceinline__ float box_centre(float qx, float qy, float4 b)
{
    const float cx = 0.5f * (b.x + b.z) - qx, cy = 0.5f * (b.y + b.w) - qy;
    return fmaf(cx, cx, cy * cy);
}

// The lane whose box is nearest: smallest bound, then smallest centre distance, then lowest lane.
// `lb` (>= 0 or +inf; a lane without a box passes ~0 as `bits`) orders by its bits.
__device__ __forceinline__ int nearest_lane(unsigned bits, float centre, unsigned &least)
{
    least = __reduce_min_sync(kFullMask, bits);
    const unsigned tie = __ballot_sync(kFullMask, bits == least);
    if (__popc(tie) == 1)
        return __ffs(tie) - 1;
    const unsigned cb = bits == least ? __float_as_uint(centre) : 0xffffffffu;
    const unsigned cl = __reduce_min_sync(kFullMask, cb);
    return __ffs(__ballot_sync(kFullMask, cb == cl)) - 1;
}

// A visitor V provides float qx, qy, thr (a box farther than thr holds nothing that matters;
// warp-uniform), bool usable(float bound, float4 box) (whether a box may hold points at all),
// and void scan(int64_t p, float4 a, float4 b) for the stored points p + lane (a) and
// p + 32 + lane (b), which may lower thr; cut() lowers thr from what has been scanned, settle()
// does where enough has come in.
template <class V>
__device__ __forceinline__ void warp_walk(const DatasetDev &ds, V &v)
{
    constexpr int S = kTileF32Knn / kSubTile;  // 8 sub-tiles per tile
    const int lane = threadIdx.x & 31;
    const int64_t ntiles = ds.n_pad / kTileF32Knn;
    const int64_t nsuper = (ntiles + kSuperTiles - 1) / kSuperTiles;
    const auto bits_of = [&](float4 b) {
        const float lb = box_bound(v.qx, v.qy, b);
        return v.usable(lb, b) ? __float_as_uint(lb) : 0xffffffffu;
    };

    // The nearest sub-tile (-1 if no box on the way to it is usable).
    int64_t seed = -1;
    {
        unsigned best = 0xffffffffu;
        float best_c = CUDART_INF_F;
        int64_t s0 = -1;
        for (int64_t g = 0; g < nsuper; g += 32) {
            unsigned bits = 0xffffffffu, least;
            float c = CUDART_INF_F;
            if (g + lane < nsuper) {
                const float4 b = ds.super_box[g + lane];
                bits = bits_of(b);
                c = box_centre(v.qx, v.qy, b);
            }
            const int j = nearest_lane(bits, c, least);
            const float cj = __shfl_sync(kFullMask, c, j);
            if (least != 0xffffffffu && (least < best || (least == best && cj < best_c))) {
                best = least;
                best_c = cj;
                s0 = g + j;
            }
        }
        if (s0 >= 0) {
            const int64_t t = s0 * kSuperTiles + lane;
            unsigned bits = 0xffffffffu, least;
            float c = CUDART_INF_F;
            if (t < ntiles) {
                const float4 b = ds.tile_box[t];
                bits = bits_of(b);
                c = box_centre(v.qx, v.qy, b);
            }
            const int64_t t0 = s0 * kSuperTiles + nearest_lane(bits, c, least);
            if (least != 0xffffffffu) {
                bits = 0xffffffffu;
                if (lane < S) {
                    const float4 b = ds.sub_box[t0 * S + lane];
                    bits = bits_of(b);
                    c = box_centre(v.qx, v.qy, b);
                }
                const int j = nearest_lane(bits, c, least);
                if (least != 0xffffffffu)
                    seed = t0 * S + j;
            }
        }
    }
    if (seed >= 0) {
        const int64_t p = seed * kSubTile;
        v.scan(p, ds.nxy2[p + lane], ds.nxy2[p + 32 + lane]);
        v.cut();
    }

    // Everything else within thr.
    for (int64_t g = 0; g < nsuper; g += 32) {
        unsigned sb = g + lane < nsuper ? bits_of(ds.super_box[g + lane]) : 0xffffffffu;
        for (;;) {
            const unsigned ms = __reduce_min_sync(kFullMask, sb);
            if (ms == 0xffffffffu || __uint_as_float(ms) > v.thr)
                break;
            const int js = __ffs(__ballot_sync(kFullMask, sb == ms)) - 1;
            if (lane == js)
                sb = 0xffffffffu;
            const int64_t t0 = (g + js) * kSuperTiles;
            unsigned tb = t0 + lane < ntiles ? bits_of(ds.tile_box[t0 + lane]) : 0xffffffffu;
            for (;;) {
                const unsigned mt = __reduce_min_sync(kFullMask, tb);
                if (mt == 0xffffffffu || __uint_as_float(mt) > v.thr)
                    break;
                const int jt = __ffs(__ballot_sync(kFullMask, tb == mt)) - 1;
                if (lane == jt)
                    tb = 0xffffffffu;
                const int64_t u0 = (t0 + jt) * S;
                unsigned ub = lane < S ? bits_of(ds.sub_box[u0 + lane]) : 0xffffffffu;
                if (u0 + lane == seed)
                    ub = 0xffffffffu;
                // Sub-tiles nearest first; the next one's points are loaded before the current
                // one's are looked at.
                float4 a, b;
                const auto next = [&]() -> int64_t {
                    const unsigned mu = __reduce_min_sync(kFullMask, ub);
                    if (mu == 0xffffffffu || __uint_as_float(mu) > v.thr)
                        return -1;
                    const int ju = __ffs(__ballot_sync(kFullMask, ub == mu)) - 1;
                    if (lane == ju)
                        ub = 0xffffffffu;
                    const int64_t p = (u0 + ju) * kSubTile;
                    a = ds.nxy2[p + lane];
                    b = ds.nxy2[p + 32 + lane];
                    return p;
                };
                int64_t p = next();
                while (p >= 0) {
                    const float4 ca = a, cb = b;
                    const int64_t cp = p;
                    p = next();
                    v.scan(cp, ca, cb);
                }
                v.settle();
            }
        }
    }
}

}  // namespace aidw
