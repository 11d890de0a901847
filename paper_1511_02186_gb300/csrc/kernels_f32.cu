// FP32 ("F32C") per-call kernels of the AIDW hot path for sm_103a.
//
//   f32_knn_kernel      grid (query blocks, data splits): phase-1 unit per CTA (neighbour lists)
//   f32_select_kernel   one thread per query: split merge, Eq. 2-6 -> phase-2 parameters
//   f32_weights_kernel  grid (query blocks, data splits): phase-2 unit per CTA (weighted sums)
//   f32_finalize_kernel one thread per query: split merge, Eq. 1 ratio in FP64
// The unit bodies live in f32_device.cuh and are shared with the persistent batched kernel.
#include <algorithm>

#include "f32_device.cuh"

namespace aidw {
namespace {

using namespace f32dev;

// Phase 2 with point groups: the CTA's four warps each take a quarter of every tile's chunks for
// the same 64 queries (2 per lane, whatever the shape's queries per thread).
constexpr int kQueriesPG = 2;

// The phase-1 kernel zeroes the power classes' counters, which the selection after it counts in.
__device__ __forceinline__ void zero_classes(uint32_t *cnt)
{
    if (cnt && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x < kClasses)
        cnt[threadIdx.x] = 0;
}

template <int KP, int Q, bool IDX>
__global__ void __launch_bounds__(kThreads)
f32_knn_kernel(DatasetDev ds, int64_t m, PassPlan pp, const float *__restrict__ qx,
               const float *__restrict__ qy, int k, float *__restrict__ part_d2,
               int32_t *__restrict__ part_idx, int *__restrict__ err, uint32_t *cls_cnt)
{
    __shared__ __align__(128) float4 tile[2][kTileF32Knn];
    __shared__ __align__(8) uint64_t bar[2];
    extern __shared__ int32_t idx_smem[];  // [Q][KP][kThreads] when IDX
    zero_classes(cls_cnt);
    init_tile_barriers(bar);
    TileSeq ts{bar, 0u};
    const int s = blockIdx.y;
    const int64_t p_begin = static_cast<int64_t>(s) * pp.split_len;
    const int64_t p_end = min(p_begin + pp.split_len, ds.n_pad);
    knn_unit<KP, Q, IDX>(ds, m, static_cast<int64_t>(blockIdx.x) * pp.q_per_block, p_begin,
                         p_end, qx, qy, k, s, part_d2, part_idx, err, tile, ts, idx_smem);
}

// KP > 0: one split, k <= KP.
template <int KP>
__global__ void __launch_bounds__(kSelectThreads)
f32_select_kernel(int64_t m, int S, int k, double r_exp, AlphaMap am,
                  const float *__restrict__ part_d2, const int32_t *__restrict__ part_idx,
                  QParamF32 *__restrict__ qp, float *__restrict__ out_alpha,
                  int32_t *__restrict__ out_knn, const uint32_t *__restrict__ perm,
                  const float *__restrict__ qx, const float *__restrict__ qy, ClassOrder co)
{
    grid_wait();
    const int64_t q = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (q < m) {
        if constexpr (KP > 0)
            select_query_one<KP>(q, m, k, r_exp, am, part_d2, part_idx, qp, out_alpha, out_knn,
                                 perm);
        else
            select_query(q, m, S, k, r_exp, am, part_d2, part_idx, qp, out_alpha, out_knn, perm);
    }
    if (!co.cnt)
        return;
    // Each query to the next place of its class (a warp's queries stay together).
    if (q < m) {
        const QParamF32 p = qp[q];
        const int cls = power_class(p, co, co.pow_b);
        const int64_t o = static_cast<int64_t>(cls) * m + class_place(co.cnt, cls);
        co.qx[o] = __ldcg(qx + q);
        co.qy[o] = __ldcg(qy + q);
        co.qp[o] = p;
        co.id[o] = perm ? __ldcg(perm + q) : static_cast<uint32_t>(q);
    }
}

// Phase 1 with one warp per query (warp_knn), in the caller's order: each query's k nearest
// squared distances (and, with IDX, stored positions mapped to caller indices) as one split's
// lists [k][m], for the selection kernel, which amortises its FP64 work over a thread per query.
template <bool IDX>
__global__ void __launch_bounds__(kThreads)
f32_knn_warp_kernel(DatasetDev ds, int64_t m, const float *qx, const float *qy, int k,
                    float *__restrict__ part_d2, int32_t *__restrict__ part_idx,
                    uint32_t *cls_cnt)
{
    grid_trigger();
    grid_wait();
    zero_classes(cls_cnt);
    constexpr int W = kThreads / 32;
    __shared__ __align__(16) float bd[W][kWarpBuffer];
    __shared__ int32_t bi[W][IDX ? kWarpBuffer : 1];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t nwarps = static_cast<int64_t>(gridDim.x) * W;
    for (int64_t q = static_cast<int64_t>(blockIdx.x) * W + w; q < m; q += nwarps) {
        const WarpEntry e = warp_knn<IDX>(ds, qx[q], qy[q], k, bd[w], bi[w]);
        if (lane < k) {
            part_d2[static_cast<int64_t>(lane) * m + q] = e.d;
            if (IDX)
                part_idx[static_cast<int64_t>(lane) * m + q] = e.i >= 0 ? ds.orig[e.i] : -1;
        }
    }
}

template <int KP, int Q, bool IDX>
__global__ void __launch_bounds__(kThreads)
f32_knn_cull_kernel(DatasetDev ds, int64_t m, int qpb, int ntiles, int ntiles_p2,
                    const float *__restrict__ sqx, const float *__restrict__ sqy, int k,
                    float *__restrict__ part_d2, int32_t *__restrict__ part_idx,
                    int *__restrict__ err, uint32_t *cls_cnt)
{
    zero_classes(cls_cnt);
    extern __shared__ unsigned long long order[];  // [ntiles_p2], then the index lists if IDX
    __shared__ __align__(128) float4 tile[2][kTileF32Knn];
    __shared__ __align__(8) uint64_t bar[2];
    __shared__ CullShared cs;
    init_tile_barriers(bar);
    TileSeq ts{bar, 0u};
    knn_cull_unit<KP, Q, IDX>(ds, m, static_cast<int64_t>(blockIdx.x) * qpb, ntiles, ntiles_p2,
                              sqx, sqy, k, part_d2, part_idx, err, tile, ts, order,
                              reinterpret_cast<int32_t *>(order + ntiles_p2), cs);
}

template <int Q, int TW, int PG>
__global__ void __launch_bounds__(kThreads)
f32_weights_kernel(DatasetDev ds, int64_t m, PassPlan pp, const float *__restrict__ qx,
                   const float *__restrict__ qy, const QParamF32 *__restrict__ qp,
                   float *__restrict__ part_sum, int *__restrict__ err)
{
    __shared__ __align__(128) float4 txy[2][TW];
    __shared__ __align__(128) float2 tz[2][TW];
    __shared__ __align__(8) uint64_t bar[2];
    init_tile_barriers(bar);
    TileSeq ts{bar, 0u};
    const int s = blockIdx.y;
    const int64_t p_begin = static_cast<int64_t>(s) * pp.split_len;
    const int64_t p_end = min(p_begin + pp.split_len, ds.n_pad);
    grid_trigger();
    grid_wait();
    const int64_t qbase = static_cast<int64_t>(blockIdx.x) * pp.q_per_block;
    weights_unit<Q, TW, PG>(ds, unit_queries(qx, qy, qp, m, qbase, pp.q_per_block), p_begin,
                            p_end, s, part_sum, err, txy, tz, ts);
}

// Phase 2 over the power classes: a block serves 256 queries of one class, with the class's loop.
// The grid has a block for every 256 queries and one more per further class; the general class,
// the slowest, comes first. Which loop a query takes depends on its own power and nearest
// distance only. The shape is fixed (2 queries per thread, 512-point tiles).
template <int POW>
__device__ __forceinline__ void weights_class_unit(const DatasetDev &ds, const UnitQueries &uq,
                                                   int64_t p_begin, int64_t p_end, int s,
                                                   float *part_sum, int *err,
                                                   float4 (*txy)[512], float2 (*tz)[512],
                                                   TileSeq &ts)
{
    weights_unit<2, 512, 1, POW>(ds, uq, p_begin, p_end, s, part_sum, err, txy, tz, ts);
}

__global__ void __launch_bounds__(kThreads, 8)
f32_weights_class_kernel(DatasetDev ds, int64_t m, PassPlan pp, ClassOrder co,
                         float *__restrict__ part_sum, int *__restrict__ err)
{
    __shared__ __align__(128) float4 txy[2][512];
    __shared__ __align__(128) float2 tz[2][512];
    __shared__ __align__(8) uint64_t bar[2];
    grid_trigger();
    grid_wait();
    constexpr int kB = 2 * kThreads;
    const int order[kClasses] = {kClassG, kClassA, kClassB};
    int64_t u = blockIdx.x, col = 0;
    int cls = -1;
    int64_t n = 0;
#pragma unroll
    for (int i = 0; i < kClasses; ++i) {
        const int64_t c = __ldcg(co.cnt + order[i]);
        if (cls < 0) {
            const int64_t blocks = (c + kB - 1) / kB;
            if (u < blocks) {
                cls = order[i];
                n = c;
            } else {
                u -= blocks;
                col += c;
            }
        }
    }
    if (cls < 0)
        return;
    init_tile_barriers(bar);
    TileSeq ts{bar, 0u};
    const int s = blockIdx.y;
    const int64_t p_begin = static_cast<int64_t>(s) * pp.split_len;
    const int64_t p_end = min(p_begin + pp.split_len, ds.n_pad);
    const UnitQueries uq{co.qx, co.qy, co.qp, cls * m + u * kB,
                         min(static_cast<int64_t>(kB), n - u * kB), col + u * kB, m};
    const int pow = cls == kClassA ? co.pow_a : (cls == kClassB ? co.pow_b : 0);
    switch (pow) {
    case 1:
        weights_class_unit<1>(ds, uq, p_begin, p_end, s, part_sum, err, txy, tz, ts);
        break;
    case 2:
        weights_class_unit<2>(ds, uq, p_begin, p_end, s, part_sum, err, txy, tz, ts);
        break;
    case 3:
        weights_class_unit<3>(ds, uq, p_begin, p_end, s, part_sum, err, txy, tz, ts);
        break;
    case 4:
        weights_class_unit<4>(ds, uq, p_begin, p_end, s, part_sum, err, txy, tz, ts);
        break;
    case 5:
        weights_class_unit<5>(ds, uq, p_begin, p_end, s, part_sum, err, txy, tz, ts);
        break;
    default:
        weights_class_unit<0>(ds, uq, p_begin, p_end, s, part_sum, err, txy, tz, ts);
        break;
    }
}

// R threads per query (a block serves 256 / R queries): each sums every R-th split's partial
// sums, the block adds the R sums up. One thread per query leaves a call with few queries and
// many splits waiting on a chain of loads.
template <int R>
__global__ void __launch_bounds__(256)
f32_finalize_kernel(int64_t m, int S, const float *__restrict__ part_sum,
                    float *__restrict__ out, const uint32_t *__restrict__ perm, ClassOrder co,
                    float z_unscale)
{
    grid_trigger();
    grid_wait();
    constexpr int C = 256 / R;
    const int col = threadIdx.x % C, r = threadIdx.x / C;
    const int64_t q = static_cast<int64_t>(blockIdx.x) * C + col;
    double W = 0.0, WZ = 0.0;
    if (q < m)
        merge_splits(q, m, r, R, S, part_sum, W, WZ);
    if constexpr (R > 1) {
        __shared__ double2 sum[R][C];
        sum[r][col] = make_double2(W, WZ);
        __syncthreads();
        if (r > 0)
            return;
#pragma unroll
        for (int i = 1; i < R; ++i) {
            W += sum[i][col].x;
            WZ += sum[i][col].y;
        }
    }
    if (q >= m)
        return;
    int64_t o = perm ? static_cast<int64_t>(__ldcg(perm + q)) : q;
    if (co.cnt) {
        // Column q of the class order: the general class, class A, class B.
        const int64_t ng = __ldcg(co.cnt + kClassG), na = __ldcg(co.cnt + kClassA);
        o = __ldcg(co.id + (q < ng        ? kClassG * m + q
                            : q < ng + na ? kClassA * m + (q - ng)
                                          : kClassB * m + (q - ng - na)));
    }
    out[o] = static_cast<float>(WZ / W * z_unscale);
}

template <int KP, int Q, bool IDX>
cudaError_t launch_cull_t(const DatasetDev &ds, const Plan &pl, const float *sqx,
                          const float *sqy, int k, const Scratch &sc, int *err, cudaStream_t st)
{
    const int ntiles = static_cast<int>(ds.n_pad / kTileF32Knn);
    int p2 = 1;
    while (p2 < ntiles)
        p2 <<= 1;
    const size_t dyn = sizeof(unsigned long long) * p2 +
                       (IDX ? sizeof(int32_t) * Q * KP * kThreads : 0);
    auto fn = f32_knn_cull_kernel<KP, Q, IDX>;
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         static_cast<int>(dyn));
    if (e != cudaSuccess)
        return e;
    fn<<<pl.knn.qblocks, kThreads, dyn, st>>>(ds, pl.m, pl.knn.q_per_block, ntiles, p2, sqx,
                                              sqy, k, static_cast<float *>(sc.part_d2),
                                              sc.part_idx, err, sc.cls.cnt);
    return cudaGetLastError();
}

template <int KP, bool IDX>
cudaError_t launch_knn_t(const DatasetDev &ds, const Plan &pl, const float *qx,
                         const float *qy, int k, const Scratch &sc, int *err, cudaStream_t st)
{
    constexpr int Q = knn_q<KP>();
    const size_t dyn = IDX ? sizeof(int32_t) * Q * KP * kThreads : 0;
    auto fn = f32_knn_kernel<KP, Q, IDX>;
    if (dyn > 0) {
        cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             static_cast<int>(dyn));
        if (e != cudaSuccess)
            return e;
    }
    dim3 grid(pl.knn.qblocks, pl.knn.splits);
    fn<<<grid, kThreads, dyn, st>>>(ds, pl.m, pl.knn, qx, qy, k,
                                    static_cast<float *>(sc.part_d2), sc.part_idx, err,
                                    sc.cls.cnt);
    return cudaGetLastError();
}

template <int KP>
int knn_slots_t(bool with_idx)
{
    constexpr int Q = knn_q<KP>();
    int n = 0;
    if (with_idx) {
        const size_t dyn = sizeof(int32_t) * Q * KP * kThreads;
        cudaFuncSetAttribute(f32_knn_kernel<KP, Q, true>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(dyn));
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, f32_knn_kernel<KP, Q, true>, kThreads,
                                                      dyn);
    } else {
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, f32_knn_kernel<KP, Q, false>,
                                                      kThreads, 0);
    }
    return n > 0 ? n : 1;
}

}  // namespace

int f32_list_length(int k, int kp_min)
{
    return f32dev::kp_for(k, kp_min);
}

int f32_knn_queries_per_block(int kp)
{
    return kThreads * (kp <= 16 ? 4 : 2);
}

int f32_w_queries_per_block(int qw, int pg)
{
    return pg > 1 ? kThreads * kQueriesPG / pg : kThreads * qw;
}

int f32_knn_slots_per_sm(int kp, bool with_idx)
{
    switch (kp) {
    case 8: return knn_slots_t<8>(with_idx);
    case 12: return knn_slots_t<12>(with_idx);
    case 16: return knn_slots_t<16>(with_idx);
    default: return knn_slots_t<32>(with_idx);
    }
}

namespace {

using WeightsKernel = void (*)(DatasetDev, int64_t, PassPlan, const float *, const float *,
                               const QParamF32 *, float *, int *);

WeightsKernel weights_kernel_for(int qw, int tw, int pg)
{
    if (pg > 1)
        return f32_weights_kernel<kQueriesPG, 512, kPointGroups>;
    if (tw == 256)
        return qw == 2 ? f32_weights_kernel<2, 256, 1>
                       : (qw == 8 ? f32_weights_kernel<8, 256, 1> : f32_weights_kernel<4, 256, 1>);
    return qw == 2 ? f32_weights_kernel<2, 512, 1>
                   : (qw == 8 ? f32_weights_kernel<8, 512, 1> : f32_weights_kernel<4, 512, 1>);
}

}  // namespace

cudaError_t launch_f32_knn(const DatasetDev &ds, const Plan &pl, const float *qx,
                           const float *qy, int k, const Scratch &sc, int *err,
                           cudaStream_t st)
{
    switch (pl.kp) {
    case 8:
        return pl.with_idx ? launch_knn_t<8, true>(ds, pl, qx, qy, k, sc, err, st)
                           : launch_knn_t<8, false>(ds, pl, qx, qy, k, sc, err, st);
    case 12:
        return pl.with_idx ? launch_knn_t<12, true>(ds, pl, qx, qy, k, sc, err, st)
                           : launch_knn_t<12, false>(ds, pl, qx, qy, k, sc, err, st);
    case 16:
        return pl.with_idx ? launch_knn_t<16, true>(ds, pl, qx, qy, k, sc, err, st)
                           : launch_knn_t<16, false>(ds, pl, qx, qy, k, sc, err, st);
    default:
        return pl.with_idx ? launch_knn_t<32, true>(ds, pl, qx, qy, k, sc, err, st)
                           : launch_knn_t<32, false>(ds, pl, qx, qy, k, sc, err, st);
    }
}

cudaError_t launch_f32_select(const Plan &pl, int k, double r_exp, const AlphaMap &am,
                              const Scratch &sc, float *out_alpha, int32_t *out_knn,
                              cudaStream_t st, const float *qx, const float *qy,
                              const uint32_t *perm)
{
    const int64_t blocks = (pl.m + kSelectThreads - 1) / kSelectThreads;
    auto fn = pl.knn.splits > 1 ? f32_select_kernel<0>
              : k <= 16         ? f32_select_kernel<16>
                                : f32_select_kernel<32>;
    return launch_chained(fn, dim3(static_cast<unsigned>(blocks)), kSelectThreads, 0, st,
                          pl.m, pl.knn.splits, k, r_exp, am,
                          static_cast<const float *>(sc.part_d2),
                          pl.with_idx ? sc.part_idx : nullptr,
                          static_cast<QParamF32 *>(sc.qparam), out_alpha, out_knn, perm, qx, qy, sc.cls);
}

cudaError_t launch_f32_knn_warp(const DatasetDev &ds, int64_t m, const float *qx,
                                const float *qy, int k, const Scratch &sc, int sm_count,
                                cudaStream_t st)
{
    constexpr int W = kThreads / 32;
    const int64_t want = (m + W - 1) / W;
    const int64_t cap = static_cast<int64_t>(sm_count) * 16;
    const unsigned grid = static_cast<unsigned>(std::max<int64_t>(1, std::min(want, cap)));
    auto fn = sc.part_idx ? f32_knn_warp_kernel<true> : f32_knn_warp_kernel<false>;
    return launch_chained(fn, dim3(grid), kThreads, 0, st, ds, m, qx, qy, k,
                          static_cast<float *>(sc.part_d2), sc.part_idx, sc.cls.cnt);
}

cudaError_t launch_f32_knn_cull(const DatasetDev &ds, const Plan &pl, const float *sqx,
                                const float *sqy, int k, const Scratch &sc, int *err,
                                cudaStream_t st)
{
    const bool q2 = pl.kq == 2;
#define AIDW_CULL(KP, Q)                                                                       \
    return pl.with_idx ? launch_cull_t<KP, Q, true>(ds, pl, sqx, sqy, k, sc, err, st)         \
                       : launch_cull_t<KP, Q, false>(ds, pl, sqx, sqy, k, sc, err, st)
    switch (pl.kp) {
    case 8:
        if (q2)
            AIDW_CULL(8, 2);
        AIDW_CULL(8, 4);
    case 12:
        if (q2)
            AIDW_CULL(12, 2);
        AIDW_CULL(12, 4);
    case 16:
        if (q2)
            AIDW_CULL(16, 2);
        AIDW_CULL(16, 4);
    default:
        AIDW_CULL(32, 2);
    }
#undef AIDW_CULL
}

cudaError_t launch_f32_weights(const DatasetDev &ds, const Plan &pl, const float *qx,
                               const float *qy, const Scratch &sc, int *err, cudaStream_t st)
{
    if (sc.cls.cnt) {
        const dim3 grid(pl.w.qblocks + kClasses - 1, pl.w.splits);
        return launch_chained(f32_weights_class_kernel, grid, kThreads, 0, st, ds, pl.m, pl.w,
                              sc.cls, static_cast<float *>(sc.part_sum), err);
    }
    dim3 grid(pl.w.qblocks, pl.w.splits);
    const WeightsKernel fn = weights_kernel_for(pl.qw, pl.tw, pl.pg);
    return launch_chained(fn, grid, kThreads, 0, st, ds, pl.m, pl.w, qx, qy,
                          static_cast<const QParamF32 *>(sc.qparam),
                          static_cast<float *>(sc.part_sum), err);
}

cudaError_t launch_f32_finalize(const DatasetDev &ds, const Plan &pl, const Scratch &sc,
                                float *out, cudaStream_t st, const uint32_t *perm)
{
    const int R = finalize_threads(pl.w.splits, pl.m);
    const unsigned blocks = static_cast<unsigned>((pl.m * R + 255) / 256);
    auto fn = R == 32 ? f32_finalize_kernel<32>
                      : (R == 8 ? f32_finalize_kernel<8> : f32_finalize_kernel<1>);
    return launch_chained(fn, dim3(blocks), 256, 0, st, pl.m, pl.w.splits,
                          static_cast<const float *>(sc.part_sum), out, perm, sc.cls,
                          ds.z_unscale);
}

}  // namespace aidw
