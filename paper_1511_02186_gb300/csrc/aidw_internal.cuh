// Internal declarations shared by the library's translation units: device-side dataset view,
// launch plans, Blackwell TMA/mbarrier helpers and the kernel launchers.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/aidw.h"

namespace aidw {

// Data points per shared-memory tile. Dataset arrays are padded to a multiple of
// kPadPoints with sentinel points at +infinity (value 0), which never enter a neighbour list
// and get weight 0, so every tile is full and every TMA copy has a whole-tile size.
constexpr int kTileF32Knn = 512;   // float4 (-x, -x, -y, -y): 8 KiB per buffer
constexpr int kTileF32W = 512;     // float4 (-x, -x, -y, -y) + float2 (z, z): 12 KiB per buffer
constexpr int kTileF64Knn = 512;   // double2 (x, y): 8 KiB per buffer
constexpr int kTileF64W = 512;     // double2 + double: 12 KiB per buffer
constexpr int kPadPoints = 2048;   // common multiple of every tile and split granule
constexpr int kSubTile = 64;       // points per sub-tile box (pruned phase 1)
constexpr int kSuperTiles = 32;    // tiles per super-tile box (the per-query phase 1)

// Added under the square of distances: it is absorbed (below half an ulp) for any distance
// above ~1e-15 of unit scale, and turns an exact coincidence (d2 == 0) into d2 == kEps so
// that log2 stays finite. FLT_MIN / DBL_MIN, the smallest normal numbers.
constexpr float kEpsF32 = 1.17549435e-38f;
constexpr double kEpsF64 = 2.2250738585072014e-308;
// Power scale used for coincident queries: w = 2^(kCoincScale (L1 - log2 d2)) is exactly 1 on
// a coincident point (d2 == eps) and underflows to 0 everywhere else.
constexpr float kCoincScaleF32 = 1.2676506e30f;  // 2^100
constexpr double kCoincScaleF64 = 8.452712498170644e270;  // 2^900 (the paper's designs)
constexpr double kCoincScaleDf = 1.2676506002282294e30;   // 2^100 (AIDW_F64 and AIDW_F64X)

// Bounded waits: an mbarrier wait gives up after this many polls and raises the error word;
// a wait on another CTA's counter gives up after kMaxWaitPolls polls of at least 256 ns
// (tens of seconds at most).
constexpr uint32_t kMaxPolls = 1u << 26;
constexpr uint32_t kMaxWaitPolls = 1u << 26;
constexpr int kErrTimeout = 1;

// Kernel shape shared by every scan kernel.
constexpr int kThreads = 128;   // threads per CTA
constexpr int kSelectThreads = 64;  // selection: small blocks spread few queries over more SMs
constexpr int kMaxSplits = 64;  // data-range splits of a phase-1 scan
// Phase 2 cuts the data at any multiple of kSplitGranule points (whole chunks of every precision's
// summation loop) into at most kMaxSplitsW splits.
constexpr int kSplitGranule = 32;
constexpr int kMaxSplitsW = 512;
// Threads that share the merge of one query's splits (1, 8 or 32): a thread's loads are a chain
// a few deep, and few queries with many splits would leave most SMs idle. 32 threads read 8
// neighbouring queries at a time, which many queries pay for (8,191 queries x 342 splits in FP64:
// 200 us against 110).
inline int finalize_threads(int splits, int64_t m)
{
    return splits >= 64 && m <= 2048 ? 32 : (splits >= 16 ? 8 : 1);
}
// Largest |log2 of d1^power| of a query in an integer power class (class_c_max: less where values
// are small).
constexpr float kClassMaxLog2 = 64.0f;
// Fewest queries and points of a batch item whose phase 2 runs by power classes: a query's share of
// the sorting does not depend on the points, its gain does (64 items of 16,384 queries, us, with and
// without: 250 points 510 / 502, 500 693 / 678, 1,000 908 / 910, 2,000 1,273 / 1,318, 4,000 1,951 /
// 2,007; 256 of 4,096: 522 / 508, 712 / 702, 934 / 933, 1,372 / 1,371, 2,161 / 2,171).
constexpr int64_t kBatchClassMinQueries = 4096;
constexpr int64_t kBatchClassMinPoints = 1000;
constexpr int kPointGroups = 4;  // phase 2 with point groups (Plan::pg)

// Levels and bounds of Eq. 5 and Eq. 6, passed to kernels by value.
struct AlphaMap {
    double level[5];
    double r_min, r_max;
};

// FP32 copies are stored negated and duplicated, (-x, -x, -y, -y) and (z, z), so that one
// shared-memory load yields the register pairs that packed FP32x2 instructions operate on for
// two queries at once (q + (-x) is exactly q - x). They are kept in curve order (along a Hilbert
// curve of the points), with orig[] mapping a stored position back to the caller's index and one
// bounding box per 512-point tile. Points packed instead of queries (12 bytes a point, three loads
// for four of them) measured the same: 18.53 against 18.54 ms at 262,144 x 262,144. The FP64 copies keep the caller's order.
struct DatasetDev {
    const float4 *nxy2;     // [n_pad] (-x, -x, -y, -y), curve order
    const float2 *zz;       // [n_pad] (z, z) / z_unscale, curve order
    const int32_t *orig;    // [n_pad] caller's index of each stored point, -1 for padding
    const float4 *tile_box; // [n_pad / kTileF32Knn] (xmin, ymin, xmax, ymax) of finite points
    const float4 *sub_box;  // [n_pad / kSubTile] the same per 64-point sub-tile
    const float4 *super_box; // [ceil(tiles / kSuperTiles)] the same per 32 tiles
    const float4 *box;      // [1] bounding box of all points
    const double2 *xy64;    // [n_pad] caller's order
    const double *z64;      // [n_pad] caller's order
    int64_t n;
    int64_t n_pad;
    float z_max;            // largest |z| of the FP32 copy, as stored
    float z_min;            // smallest |z| of it other than 0 (+inf: all are 0)
    float z_unscale;        // power of two that takes a stored value back to the caller's
};

// How one scan pass is cut into work: query blocks (one CTA each) times data-range splits,
// each split a whole number of granules (kPadPoints points in phase 1, kSplitGranule in phase 2).
struct PassPlan {
    int q_per_block;   // queries handled by one CTA
    int qblocks;       // ceil(m / q_per_block)
    int splits;        // S: data-range splits, each scanned by its own CTA
    int64_t split_len; // points per split (whole granules)
};

struct Plan {
    int64_t m;
    PassPlan knn;  // phase 1 scan
    PassPlan w;    // phase 2 scan
    bool with_idx; // keep neighbour indices (needed for the kNN output)
    int kp;        // FP32 phase 1: register k-list length (8, 12, 16 or 32)
    int qw;        // FP32 phase 2: queries per thread (2, 4 or 8)
    int tw;        // FP32 phase 2: data points per shared-memory tile (256 or 512)
    int knn_slots; // phase-1 CTAs resident on the whole GPU (occupancy x SMs)
    int kq;        // pruned phase 1: queries per thread (2 or 4)
    int pg;        // phase 2: point groups per CTA (1: every thread sees every point)
    int pow_a;     // FP32 phase 2 by power classes: the integer powers of the two saturated levels
    int pow_b;     // of Eq. 6 (0: none); both 0: phase 2 runs in the queries' own order
    float c_max;   // ClassOrder::c_max
};

// Per-query parameters of phase 2 produced by the selection kernel.
//   F32: w = ex2(fma(log2(d2), neg_s, c)), neg_s = -alpha/2, c = alpha/2 * log2(d1^2)
//   F64, F64X: kappa = alpha / 2 (the coincidence scale for a query on a data point) and the
//   nearest squared distance the weights are relative to.
struct QParamF32 {
    float neg_s;
    float c;
};
struct QParamF64 {
    double kappa;
    double d1sq;
};

// The order FP32 phase 2 runs in when the queries are sorted into power classes (Plan::pow_a and
// pow_b): class kClassA (power pow_a), kClassG (any power) and kClassB (pow_b), each in a region
// of m entries, its query count in cnt[class].
enum PowerClass { kClassA = 0, kClassG = 1, kClassB = 2, kClasses = 3 };
struct ClassOrder {
    uint32_t *cnt;  // [kClasses], zeroed by the phase-1 kernel
    float *qx, *qy; // [kClasses][m]
    QParamF32 *qp;  // [kClasses][m]
    uint32_t *id;   // [kClasses][m] caller's query index
    int pow_a, pow_b;
    float c_max;    // largest log2 of d1^power in class A or B
};

// Scratch buffers of one interpolation (device memory owned by the library or by the
// caller of the allocation-free entry point).
struct Scratch {
    void *part_d2;     // [S_knn][k][m] float (F32) or double (F64): per-split sorted lists
    int32_t *part_idx; // [S_knn][k][m] or null when indices are not kept
    void *qparam;      // [m] QParamF32 / QParamF64
    void *part_sum;    // [S_w][4][m] float (w_hi, w_lo, wz_hi, wz_lo) or double
    ClassOrder cls;    // cnt null: no power classes
};

// Whether the unscaled sums of the integer power classes stay in range for a dataset, and a level
// of Eq. 6 as an integer power the class loops are built for (0: none).
bool power_classes_fit(int64_t n, float z_max);
// Largest log2 of d1^power for which a dataset's products d^-power z stay clear of underflow.
float class_c_max(const DatasetDev &ds);
int integer_level(double a);
size_t scratch_bytes(int precision, const Plan &pl, int k);
void scratch_carve(void *base, int precision, const Plan &pl, int k, Scratch *s);

// ---- launchers (all stream-ordered, return cudaGetLastError()) --------------------------
cudaError_t launch_f32_knn(const DatasetDev &ds, const Plan &pl, const float *qx,
                           const float *qy, int k, const Scratch &sc, int *err,
                           cudaStream_t st);
cudaError_t launch_f32_select(const Plan &pl, int k, double r_exp, const AlphaMap &am,
                              const Scratch &sc, float *out_alpha, int32_t *out_knn,
                              cudaStream_t st, const float *qx, const float *qy,
                              const uint32_t *perm = nullptr);
cudaError_t launch_f32_weights(const DatasetDev &ds, const Plan &pl, const float *qx,
                               const float *qy, const Scratch &sc, int *err, cudaStream_t st);
cudaError_t launch_f32_finalize(const DatasetDev &ds, const Plan &pl, const Scratch &sc, float *out,
                                cudaStream_t st, const uint32_t *perm = nullptr);
// Phase 1 with one warp per query, in the caller's order (queries that lie far apart compared
// with the data points): one split's lists in sc.part_d2 (and sc.part_idx when non-null).
cudaError_t launch_f32_knn_warp(const DatasetDev &ds, int64_t m, const float *qx,
                                const float *qy, int k, const Scratch &sc, int sm_count,
                                cudaStream_t st);
// Phase 1 over curve-ordered queries with nearest-first tile visiting and bounding-box pruning
// (one split); sqx / sqy are the queries in curve order.
constexpr int64_t kMaxCullTiles = 8192;
cudaError_t launch_f32_knn_cull(const DatasetDev &ds, const Plan &pl, const float *sqx,
                                const float *sqy, int k, const Scratch &sc, int *err,
                                cudaStream_t st);

// Spatial helpers (spatial.cu).
size_t radix_scratch_bytes(int64_t n);
cudaError_t radix_sort_pairs(uint32_t *keys, uint32_t *vals, int64_t n, void *tmp,
                             cudaStream_t st, int bits = 32);
cudaError_t bbox_of(const float2 *xy, int64_t n, uint32_t *scratch4, float4 *box,
                    cudaStream_t st);
cudaError_t curve_keys(const float *x, const float *y, const float2 *xy, int64_t n,
                        int64_t n_total, const float4 *box, uint32_t *keys, uint32_t *vals,
                        cudaStream_t st);
cudaError_t tile_boxes(const float4 *nxy2, int64_t ntiles, float4 *boxes, cudaStream_t st);
cudaError_t sub_tile_boxes(const float4 *nxy2, int64_t nsub, float4 *boxes, cudaStream_t st);
// Box of every group of kSuperTiles consecutive tile boxes (the last group may be shorter).
cudaError_t super_tile_boxes(const float4 *tile_boxes, int64_t ntiles, int64_t nsuper,
                             float4 *boxes, cudaStream_t st);
cudaError_t gather_queries(const float *qx, const float *qy, const uint32_t *perm, int64_t m,
                           float *sqx, float *sqy, cudaStream_t st);
cudaError_t curve_keys_f64(const double *x, const double *y, int64_t n, const float4 *box,
                            uint32_t *keys, uint32_t *vals, cudaStream_t st);
cudaError_t gather_queries_f64(const double *qx, const double *qy, const uint32_t *perm,
                               int64_t m, double *sqx, double *sqy, cudaStream_t st);

cudaError_t launch_f64_knn(const DatasetDev &ds, const Plan &pl, const double *qx,
                           const double *qy, int k, const Scratch &sc, int *err,
                           cudaStream_t st);
cudaError_t launch_f64_select(const Plan &pl, int k, double r_exp, const AlphaMap &am,
                              const Scratch &sc, float *out_alpha, int32_t *out_knn,
                              cudaStream_t st, const uint32_t *perm = nullptr);
// Phase 1 over curve-ordered FP64 queries, pruned like launch_f32_knn_cull; with pl.with_idx the
// lists are the k smallest (distance, caller index) pairs, so ties go to the lower index as in
// the caller-order scan; sqx / sqy are the queries in curve order and the dataset's points are read
// through its order map.
cudaError_t launch_f64_knn_cull(const DatasetDev &ds, const Plan &pl, const double *sqx,
                                const double *sqy, int k, const Scratch &sc, int *err,
                                cudaStream_t st);
// Phase 1 with one warp per query in the caller's order (one split's lists [k][m]); with
// pl.with_idx the lists are the k smallest (distance, caller index) pairs, as above.
cudaError_t launch_f64_knn_warp(const DatasetDev &ds, const Plan &pl, const double *qx,
                                const double *qy, int k, const Scratch &sc, int sm_count,
                                cudaStream_t st);
cudaError_t launch_f64_weights(const DatasetDev &ds, const Plan &pl, const double *qx,
                               const double *qy, const Scratch &sc, int *err,
                               cudaStream_t st);
cudaError_t launch_f64_finalize(const Plan &pl, const Scratch &sc, double *out,
                                cudaStream_t st, const uint32_t *perm = nullptr);
// AIDW_F64X phase 2 (kernels_f64x.cu); leaves part_sum in the layout launch_f64_finalize reads.
cudaError_t launch_f64x_weights(const DatasetDev &ds, const Plan &pl, const double *qx,
                                const double *qy, const Scratch &sc, int *err,
                                cudaStream_t st);

// Shape of the kernels: queries per CTA of each scan and the CTA slots per SM that occupancy
// allows (used to cut splits into whole waves). FP32 shapes follow the tuning fields of
// aidw_tune_config (kp: k-list length, qw: phase-2 queries per thread, tw: tile points).
int f32_knn_queries_per_block(int kp);
int f32_w_queries_per_block(int qw, int pg);
int f32_knn_slots_per_sm(int kp, bool with_idx);
// k-list length for k under a minimum (aidw_tune_config.knn_list).
int f32_list_length(int k, int kp_min);
// Queries per thread of the pruned phase 1 for list length kp under the shape's request
// (aidw_tune_config.knn_queries_per_thread; 0 = 4 for lists of up to 16, lists of 32 take 2).
inline int cull_queries_per_thread(int kp, int requested)
{
    return kp > 16 ? 2 : (requested == 2 ? 2 : 4);
}
// Built-in shape and the check of a caller's shape (autotune.cu).
aidw_tune_config tune_default();
bool tune_valid(const aidw_tune_config &c);
int f64_knn_queries_per_block(int k);
int f64_w_queries_per_block(int pg);
int f64_knn_slots_per_sm(int k, bool with_idx);
int f64x_w_queries_per_block(int pg);

// Pipe-rate microbenchmarks (probe.cu).
cudaError_t run_pipe_probe(int sm_count, aidw_pipe_rates *out);

// ---- programmatic dependent launch --------------------------------------------------------
// The kernels of one interpolation form a chain on one stream. Each is launched so that its blocks
// may start once every block of the kernel before it has started (grid_trigger), and waits
// (grid_wait) for that kernel to finish before it touches anything but the dataset and constant
// tables: launch latency, block start-up and table loads overlap the tail of the kernel before.
// What an earlier kernel of the chain or of the stream writes (the caller's queries among it) is
// read with __ldcg or through a pointer without __restrict__: a plain load of a const __restrict__
// array may become a read-only load, which wants the array unchanged from the kernel's start on,
// and that may now come before the array is written.
// A kernel without grid_trigger releases the next one when its blocks end: the FP64 phase 1, and the
// selections, which the phase-2 blocks behind them would crowd and then lie unevenly on the SMs
// (us, FP64 1,024 x 1,024: without chaining 74, chained 63, with triggers there too 80; FP32 with /
// without the selection's trigger: 1,024 x 1,024 33 / 31, 5,000 x 4,000 84 / 64, 5,000 x 30,000 150 /
// 120, 32,000 x 4,000 202 / 156, 34,231 x 4,373 over ordered queries 303 / 261, and before
// chaining 300).
#if defined(__CUDACC__)

template <typename... P, typename... A>
inline cudaError_t launch_chained(void (*fn)(P...), dim3 grid, unsigned threads, size_t smem,
                                  cudaStream_t st, A... args)
{
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, fn, static_cast<P>(args)...);
}

__device__ __forceinline__ void grid_wait()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

__device__ __forceinline__ void grid_trigger()
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// ---- device helpers: Blackwell bulk-copy (TMA) and mbarrier ------------------------------

__device__ __forceinline__ uint32_t smem_addr(const void *p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count)
                 : "memory");
}

__device__ __forceinline__ void fence_mbar_init()
{
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void fence_proxy_async_smem()
{
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t *bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)),
                 "r"(bytes)
                 : "memory");
}

// One-dimensional bulk copy global -> shared through the TMA unit; completion is signalled
// on `bar` as transaction bytes. dst, src and bytes must be multiples of 16.
__device__ __forceinline__ void tma_load_1d(void *dst, const void *src, uint32_t bytes,
                                            uint64_t *bar)
{
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
        ::"r"(smem_addr(dst)), "l"(src), "r"(bytes), "r"(smem_addr(bar))
        : "memory");
}

// Bounded wait for phase `parity` of `bar`. Returns false (and leaves the caller to raise
// the error word) if the phase did not complete within max_polls polls.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity,
                                          uint32_t max_polls = kMaxPolls)
{
    uint32_t addr = smem_addr(bar);
    for (uint32_t i = 0; i < max_polls; ++i) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done)
            : "r"(addr), "r"(parity)
            : "memory");
        if (done)
            return true;
    }
    return false;
}

__device__ __forceinline__ uint32_t ld_acquire(const uint32_t *p)
{
    uint32_t v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// Thread 0 waits (bounded: max_polls acquire loads, 256 ns apart at least) until
// *p >= target; the outcome is shared with the CTA through the shared word `flag`.
__device__ __forceinline__ bool cta_wait_count(const uint32_t *p, uint32_t target, int *flag,
                                               uint32_t max_polls = kMaxWaitPolls)
{
    if (threadIdx.x == 0) {
        bool ok = false;
        for (uint32_t i = 0; i < max_polls; ++i) {
            if (ld_acquire(p) >= target) {
                ok = true;
                break;
            }
            __nanosleep(256);
        }
        *flag = ok ? 1 : 0;
    }
    __syncthreads();
    const bool ok = *flag != 0;
    __syncthreads();
    return ok;
}

// MUFU approximations with flush-to-zero (single SFU instruction each).
__device__ __forceinline__ float lg2_approx(float x)
{
    float y;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ float ex2_approx(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ float rsq_approx(float x)
{
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ float rcp_approx(float x)
{
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Eq. 5 (Sec. 2.2 Step 2): fuzzy membership of the NN statistic, with pi / R_max as printed.
__device__ __forceinline__ double membership_eq5(double R, const AlphaMap &am)
{
    if (R <= am.r_min)
        return 0.0;
    if (R >= am.r_max)
        return 1.0;
    return 0.5 - 0.5 * cos((3.141592653589793 / am.r_max) * (R - am.r_min));
}

// Eq. 6 (Sec. 2.2 Step 3): alpha is alpha_1 up to mu = 0.1, alpha_5 from mu = 0.9, and in
// between runs linearly from alpha_s at mu = 0.1 + 0.2 (s - 1) to alpha_(s+1) 0.2 later.
__device__ __forceinline__ double alpha_eq6(double mu, const AlphaMap &am)
{
    if (mu <= 0.1)
        return am.level[0];
    if (mu >= 0.9)
        return am.level[4];
    int seg = static_cast<int>((mu - 0.1) * 5.0);
    seg = seg < 0 ? 0 : (seg > 3 ? 3 : seg);
    const double t = (mu - (0.1 + 0.2 * seg)) * 5.0;
    return am.level[seg] * (1.0 - t) + am.level[seg + 1] * t;
}

// Kahan step: adds v to the running sum h whose compensation (excess added so far) is c.
template <typename T>
__device__ __forceinline__ void kahan_add(T &h, T &c, T v)
{
    const T y = v - c;
    const T t = h + y;
    c = (t - h) - y;
    h = t;
}

#endif  // __CUDACC__

}  // namespace aidw
