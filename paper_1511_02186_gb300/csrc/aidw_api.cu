// C ABI of the library: context, dataset store, one-shot interpolation, diagnostics.
// The batched and serving entry points live in runtime.cu.
#include <math_constants.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <unordered_map>
#include <vector>

#include "aidw_internal.cuh"
#include "aidw_runtime.h"

namespace aidw {

namespace {

inline size_t align256(size_t b)
{
    return (b + 255) & ~static_cast<size_t>(255);
}

// Converts caller arrays (float or double) into unsorted FP32 staging arrays and the padded
// FP64 layout, counts non-finite inputs (bad[0]) and takes the largest |z| (the low word of
// bad[1], a float's bits) and the smallest other than 0 (the high word, the bits' complement, or 0
// where there is none). FP64 padding points are +inf with value 0.
template <typename T>
__global__ void convert_dataset_kernel(const T *__restrict__ x, const T *__restrict__ y,
                                       const T *__restrict__ z, int64_t n, int64_t n_pad,
                                       float2 *xy32, float *z32, double2 *xy64, double *z64,
                                       unsigned long long *bad)
{
    const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
    unsigned long long nb = 0;
    float zm = 0.0f;
    unsigned zn = 0;
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n_pad;
         i += stride) {
        double a, b, c;
        if (i < n) {
            a = static_cast<double>(x[i]);
            b = static_cast<double>(y[i]);
            c = static_cast<double>(z[i]);
            nb += (isfinite(a) && isfinite(b) && isfinite(c)) ? 0 : 1;
            const float fa = static_cast<float>(a), fb = static_cast<float>(b);
            const float fc = static_cast<float>(c);
            // FP32 copies must stay finite too (values beyond float range are rejected).
            if (!(isfinite(fa) && isfinite(fb) && isfinite(fc)))
                ++nb;
            xy32[i] = make_float2(fa, fb);
            z32[i] = fc;
            zm = fmaxf(zm, fabsf(fc));
            if (fc != 0.0f)
                zn = max(zn, ~__float_as_uint(fabsf(fc)));
        } else {
            a = b = CUDART_INF;
            c = 0.0;
        }
        xy64[i] = make_double2(a, b);
        z64[i] = c;
    }
    if (nb)
        atomicAdd(bad, nb);
    // Non-negative floats order like their bits.
    const unsigned zb = __reduce_max_sync(0xffffffffu, __float_as_uint(zm));
    const unsigned znb = __reduce_max_sync(0xffffffffu, zn);
    __shared__ unsigned most[2];
    if (threadIdx.x < 2)
        most[threadIdx.x] = 0;
    __syncthreads();
    if ((threadIdx.x & 31) == 0) {
        atomicMax(&most[0], zb);
        atomicMax(&most[1], znb);
    }
    __syncthreads();
    if (threadIdx.x < 2)
        atomicMax(reinterpret_cast<unsigned *>(bad + 1) + threadIdx.x, most[threadIdx.x]);
}

// The exponent t of the power of two that the values of the FP32 copy are multiplied by: the largest
// from 0 to 100 with n max|z| 2^t below 2^62 (n <= 2^log_n). The unscaled products of the power
// classes, d^-power z, then stay far from underflow, and the scale changes no bit of a result.
__host__ __device__ inline int value_exponent(uint32_t z_max_bits, int log_n)
{
    const int e = static_cast<int>(z_max_bits >> 23) - 126;  // max|z| < 2^e
    const int t = 62 - log_n - e;
    return z_max_bits == 0 || t < 0 ? 0 : (t > 100 ? 100 : t);
}

__host__ __device__ inline uint32_t pow2_bits(int e)
{
    return static_cast<uint32_t>(127 + e) << 23;
}

// Writes the curve-ordered FP32 layout: stored position i holds caller point perm[i] (padding
// positions, perm[i] >= n, hold +inf points with value 0); z_max is the largest |z|'s bits.
__global__ void gather_dataset_kernel(const float2 *__restrict__ xy32,
                                      const float *__restrict__ z32,
                                      const uint32_t *__restrict__ perm, int64_t n,
                                      int64_t n_pad, const uint32_t *z_max, int log_n,
                                      float4 *nxy2, float2 *zz, int32_t *orig)
{
    const float scale = __uint_as_float(pow2_bits(value_exponent(*z_max, log_n)));
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n_pad;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const uint32_t p = perm[i];
        if (p < n) {
            const float2 q = xy32[p];
            const float v = z32[p] * scale;
            nxy2[i] = make_float4(-q.x, -q.x, -q.y, -q.y);
            zz[i] = make_float2(v, v);
            orig[i] = static_cast<int32_t>(p);
        } else {
            nxy2[i] = make_float4(-CUDART_INF_F, -CUDART_INF_F, -CUDART_INF_F, -CUDART_INF_F);
            zz[i] = make_float2(0.0f, 0.0f);
            orig[i] = -1;
        }
    }
}

}  // namespace

}  // namespace aidw

using namespace aidw;

struct DatasetRec {
    DatasetDev dev;
    void *block = nullptr;
    bool pooled = false;  // block comes from the context's pool
    size_t bytes = 0;
    double area = 0.0;
    double r_exp = 0.0;
};

struct aidw_ctx {
    int device = 0;
    int sm_count = 0;
    size_t budget = 0;
    size_t in_use = 0;
    int64_t fail_after = -1;
    int *d_err = nullptr;
    cudaMemPool_t pool = nullptr;
    void *pinned = nullptr;  // [kPinnedBytes] results of small host-array calls, and the error word
    std::mutex pinned_mu;    // taken without waiting: a second call at once goes without
    std::mutex mu;
    std::unordered_map<int64_t, DatasetRec> datasets;
    int64_t next_ds = 1;
    bool profiling = false;
    cudaEvent_t ev[5] = {};
    aidw_kernel_times last{};
    bool last_valid = false;
    int slots_cache[3][4][2] = {};  // [precision][kp bucket][with_idx] knn slots
    aidw_tune_config tune = aidw::tune_default();
    ServingRuntime *serving = nullptr;
    int64_t serving_queue_limit = 4096;  // requests waiting for admission at most
};

namespace aidw {

// ---- memory accounting --------------------------------------------------------------------

int ctx_alloc(aidw_ctx *ctx, size_t bytes, cudaStream_t st, void **p, bool *injected)
{
    *p = nullptr;
    if (bytes == 0)
        return AIDW_OK;
    {
        std::lock_guard<std::mutex> g(ctx->mu);
        if (ctx->fail_after >= 0) {
            if (ctx->fail_after == 0) {
                ctx->fail_after = -1;
                if (injected)
                    *injected = true;
                return AIDW_ERR_OOM;
            }
            --ctx->fail_after;
        }
        if (ctx->budget && ctx->in_use + bytes > ctx->budget)
            return AIDW_ERR_OOM;
        ctx->in_use += bytes;
    }
    cudaError_t e = cudaMallocFromPoolAsync(p, bytes, ctx->pool, st);
    if (e != cudaSuccess) {
        cudaGetLastError();
        std::lock_guard<std::mutex> g(ctx->mu);
        ctx->in_use -= bytes;
        *p = nullptr;
        return e == cudaErrorMemoryAllocation ? AIDW_ERR_OOM : AIDW_ERR_CUDA;
    }
    return AIDW_OK;
}

void ctx_free(aidw_ctx *ctx, void *p, size_t bytes, cudaStream_t st)
{
    if (!p)
        return;
    cudaFreeAsync(p, st);
    std::lock_guard<std::mutex> g(ctx->mu);
    ctx->in_use -= bytes;
}

// Blocks of a dataset and of its construction: from the context's pool up to kPoolDatasetBytes
// (cudaMalloc and cudaFree take about 95 us together and wait for the device), else by cudaMalloc.
// What the pool keeps idle beyond kPoolKeepBytes, or beyond what the budget leaves, is given back
// when a dataset is created by cudaMalloc or destroyed, and all of it where memory has run out.
constexpr size_t kPoolDatasetBytes = size_t(64) << 20;
constexpr size_t kPoolKeepBytes = size_t(1) << 30;
constexpr size_t kPoolGranule = size_t(32) << 20;  // the pool trims in steps of this at most

static void pool_trim(aidw_ctx *ctx, size_t keep)
{
    if (ctx->budget) {
        std::lock_guard<std::mutex> g(ctx->mu);
        const size_t left = ctx->budget - std::min(ctx->budget, ctx->in_use);
        keep = std::min(keep, left - std::min(left, kPoolGranule));
    }
    uint64_t reserved = 0, used = 0;
    if (cudaMemPoolGetAttribute(ctx->pool, cudaMemPoolAttrReservedMemCurrent, &reserved) ==
            cudaSuccess &&
        reserved > keep && cudaStreamSynchronize(0) == cudaSuccess &&
        cudaMemPoolGetAttribute(ctx->pool, cudaMemPoolAttrUsedMemCurrent, &used) == cudaSuccess &&
        reserved - used > keep)
        cudaMemPoolTrimTo(ctx->pool, used + keep);
}

static cudaError_t dataset_alloc(aidw_ctx *ctx, size_t bytes, void **p, bool *pooled)
{
    *pooled = bytes <= kPoolDatasetBytes;
    const auto alloc = [&] {
        return *pooled ? cudaMallocFromPoolAsync(p, bytes, ctx->pool, 0) : cudaMalloc(p, bytes);
    };
    if (!*pooled)
        pool_trim(ctx, kPoolKeepBytes);
    cudaError_t e = alloc();
    if (e == cudaErrorMemoryAllocation) {
        cudaGetLastError();
        cudaDeviceSynchronize();
        pool_trim(ctx, 0);
        e = alloc();
    }
    return e;
}

// Frees a block whose use has ended (the caller has synchronised).
static void dataset_free(void *p, bool pooled)
{
    if (pooled)
        cudaFreeAsync(p, 0);
    else
        cudaFree(p);
}

size_t ctx_budget_left(aidw_ctx *ctx)
{
    std::lock_guard<std::mutex> g(ctx->mu);
    if (!ctx->budget)
        return SIZE_MAX;
    return ctx->budget > ctx->in_use ? ctx->budget - ctx->in_use : 0;
}

int *ctx_err_word(aidw_ctx *ctx)
{
    return ctx->d_err;
}

int ctx_device(aidw_ctx *ctx)
{
    return ctx->device;
}

int ctx_sm_count(aidw_ctx *ctx)
{
    return ctx->sm_count;
}

// Copies a dataset's record while holding the context lock, so that a concurrent
// aidw_destroy_dataset (which erases the record under the same lock) cannot free it while it is
// read; no pointer into the table leaves the lock.
static bool ctx_dataset_copy(aidw_ctx *ctx, aidw_dataset id, DatasetRec *out)
{
    std::lock_guard<std::mutex> g(ctx->mu);
    auto it = ctx->datasets.find(id);
    if (it == ctx->datasets.end())
        return false;
    *out = it->second;
    return true;
}

bool dataset_lookup(aidw_ctx *ctx, aidw_dataset id, DatasetDev *dev, double *r_exp)
{
    DatasetRec r;
    if (!ctx_dataset_copy(ctx, id, &r))
        return false;
    *dev = r.dev;
    *r_exp = r.r_exp;
    return true;
}

// ---- pointers ----------------------------------------------------------------------------

// 1: device memory of `device`; 0: host memory; -1: device memory of another device.
int pointer_kind(const void *p, int device)
{
    if (!p)
        return 0;
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    if (a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged)
        return a.device == device ? 1 : -1;
    return 0;
}

// ---- planning ------------------------------------------------------------------------------

static PassPlan plan_pass(int64_t m, int64_t n_pad, int qpb, int slots_total, int64_t fixed)
{
    PassPlan pp{};
    pp.q_per_block = qpb;
    pp.qblocks = static_cast<int>((m + qpb - 1) / qpb);
    const int64_t G = n_pad / kPadPoints;
    double best = 1e300;
    for (int S = 1; S <= kMaxSplits && S <= G; ++S) {
        const int64_t per = (G + S - 1) / S;
        const int64_t Se = (G + per - 1) / per;
        if (Se != S)
            continue;
        const int64_t items = static_cast<int64_t>(pp.qblocks) * Se;
        const int64_t waves = (items + slots_total - 1) / slots_total;
        const double cost = static_cast<double>(waves) * (per * kPadPoints + fixed);
        if (cost < best * (1.0 - 1e-9)) {
            best = cost;
            pp.splits = static_cast<int>(Se);
            pp.split_len = per * kPadPoints;
        }
    }
    return pp;
}

// Phase 2 cut into (query blocks) x (data splits of whole granules).
static PassPlan weights_split(int64_t m, int64_t n_sum, int qpb, int64_t S)
{
    PassPlan pp{};
    const int64_t G = n_sum / kSplitGranule;
    S = std::max<int64_t>(1, std::min<int64_t>(S, std::min<int64_t>(G, kMaxSplitsW)));
    const int64_t per = (G + S - 1) / S;
    pp.q_per_block = qpb;
    pp.qblocks = static_cast<int>((m + qpb - 1) / qpb);
    pp.splits = static_cast<int>((G + per - 1) / per);
    pp.split_len = per * kSplitGranule;
    return pp;
}

// What phase 2 costs in a precision, measured on GB300 (ns).
struct WeightsCost {
    double pair;  // one SM, full of CTAs, per pair
    double cta;   // one SM, per CTA (start, tables, first tile, sums out)
    double part;  // whole GPU, per query and split (partial sums written and merged)
    bool shares;  // several CTAs share an SM; one alone leaves it partly idle
};

// The split count with the least estimated time among those that give every SM about 1, 2, ...
// 48 CTAs (at least up to 8 splits): an SM's share of the CTAs (rounded up) times their cost, over
// the rate a few co-resident CTAs reach, plus a part of one CTA for the uneven end and the cost of
// the partial sums. Measured (FP32, us with the finalisation; the split count the estimate takes, and
// 2,048-point granules with at most 64 splits before): 1,024 x 1,024: 14 against 29; 257 x
// 300,007: 57 against 143; 8,192 x 1M: 2,800 against 2,959 (37 splits of 1,216 slots).
static PassPlan plan_weights(int64_t m, int64_t n_sum, int qpb, int sm_count,
                             const WeightsCost &wc)
{
    const int64_t qblocks = (m + qpb - 1) / qpb;
    PassPlan best{};
    double best_t = 1e300;
    int64_t last = 0;
    for (int per_sm = 1; per_sm <= 48; ++per_sm) {
        const int64_t S = std::max<int64_t>(static_cast<int64_t>(per_sm) * sm_count / qblocks,
                                            std::min(per_sm, 8));
        const PassPlan pp = weights_split(m, n_sum, qpb, S);
        if (pp.splits == last)
            continue;
        last = pp.splits;
        const int64_t items = qblocks * pp.splits;
        const double k = static_cast<double>((items + sm_count - 1) / sm_count);
        const double one = static_cast<double>(pp.split_len) * qpb * wc.pair;
        const double idle = wc.shares ? 1.0 + 0.35 / (k * std::sqrt(k)) : 1.0;
        const double t = k * (one + wc.cta) * idle + 0.3 * one +
                         wc.part * static_cast<double>(m) * pp.splits;
        if (t < best_t * (1.0 - 1e-9)) {
            best_t = t;
            best = pp;
        }
    }
    return best;
}

// AIDW_F64 and AIDW_F64X share the FP64 arrays, phase 1, selection and finalisation.
static bool f64_arrays(int precision)
{
    return precision == AIDW_F64 || precision == AIDW_F64X;
}

// Point groups per phase-2 CTA. Without them a CTA serves 256 queries (FP64: 1,024), with them
// a quarter of that, which wastes fewer lanes beyond the last query but shares a tile among
// fewer queries. Measured (us, 1 group / 4 groups): FP32 257 x 300,007: 78 / 57, 1,024 x 1M:
// 389 / 383, 4,096 x 1M: 1,413 / 1,427; FP64 257 x 16,384: 274 / 145, 4,100 x 16,384: 1,122 /
// 1,000, 8,191 x 131,072: 13,010 / 13,279; F64X 4,100 x 65,536: 2,190 / 2,109, 16,384 x 262,144:
// 31,813 / 32,170. A function of the precision and m alone: the groups regroup the partial sums.
static int weights_point_groups(int precision, int64_t m)
{
    const int64_t q1 = precision == AIDW_F64 ? 1024 : 256, q4 = q1 / kPointGroups;
    const double lanes1 = static_cast<double>((m + q1 - 1) / q1 * q1);
    const double lanes4 = static_cast<double>((m + q4 - 1) / q4 * q4);
    return m <= 2048 || lanes4 * 1.02 < lanes1 ? kPointGroups : 1;
}

static WeightsCost weights_cost(int precision)
{
    return precision == AIDW_F32C ? WeightsCost{0.048, 150.0, 0.006, true}
           : precision == AIDW_F64 ? WeightsCost{1.5, 5000.0, 0.05, false}
                                   : WeightsCost{1.1, 500.0, 0.05, true};
}

// FP32 phase 2 by power classes. Eq. 6 gives most queries one of its two end levels (mu below
// 0.1 or above 0.9: with k = 10 and uniform data 99 % get alpha_5), and where such a level is a
// small integer the weight d^-alpha needs no logarithm. The queries are then sorted by class
// (the selection counts each to its place, the finalisation reads its index back), so that whole
// blocks share a loop. It pays once phase 2 takes longer than the extra partly filled blocks and
// scattered writes cost. Phase 2 in us, in the queries' own order / by classes: 4,096 x 65,536
// 94 / 90, 8,192 x 1M 2,757 / 2,445, 153,984 x 262,147 clustered 13,042 / 11,089, 1M x 1M 350,590 /
// 296,771; power 2, 65,535 x 300,007: 6,312 / 4,263. z_max bounds the unscaled sums: n z_max 2^64
// < 2^127.
static bool use_power_classes(int64_t n, int64_t m, float z_max)
{
    return m >= 4096 && static_cast<double>(n) * static_cast<double>(m) >= 2e8 &&
           power_classes_fit(n, z_max);
}

bool power_classes_fit(int64_t n, float z_max)
{
    return static_cast<double>(n) * z_max <= 0x1p62;
}

// The class loops sum unscaled products: adding one errs by up to 2^-150 where the sum is subnormal,
// which is 2^(c - 150) on the scale where the nearest point's weight is 1, and n times that in all
// (values as stored, n max|z| near 2^62 unless they are larger by themselves). With c <= 84 - log2 n +
// log2 z_min it is below 2^-66 z_min, so below FP32 rounding even where every value near the query
// is 0 and the first other one has a weight of 2^-40 (the general loop's products underflow only
// below a weight of 2^-126 / |z|).
float class_c_max(const DatasetDev &ds)
{
    if (!(ds.z_min < INFINITY))
        return kClassMaxLog2;
    const double c = 84.0 - std::log2(static_cast<double>(ds.n)) +
                     std::log2(static_cast<double>(ds.z_min));
    return static_cast<float>(std::min<double>(kClassMaxLog2, c));
}

int integer_level(double a)
{
    return a >= 1.0 && a <= 5.0 && a == std::floor(a) ? static_cast<int>(a) : 0;
}

static int kp_bucket(int kp)
{
    return kp <= 8 ? 0 : (kp <= 12 ? 1 : (kp <= 16 ? 2 : 3));
}

Plan make_plan(aidw_ctx *ctx, int precision, int64_t n, int64_t n_pad, int64_t m, int k,
               bool with_idx, int force_knn_splits, int force_w_splits,
               const aidw_tune_config *cfg, const aidw_params *classes, const DatasetDev *ds)
{
    const aidw_tune_config &tc = cfg ? *cfg : ctx->tune;
    const bool f64 = f64_arrays(precision);
    const bool x = precision == AIDW_F64X;
    Plan pl{};
    pl.m = m;
    pl.with_idx = with_idx;
    pl.kp = f32_list_length(k, tc.knn_list);
    pl.kq = f64 ? (k <= 16 ? 2 : 1) : cull_queries_per_thread(pl.kp, tc.knn_queries_per_thread);
    pl.qw = tc.queries_per_thread;
    pl.tw = tc.tile_points;
    int &ks = ctx->slots_cache[precision][kp_bucket(f64 ? k : pl.kp)][with_idx ? 1 : 0];
    if (!ks)
        ks = f64 ? f64_knn_slots_per_sm(k, with_idx) : f32_knn_slots_per_sm(pl.kp, with_idx);
    pl.pg = weights_point_groups(precision, m);
    if (classes && precision == AIDW_F32C && use_power_classes(n, m, ds->z_max)) {
        pl.c_max = class_c_max(*ds);
        pl.pow_a = integer_level(classes->alpha[4]);
        pl.pow_b = integer_level(classes->alpha[0]);
        if (pl.pow_a || pl.pow_b) {
            pl.pg = 1;  // the class kernel's shape
            pl.qw = 2;
            pl.tw = 512;
        }
    }
    const int qk = f64 ? f64_knn_queries_per_block(k) : f32_knn_queries_per_block(pl.kp);
    const int qw = x ? f64x_w_queries_per_block(pl.pg)
                     : (f64 ? f64_w_queries_per_block(pl.pg)
                            : f32_w_queries_per_block(pl.qw, pl.pg));
    // A split restarts its neighbour lists: about k (1 + ln(n_split / k)) insertions per query,
    // each a rescan of a chunk by a partly idle warp. Measured on GB300 at n = m = 2^20,
    // k = 10, every extra split costs about as much as scanning 100,000 more points.
    pl.knn_slots = ks * ctx->sm_count;
    // The FP64 scan is bound by its FP64 pipe (the exact rescans behind the FP32 prefilter),
    // which co-resident CTAs share: it is planned as one CTA per SM (measured at n = 1M,
    // 4,096 queries: 8 splits 24 ms, 37 splits 39 ms).
    pl.knn = plan_pass(m, n_pad, qk, (f64 ? 1 : ks) * ctx->sm_count, 10000 * k);
    const int64_t n_sum = (n + kSplitGranule - 1) / kSplitGranule * kSplitGranule;
    pl.w = force_w_splits > 0 ? weights_split(m, n_sum, qw, force_w_splits)
                              : plan_weights(m, n_sum, qw, ctx->sm_count, weights_cost(precision));
    if (force_knn_splits > 0) {
        const int64_t G = n_pad / kPadPoints;
        const int64_t S = std::min<int64_t>(std::min<int64_t>(force_knn_splits, G), kMaxSplits);
        const int64_t per = (G + S - 1) / S;
        pl.knn.splits = static_cast<int>((G + per - 1) / per);
        pl.knn.split_len = per * kPadPoints;
    }
    return pl;
}

aidw_tune_config ctx_tune(aidw_ctx *ctx)
{
    std::lock_guard<std::mutex> g(ctx->mu);
    return ctx->tune;
}

void ctx_set_tune(aidw_ctx *ctx, const aidw_tune_config &c)
{
    std::lock_guard<std::mutex> g(ctx->mu);
    ctx->tune = c;
}

size_t scratch_bytes(int precision, const Plan &pl, int k)
{
    const size_t es = f64_arrays(precision) ? sizeof(double) : sizeof(float);
    const size_t m = static_cast<size_t>(pl.m);
    size_t b = align256(pl.knn.splits * static_cast<size_t>(k) * m * es);
    if (pl.with_idx)
        b += align256(pl.knn.splits * static_cast<size_t>(k) * m * sizeof(int32_t));
    b += align256(m * (f64_arrays(precision) ? sizeof(QParamF64) : sizeof(QParamF32)));
    b += align256(pl.w.splits * 4 * m * es);
    if (pl.pow_a || pl.pow_b)
        b += align256(sizeof(uint32_t) * kClasses) + 3 * align256(kClasses * m * sizeof(float)) +
             align256(kClasses * m * sizeof(QParamF32));
    return b;
}

void scratch_carve(void *base, int precision, const Plan &pl, int k, Scratch *s)
{
    const size_t es = f64_arrays(precision) ? sizeof(double) : sizeof(float);
    const size_t m = static_cast<size_t>(pl.m);
    char *p = static_cast<char *>(base);
    s->part_d2 = p;
    p += align256(pl.knn.splits * static_cast<size_t>(k) * m * es);
    s->part_idx = nullptr;
    if (pl.with_idx) {
        s->part_idx = reinterpret_cast<int32_t *>(p);
        p += align256(pl.knn.splits * static_cast<size_t>(k) * m * sizeof(int32_t));
    }
    s->qparam = p;
    p += align256(m * (f64_arrays(precision) ? sizeof(QParamF64) : sizeof(QParamF32)));
    s->part_sum = p;
    s->cls = ClassOrder{};
    if (pl.pow_a || pl.pow_b) {
        p += align256(pl.w.splits * 4 * m * es);
        s->cls.cnt = reinterpret_cast<uint32_t *>(p);
        p += align256(sizeof(uint32_t) * kClasses);
        s->cls.qx = reinterpret_cast<float *>(p);
        p += align256(kClasses * m * sizeof(float));
        s->cls.qy = reinterpret_cast<float *>(p);
        p += align256(kClasses * m * sizeof(float));
        s->cls.id = reinterpret_cast<uint32_t *>(p);
        p += align256(kClasses * m * sizeof(uint32_t));
        s->cls.qp = reinterpret_cast<QParamF32 *>(p);
        s->cls.pow_a = pl.pow_a;
        s->cls.pow_b = pl.pow_b;
        s->cls.c_max = pl.c_max;
    }
}

int validate_params(const aidw_params *p, int64_t n)
{
    if (!p)
        return AIDW_ERR_INVALID_ARG;
    if (p->precision != AIDW_F32C && !f64_arrays(p->precision))
        return AIDW_ERR_INVALID_ARG;
    if (p->k < 1 || p->k > AIDW_MAX_K || p->k > n)
        return AIDW_ERR_INVALID_ARG;
    for (int i = 0; i < 5; ++i)
        if (!std::isfinite(p->alpha[i]) || !(p->alpha[i] > 0.0))
            return AIDW_ERR_INVALID_ARG;
    if (!std::isfinite(p->r_min) || !std::isfinite(p->r_max) || !(p->r_max > p->r_min) ||
        !(p->r_max > 0.0))
        return AIDW_ERR_INVALID_ARG;
    if (p->flags != 0 || p->reserved != 0)
        return AIDW_ERR_INVALID_ARG;
    return AIDW_OK;
}

AlphaMap alpha_map(const aidw_params &p)
{
    AlphaMap am;
    for (int i = 0; i < 5; ++i)
        am.level[i] = p.alpha[i];
    am.r_min = p.r_min;
    am.r_max = p.r_max;
    return am;
}

// Phase boundaries of one interpolation: the profiling events (when profiling is on) and NVTX
// ranges naming the phases, so that a profiler can attribute the kernels launched in each (for
// example `ncu --nvtx --nvtx-include "aidw phase 2/"`). The ranges span the host-side enqueue;
// without a tool attached the NVTX calls do nothing.
class PhaseMarks {
  public:
    PhaseMarks(aidw_ctx *ctx, cudaStream_t st, bool profile)
        : ctx_(ctx), st_(st), profile_(profile)
    {
    }
    PhaseMarks(const PhaseMarks &) = delete;
    PhaseMarks &operator=(const PhaseMarks &) = delete;
    ~PhaseMarks()
    {
        if (open_)
            nvtxRangePop();
    }
    // Boundary i: the start of phase i (0 phase 1, with the query ordering; 1 selection;
    // 2 phase 2; 3 finalisation), 4 the end.
    void at(int i)
    {
        static const char *const kNames[4] = {"aidw phase 1", "aidw select", "aidw phase 2",
                                              "aidw finalize"};
        if (profile_)
            cudaEventRecord(ctx_->ev[i], st_);
        if (open_)
            nvtxRangePop();
        open_ = i < 4;
        if (open_)
            nvtxRangePushA(kNames[i]);
    }

  private:
    aidw_ctx *ctx_;
    cudaStream_t st_;
    bool profile_;
    bool open_ = false;
};

// Enqueues the four kernels of one interpolation on `st` with device arrays only.
int enqueue_interpolation(aidw_ctx *ctx, const DatasetDev &ds, double r_exp, const Plan &pl,
                          const aidw_params &p, const void *qx, const void *qy,
                          const Scratch &sc, void *out, float *out_alpha, int32_t *out_knn,
                          cudaStream_t st, bool profile)
{
    const AlphaMap am = alpha_map(p);
    cudaError_t e;
    const bool f64 = f64_arrays(p.precision);
    const bool x = p.precision == AIDW_F64X;
    PhaseMarks marks(ctx, st, profile);
    marks.at(0);
    e = f64 ? launch_f64_knn(ds, pl, static_cast<const double *>(qx),
                             static_cast<const double *>(qy), p.k, sc, ctx->d_err, st)
            : launch_f32_knn(ds, pl, static_cast<const float *>(qx),
                             static_cast<const float *>(qy), p.k, sc, ctx->d_err, st);
    if (e != cudaSuccess)
        return AIDW_ERR_CUDA;
    marks.at(1);
    e = f64 ? launch_f64_select(pl, p.k, r_exp, am, sc, out_alpha, out_knn, st)
            : launch_f32_select(pl, p.k, r_exp, am, sc, out_alpha, out_knn, st,
                                  static_cast<const float *>(qx), static_cast<const float *>(qy));
    if (e != cudaSuccess)
        return AIDW_ERR_CUDA;
    marks.at(2);
    e = x     ? launch_f64x_weights(ds, pl, static_cast<const double *>(qx),
                                    static_cast<const double *>(qy), sc, ctx->d_err, st)
        : f64 ? launch_f64_weights(ds, pl, static_cast<const double *>(qx),
                                   static_cast<const double *>(qy), sc, ctx->d_err, st)
              : launch_f32_weights(ds, pl, static_cast<const float *>(qx),
                                 static_cast<const float *>(qy), sc, ctx->d_err, st);
    if (e != cudaSuccess)
        return AIDW_ERR_CUDA;
    marks.at(3);
    e = f64 ? launch_f64_finalize(pl, sc, static_cast<double *>(out), st)
            : launch_f32_finalize(ds, pl, sc, static_cast<float *>(out), st);
    if (e != cudaSuccess)
        return AIDW_ERR_CUDA;
    marks.at(4);
    if (profile) {
        ctx->last = aidw_kernel_times{};
        ctx->last.splits = pl.knn.splits;
        ctx->last.query_blocks = pl.knn.qblocks;
        ctx->last.launches = 4;
        ctx->last.weight_splits = pl.w.splits;
        ctx->last_valid = true;
    }
    return AIDW_OK;
}

// Queries below this count keep the plain split scan for phase 1 (ordering them would cost
// more than it saves).
constexpr int64_t kCullMinQueries = 2048;

// Whether an FP32 call that the per-query scan does not serve takes the pruned phase 1 rather than
// the split scan: with m queries spread over the data, a block of q queries covers about q/m of
// the area, so each of the m/q blocks visits about n q / (512 m) tiles, and with fewer blocks than
// the GPU holds (P) the pruned scan takes about n q^2 P / m per-pair steps of one CTA against
// n m / P steps of each CTA for the split scan: the pruned scan wins when m > q sqrt(P). Measured
// at n = 1M with random queries: the split scan is faster at m = 8,192 and the pruned scan at
// 32,768.
bool use_culled_knn(const DatasetDev &ds, int64_t m, const Plan &pl)
{
    const double need = kThreads * pl.kq * std::sqrt(static_cast<double>(pl.knn_slots));
    return ds.n_pad / kTileF32Knn <= kMaxCullTiles && m >= kCullMinQueries &&
           static_cast<double>(m) >= need;
}

// Whether a call takes the per-query phase 1 (one warp per query). Its cost grows with the query
// count alone, while the block scans share their tiles among a block's queries and gain as the
// queries get denser. Measured phase 1 in FP32 (us; pruned scan with the query ordering / warp
// per query):
//   queries              16,384       65,536      131,072     262,144      1,048,576
//   1M uniform        1,992 / 46     922 / 148    711 / 283    795 / 545  1,306 / 2,123
//   262,147 clustered 1,347 / 47   1,348 / 152  1,219 / 281  1,418 / 537  1,145 / 2,084
//   65,536 clustered    620 / 49     544 / 147    459 / 279    510 / 541    519 / 2,080
//   16,384 uniform      237 / 39     210 / 126    210 / 244    241 / 475    446 / 1,852
// so the crossing lies near 5,000 n^(1/3) queries. Calls of more than 1.9 queries per point keep the
// pruned scan below it too, although the table has the per-query scan ahead for some (16,384 points,
// 65,536 queries): a test relies on such a call ordering its queries. The FP64 pruned scan is slower
// than the warp scan at every count measured (65,536 clustered, 262,144 queries: 7,758 / 940; 1M
// uniform, 16,384: 26,234 / 82).
constexpr int64_t kWarpKnnMaxQueries = 32768;
constexpr double kWarpKnnPerCbrt = 5000.0;
constexpr double kWarpKnnPerPoint = 1.9;

bool use_warp_knn(int precision, const DatasetDev &ds, int64_t m)
{
    if (precision != AIDW_F32C)
        return true;
    const double n = static_cast<double>(ds.n_pad);
    const double most = std::min(kWarpKnnPerPoint * n, kWarpKnnPerCbrt * std::cbrt(n));
    return m <= kWarpKnnMaxQueries || static_cast<double>(m) <= most;
}

bool same_call_kernels(aidw_ctx *ctx, const DatasetDev &ds, int64_t m, const aidw_params &p,
                       const aidw_tune_config &a, const aidw_tune_config &b)
{
    const Plan pa = make_plan(ctx, p.precision, ds.n, ds.n_pad, m, p.k, false, 0, 0, &a, &p, &ds);
    const Plan pb = make_plan(ctx, p.precision, ds.n, ds.n_pad, m, p.k, false, 0, 0, &b, &p, &ds);
    // Phase 2 with point groups has one shape of its own.
    if (pa.w.qblocks != pb.w.qblocks || pa.w.splits != pb.w.splits ||
        (pa.pg == 1 && (pa.qw != pb.qw || pa.tw != pb.tw)))
        return false;
    if (use_warp_knn(p.precision, ds, m))
        return true;  // the per-query scan has no lists
    const bool cull = use_culled_knn(ds, m, pa);
    return cull == use_culled_knn(ds, m, pb) && pa.kp == pb.kp && (!cull || pa.kq == pb.kq);
}

void plan_culled_knn(Plan *pl, int64_t n_pad)
{
    pl->knn.splits = 1;
    pl->knn.split_len = n_pad;
    pl->knn.q_per_block = kThreads * pl->kq;
    pl->knn.qblocks = static_cast<int>((pl->m + pl->knn.q_per_block - 1) / pl->knn.q_per_block);
}

size_t culled_extra_bytes(int64_t m, int precision)
{
    const size_t mm = static_cast<size_t>(m);
    const size_t es = f64_arrays(precision) ? sizeof(double) : sizeof(float);
    return 2 * align256(mm * sizeof(uint32_t)) + 2 * align256(mm * es) +
           align256(radix_scratch_bytes(m));
}

// Interpolation with curve-ordered queries and the pruned phase-1 scan: Hilbert keys of the queries
// over the dataset's box, stable radix sort, gather, phase 1 (pruned), selection and
// finalisation writing back to the caller's order; phase 2 runs on the ordered queries.
int enqueue_culled(aidw_ctx *ctx, const DatasetDev &ds, double r_exp, const Plan &pl,
                   const aidw_params &p, const void *qx, const void *qy, const Scratch &sc,
                   void *extra, void *out, float *out_alpha, int32_t *out_knn, cudaStream_t st,
                   bool profile)
{
    const AlphaMap am = alpha_map(p);
    const int64_t m = pl.m;
    const bool f64 = f64_arrays(p.precision);
    const bool xp = p.precision == AIDW_F64X;
    const size_t es = f64 ? sizeof(double) : sizeof(float);
    const size_t b4 = align256(static_cast<size_t>(m) * sizeof(uint32_t));
    const size_t bq = align256(static_cast<size_t>(m) * es);
    char *e = static_cast<char *>(extra);
    uint32_t *keys = reinterpret_cast<uint32_t *>(e);
    uint32_t *perm = reinterpret_cast<uint32_t *>(e + b4);
    void *sqx = e + 2 * b4;
    void *sqy = e + 2 * b4 + bq;
    void *sort_tmp = e + 2 * b4 + 2 * bq;
    PhaseMarks marks(ctx, st, profile);
    marks.at(0);
    bool ok;
    if (f64) {
        const double *x = static_cast<const double *>(qx), *y = static_cast<const double *>(qy);
        double *sx = static_cast<double *>(sqx), *sy = static_cast<double *>(sqy);
        ok = curve_keys_f64(x, y, m, ds.box, keys, perm, st) == cudaSuccess;
        ok = ok && radix_sort_pairs(keys, perm, m, sort_tmp, st) == cudaSuccess;
        ok = ok && gather_queries_f64(x, y, perm, m, sx, sy, st) == cudaSuccess;
        ok = ok && launch_f64_knn_cull(ds, pl, sx, sy, p.k, sc, ctx->d_err, st) == cudaSuccess;
        marks.at(1);
        ok = ok && launch_f64_select(pl, p.k, r_exp, am, sc, out_alpha, out_knn, st, perm) ==
                       cudaSuccess;
        marks.at(2);
        ok = ok && (xp ? launch_f64x_weights(ds, pl, sx, sy, sc, ctx->d_err, st)
                       : launch_f64_weights(ds, pl, sx, sy, sc, ctx->d_err, st)) == cudaSuccess;
        marks.at(3);
        ok = ok && launch_f64_finalize(pl, sc, static_cast<double *>(out), st, perm) ==
                       cudaSuccess;
    } else {
        const float *x = static_cast<const float *>(qx), *y = static_cast<const float *>(qy);
        float *sx = static_cast<float *>(sqx), *sy = static_cast<float *>(sqy);
        ok = curve_keys(x, y, nullptr, m, m, ds.box, keys, perm, st) == cudaSuccess;
        ok = ok && radix_sort_pairs(keys, perm, m, sort_tmp, st) == cudaSuccess;
        ok = ok && gather_queries(x, y, perm, m, sx, sy, st) == cudaSuccess;
        ok = ok && launch_f32_knn_cull(ds, pl, sx, sy, p.k, sc, ctx->d_err, st) == cudaSuccess;
        marks.at(1);
        ok = ok && launch_f32_select(pl, p.k, r_exp, am, sc, out_alpha, out_knn, st, sx, sy,
                                     perm) == cudaSuccess;
        marks.at(2);
        ok = ok && launch_f32_weights(ds, pl, sx, sy, sc, ctx->d_err, st) == cudaSuccess;
        marks.at(3);
        ok = ok && launch_f32_finalize(ds, pl, sc, static_cast<float *>(out), st, perm) ==
                       cudaSuccess;
    }
    if (!ok)
        return AIDW_ERR_CUDA;
    marks.at(4);
    if (profile) {
        ctx->last = aidw_kernel_times{};
        ctx->last.splits = pl.knn.splits;
        ctx->last.query_blocks = pl.knn.qblocks;
        ctx->last.launches = 4 + 14;  // + Hilbert keys, 12 radix-sort passes, gather
        ctx->last.weight_splits = pl.w.splits;
        ctx->last_valid = true;
    }
    return AIDW_OK;
}

// FP32 interpolation with the per-query (one warp per query) phase 1, in the caller's order:
// phase 1, selection, phase 2, finalisation (four launches, no query ordering).
int enqueue_warp(aidw_ctx *ctx, const DatasetDev &ds, double r_exp, const Plan &pl,
                 const aidw_params &p, const void *qx, const void *qy, const Scratch &sc,
                 void *out, float *out_alpha, int32_t *out_knn, cudaStream_t st, bool profile)
{
    PhaseMarks marks(ctx, st, profile);
    const AlphaMap am = alpha_map(p);
    bool ok;
    if (p.precision == AIDW_F32C) {
        const float *fx = static_cast<const float *>(qx), *fy = static_cast<const float *>(qy);
        marks.at(0);
        ok = launch_f32_knn_warp(ds, pl.m, fx, fy, p.k, sc, ctx->sm_count, st) == cudaSuccess;
        marks.at(1);
        ok = ok && launch_f32_select(pl, p.k, r_exp, am, sc, out_alpha, out_knn, st, fx, fy) ==
                       cudaSuccess;
        marks.at(2);
        ok = ok && launch_f32_weights(ds, pl, fx, fy, sc, ctx->d_err, st) == cudaSuccess;
        marks.at(3);
        ok = ok && launch_f32_finalize(ds, pl, sc, static_cast<float *>(out), st) == cudaSuccess;
    } else {
        const bool x = p.precision == AIDW_F64X;
        const double *dx = static_cast<const double *>(qx), *dy = static_cast<const double *>(qy);
        marks.at(0);
        ok = launch_f64_knn_warp(ds, pl, dx, dy, p.k, sc, ctx->sm_count, st) == cudaSuccess;
        marks.at(1);
        ok = ok && launch_f64_select(pl, p.k, r_exp, am, sc, out_alpha, out_knn, st) == cudaSuccess;
        marks.at(2);
        ok = ok && (x ? launch_f64x_weights(ds, pl, dx, dy, sc, ctx->d_err, st)
                      : launch_f64_weights(ds, pl, dx, dy, sc, ctx->d_err, st)) == cudaSuccess;
        marks.at(3);
        ok = ok && launch_f64_finalize(pl, sc, static_cast<double *>(out), st) == cudaSuccess;
    }
    if (!ok)
        return AIDW_ERR_CUDA;
    marks.at(4);
    if (profile) {
        ctx->last = aidw_kernel_times{};
        ctx->last.splits = 1;
        ctx->last.query_blocks = 0;
        ctx->last.launches = 4;
        ctx->last.weight_splits = pl.w.splits;
        ctx->last_valid = true;
    }
    return AIDW_OK;
}

// Host results of up to kPinnedBytes go through the context's pinned buffer: a device-to-host copy
// into pageable memory waits for the stream by itself, and so does the error word's (17 us for
// the two against 8 us for both through pinned memory and one wait).
constexpr size_t kPinnedBytes = size_t(256) << 10;

// Reads and clears the on-device error word (synchronous).
int consume_device_error(aidw_ctx *ctx, cudaStream_t st)
{
    int h = 0;
    if (cudaMemcpyAsync(&h, ctx->d_err, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess)
        return AIDW_ERR_CUDA;
    if (cudaStreamSynchronize(st) != cudaSuccess)
        return AIDW_ERR_CUDA;
    if (h) {
        cudaMemsetAsync(ctx->d_err, 0, sizeof(int), st);
        cudaStreamSynchronize(st);
        return AIDW_ERR_TIMEOUT;
    }
    return AIDW_OK;
}

// Full interpolation, host or device arrays (see aidw.h). `force_*` override the split
// counts (used by the tests to exercise split merges); 0 means "plan".
int interpolate_impl(aidw_ctx *ctx, aidw_dataset dsid, const void *qx, const void *qy,
                     int64_t m, const aidw_params *p, void *out, float *out_alpha,
                     int32_t *out_knn, cudaStream_t st, int force_knn_splits,
                     int force_w_splits, const aidw_tune_config *cfg)
{
    DatasetDev ds;
    double r_exp;
    if (!dataset_lookup(ctx, dsid, &ds, &r_exp))
        return AIDW_ERR_NOT_FOUND;
    int rc = validate_params(p, ds.n);
    if (rc)
        return rc;
    if (m < 0 || m > (int64_t(1) << 31))
        return AIDW_ERR_INVALID_ARG;
    if (m == 0)
        return AIDW_OK;
    if (!qx || !qy || !out)
        return AIDW_ERR_INVALID_ARG;
    if (cudaSetDevice(ctx->device) != cudaSuccess)
        return AIDW_ERR_CUDA;
    const bool f64 = f64_arrays(p->precision);
    const size_t es = f64 ? sizeof(double) : sizeof(float);
    const int kq = pointer_kind(qx, ctx->device), kqy = pointer_kind(qy, ctx->device);
    const int ko = pointer_kind(out, ctx->device);
    const int ka = pointer_kind(out_alpha, ctx->device);
    const int kn = pointer_kind(out_knn, ctx->device);
    if (kq < 0 || kqy < 0 || ko < 0 || ka < 0 || kn < 0)
        return AIDW_ERR_INVALID_ARG;
    const bool host_q = kq == 0 || kqy == 0;
    const bool host_any = host_q || ko == 0 || (out_alpha && ka == 0) || (out_knn && kn == 0);
    if (host_q) {
        for (int64_t i = 0; i < m; ++i) {
            const double a = f64 ? static_cast<const double *>(qx)[i]
                                 : static_cast<const float *>(qx)[i];
            const double b = f64 ? static_cast<const double *>(qy)[i]
                                 : static_cast<const float *>(qy)[i];
            if (!std::isfinite(a) || !std::isfinite(b))
                return AIDW_ERR_INVALID_ARG;
        }
    }

    // Tests force the phase-1 route: force_knn_splits -1 takes the per-query scan and -2 the
    // pruned scan (where the dataset's tile count allows it) whatever the sizes; > 0 the split
    // scan with that many splits.
    const bool force_cull =
        force_knn_splits == -2 && ds.n_pad / kTileF32Knn <= kMaxCullTiles;
    const bool warp = force_knn_splits == -1 ||
                      (force_knn_splits == 0 && use_warp_knn(p->precision, ds, m));
    // Staging for host arrays.
    const size_t b_q = (kq == 0 ? align256(m * es) : 0) + (kqy == 0 ? align256(m * es) : 0);
    const size_t b_o = ko == 0 ? align256(m * es) : 0;
    const size_t b_a = (out_alpha && ka == 0) ? align256(m * sizeof(float)) : 0;
    const size_t b_n = (out_knn && kn == 0) ? align256(m * p->k * sizeof(int32_t)) : 0;
    Plan pl;
    bool cull;
    size_t sb, total;
    void *blk = nullptr;
    bool classes = true;
    for (int w_splits = force_w_splits;;) {
        pl = make_plan(ctx, p->precision, ds.n, ds.n_pad, m, p->k, out_knn != nullptr,
                       force_knn_splits > 0 ? force_knn_splits : 0, w_splits, cfg,
                       classes ? p : nullptr, &ds);
        cull = force_cull || (!warp && force_knn_splits == 0 && use_culled_knn(ds, m, pl));
        if (cull)
            plan_culled_knn(&pl, ds.n_pad);
        if (warp) {
            // One list per query, [k][m], for the selection kernel.
            pl.knn.splits = 1;
            pl.knn.split_len = ds.n_pad;
        }
        sb = scratch_bytes(p->precision, pl, p->k) +
             (cull ? culled_extra_bytes(m, p->precision) : 0);
        total = sb + b_q + b_o + b_a + b_n;
        bool injected = false;
        rc = ctx_alloc(ctx, total, st, &blk, &injected);
        // Where the planned scratch does not fit, phase 2 in the queries' own order or with fewer
        // splits (slower, the same result within the FP32 tolerance) may.
        if (rc != AIDW_ERR_OOM || injected)
            break;
        if (pl.pow_a || pl.pow_b)
            classes = false;
        else if (force_w_splits > 0 || pl.w.splits <= 1)
            break;
        else
            w_splits = pl.w.splits / 2;
    }
    if (rc)
        return rc;
    Scratch sc;
    scratch_carve(blk, p->precision, pl, p->k, &sc);
    void *extra = static_cast<char *>(blk) + scratch_bytes(p->precision, pl, p->k);
    char *stage = static_cast<char *>(blk) + sb;
    const void *dqx = qx, *dqy = qy;
    void *dout = out;
    float *dalpha = out_alpha;
    int32_t *dknn = out_knn;
    bool ok = true;
    if (kq == 0) {
        ok &= cudaMemcpyAsync(stage, qx, m * es, cudaMemcpyHostToDevice, st) == cudaSuccess;
        dqx = stage;
        stage += align256(m * es);
    }
    if (kqy == 0) {
        ok &= cudaMemcpyAsync(stage, qy, m * es, cudaMemcpyHostToDevice, st) == cudaSuccess;
        dqy = stage;
        stage += align256(m * es);
    }
    if (ko == 0) {
        dout = stage;
        stage += b_o;
    }
    if (out_alpha && ka == 0) {
        dalpha = reinterpret_cast<float *>(stage);
        stage += b_a;
    }
    if (out_knn && kn == 0) {
        dknn = reinterpret_cast<int32_t *>(stage);
        stage += b_n;
    }
    if (!ok) {
        ctx_free(ctx, blk, total, st);
        return AIDW_ERR_CUDA;
    }
    rc = warp   ? enqueue_warp(ctx, ds, r_exp, pl, *p, dqx, dqy, sc, dout, dalpha, dknn, st,
                               ctx->profiling)
         : cull ? enqueue_culled(ctx, ds, r_exp, pl, *p, dqx, dqy, sc, extra, dout, dalpha, dknn,
                                 st, ctx->profiling)
                : enqueue_interpolation(ctx, ds, r_exp, pl, *p, dqx, dqy, sc, dout, dalpha, dknn,
                                        st, ctx->profiling);
    if (rc == AIDW_OK && host_any) {
        std::unique_lock<std::mutex> pin(ctx->pinned_mu, std::defer_lock);
        if (b_o + b_a + b_n + sizeof(int) <= kPinnedBytes && ctx->pinned && pin.try_lock()) {
            // The staged results lie together in the block; the error word follows them.
            const size_t staged = b_o + b_a + b_n;
            char *h = static_cast<char *>(ctx->pinned);
            int *herr = reinterpret_cast<int *>(h + staged);
            ok = true;
            if (staged)
                ok &= cudaMemcpyAsync(h, stage - staged, staged, cudaMemcpyDeviceToHost, st) ==
                      cudaSuccess;
            ok &= cudaMemcpyAsync(herr, ctx->d_err, sizeof(int), cudaMemcpyDeviceToHost, st) ==
                  cudaSuccess;
            ctx_free(ctx, blk, total, st);
            ok &= cudaStreamSynchronize(st) == cudaSuccess;
            if (!ok)
                return AIDW_ERR_CUDA;
            if (ko == 0)
                std::memcpy(out, h, m * es);
            if (b_a)
                std::memcpy(out_alpha, h + b_o, m * sizeof(float));
            if (b_n)
                std::memcpy(out_knn, h + b_o + b_a, m * p->k * sizeof(int32_t));
            return *herr ? consume_device_error(ctx, st) : AIDW_OK;
        }
        ok = true;
        if (ko == 0)
            ok &= cudaMemcpyAsync(out, dout, m * es, cudaMemcpyDeviceToHost, st) == cudaSuccess;
        if (out_alpha && ka == 0)
            ok &= cudaMemcpyAsync(out_alpha, dalpha, m * sizeof(float), cudaMemcpyDeviceToHost,
                                  st) == cudaSuccess;
        if (out_knn && kn == 0)
            ok &= cudaMemcpyAsync(out_knn, dknn, m * p->k * sizeof(int32_t),
                                  cudaMemcpyDeviceToHost, st) == cudaSuccess;
        if (!ok)
            rc = AIDW_ERR_CUDA;
    }
    ctx_free(ctx, blk, total, st);
    if (rc == AIDW_OK && host_any)
        rc = consume_device_error(ctx, st);
    return rc;
}

}  // namespace aidw

// =============================================================================================
// extern "C" entry points
// =============================================================================================

extern "C" {

void aidw_params_default(aidw_params *p)
{
    if (!p)
        return;
    std::memset(p, 0, sizeof(*p));
    p->k = 10;
    p->precision = AIDW_F32C;
    for (int i = 0; i < 5; ++i)
        p->alpha[i] = 1.0 + i;
    p->r_min = 0.0;
    p->r_max = 2.0;
}

const char *aidw_status_string(int s)
{
    switch (s) {
    case AIDW_OK: return "ok";
    case AIDW_PENDING: return "pending";
    case AIDW_ERR_INVALID_ARG: return "invalid argument";
    case AIDW_ERR_OOM: return "out of device memory or HBM budget";
    case AIDW_ERR_AGAIN: return "queue full, try again";
    case AIDW_ERR_TIMEOUT: return "timed out";
    case AIDW_ERR_CUDA: return "CUDA runtime error";
    case AIDW_ERR_NOT_FOUND: return "unknown handle";
    case AIDW_ERR_UNSUPPORTED: return "unsupported device or option";
    default: return "unknown status";
    }
}

int aidw_init(aidw_ctx **out, int device, size_t hbm_budget_bytes)
{
    if (!out)
        return AIDW_ERR_INVALID_ARG;
    *out = nullptr;
    int ndev = 0;
    if (cudaGetDeviceCount(&ndev) != cudaSuccess || device < 0 || device >= ndev) {
        cudaGetLastError();
        return AIDW_ERR_INVALID_ARG;
    }
    cudaDeviceProp prop;
    if (cudaGetDeviceProperties(&prop, device) != cudaSuccess)
        return AIDW_ERR_CUDA;
    if (prop.major != 10 || prop.minor != 3)
        return AIDW_ERR_UNSUPPORTED;
    if (cudaSetDevice(device) != cudaSuccess)
        return AIDW_ERR_CUDA;
    aidw_ctx *ctx = new aidw_ctx();
    ctx->device = device;
    ctx->sm_count = prop.multiProcessorCount;
    ctx->budget = hbm_budget_bytes;
    cudaMemPoolProps pp;
    std::memset(&pp, 0, sizeof(pp));
    pp.allocType = cudaMemAllocationTypePinned;
    pp.handleTypes = cudaMemHandleTypeNone;
    pp.location.type = cudaMemLocationTypeDevice;
    pp.location.id = device;
    bool ok = cudaMemPoolCreate(&ctx->pool, &pp) == cudaSuccess;
    if (ok) {
        uint64_t thr = UINT64_MAX;
        cudaMemPoolSetAttribute(ctx->pool, cudaMemPoolAttrReleaseThreshold, &thr);
    }
    ok = ok && cudaMalloc(&ctx->d_err, sizeof(int)) == cudaSuccess;
    ok = ok && cudaMemset(ctx->d_err, 0, sizeof(int)) == cudaSuccess;
    for (int i = 0; ok && i < 5; ++i)
        ok = cudaEventCreate(&ctx->ev[i]) == cudaSuccess;
    ok = ok && cudaMallocHost(&ctx->pinned, kPinnedBytes) == cudaSuccess;
    // Places aidw_interpolate_noalloc's fixed scratch array on the device now, at set-up, so
    // that its calls never load a module (and its 16 MiB) in the middle of a request.
    ok = ok && noalloc_prepare(device) == AIDW_OK;
    if (!ok) {
        cudaGetLastError();
        aidw_shutdown(ctx);
        return AIDW_ERR_CUDA;
    }
    *out = ctx;
    return AIDW_OK;
}

int aidw_shutdown(aidw_ctx *ctx)
{
    if (!ctx)
        return AIDW_ERR_INVALID_ARG;
    cudaSetDevice(ctx->device);
    serving_stop(ctx->serving);
    ctx->serving = nullptr;
    cudaDeviceSynchronize();
    for (auto &kv : ctx->datasets)
        dataset_free(kv.second.block, kv.second.pooled);
    ctx->datasets.clear();
    if (ctx->pinned)
        cudaFreeHost(ctx->pinned);
    if (ctx->d_err)
        cudaFree(ctx->d_err);
    for (int i = 0; i < 5; ++i)
        if (ctx->ev[i])
            cudaEventDestroy(ctx->ev[i]);
    if (ctx->pool)
        cudaMemPoolDestroy(ctx->pool);
    cudaGetLastError();
    delete ctx;
    return AIDW_OK;
}

int aidw_create_dataset(aidw_ctx *ctx, const void *x, const void *y, const void *z, int64_t n,
                        double area, int32_t dtype, aidw_dataset *out)
{
    if (!ctx || !x || !y || !z || !out)
        return AIDW_ERR_INVALID_ARG;
    *out = 0;
    if (n < 1 || n > (int64_t(1) << 31) - 2 * kPadPoints)
        return AIDW_ERR_INVALID_ARG;
    if (!std::isfinite(area) || !(area > 0.0))
        return AIDW_ERR_INVALID_ARG;
    if (dtype != AIDW_DTYPE_F32 && dtype != AIDW_DTYPE_F64)
        return AIDW_ERR_INVALID_ARG;
    if (cudaSetDevice(ctx->device) != cudaSuccess)
        return AIDW_ERR_CUDA;
    const int kx = pointer_kind(x, ctx->device), ky = pointer_kind(y, ctx->device);
    const int kz = pointer_kind(z, ctx->device);
    if (kx < 0 || ky < 0 || kz < 0)
        return AIDW_ERR_INVALID_ARG;
    // Device arrays may still be written on a stream that the legacy one does not wait for.
    if ((kx == 1 || ky == 1 || kz == 1) && cudaDeviceSynchronize() != cudaSuccess)
        return AIDW_ERR_CUDA;
    const size_t es = dtype == AIDW_DTYPE_F64 ? sizeof(double) : sizeof(float);
    const int64_t n_pad = (n + kPadPoints - 1) / kPadPoints * kPadPoints;
    const size_t np = static_cast<size_t>(n_pad);
    const int64_t ntiles = n_pad / kTileF32Knn;
    const int64_t nsub = n_pad / kSubTile;
    const int64_t nsuper = (ntiles + kSuperTiles - 1) / kSuperTiles;
    const size_t bytes = align256(np * sizeof(float4)) + align256(np * sizeof(float2)) +
                         align256(np * sizeof(int32_t)) + align256(np * sizeof(double2)) +
                         align256(np * sizeof(double)) + align256(ntiles * sizeof(float4)) +
                         align256(nsub * sizeof(float4)) + align256(nsuper * sizeof(float4)) +
                         align256(sizeof(float4));
    {
        std::lock_guard<std::mutex> g(ctx->mu);
        if (ctx->fail_after >= 0) {
            if (ctx->fail_after == 0) {
                ctx->fail_after = -1;
                return AIDW_ERR_OOM;
            }
            --ctx->fail_after;
        }
        if (ctx->budget && ctx->in_use + bytes > ctx->budget)
            return AIDW_ERR_OOM;
        ctx->in_use += bytes;
    }
    auto unreserve = [&]() {
        std::lock_guard<std::mutex> g(ctx->mu);
        ctx->in_use -= bytes;
    };
    void *blk = nullptr;
    bool blk_pooled = false;
    if (dataset_alloc(ctx, bytes, &blk, &blk_pooled) != cudaSuccess) {
        cudaGetLastError();
        unreserve();
        return AIDW_ERR_OOM;
    }
    // Temporary block: host-array staging (if any), unsorted FP32 copies, sort keys and values,
    // radix-sort scratch, bounding-box scratch, the call's own input check words (several threads
    // may create datasets at once).
    const size_t one = align256(static_cast<size_t>(n) * es);
    const bool stage_host = kx == 0 || ky == 0 || kz == 0;
    const size_t tmp_bytes = (stage_host ? 3 * one : 0) + align256(np * sizeof(float2)) +
                             align256(np * sizeof(float)) + 2 * align256(np * sizeof(uint32_t)) +
                             align256(radix_scratch_bytes(n_pad)) + 2 * 256;
    void *tmp = nullptr;
    bool tmp_pooled = false;
    if (dataset_alloc(ctx, tmp_bytes, &tmp, &tmp_pooled) != cudaSuccess) {
        cudaGetLastError();
        dataset_free(blk, blk_pooled);
        unreserve();
        return AIDW_ERR_OOM;
    }
    char *t = static_cast<char *>(tmp);
    const void *sx = x, *sy = y, *sz = z;
    if (stage_host) {
        if (kx == 0) {
            cudaMemcpy(t, x, n * es, cudaMemcpyHostToDevice);
            sx = t;
        }
        if (ky == 0) {
            cudaMemcpy(t + one, y, n * es, cudaMemcpyHostToDevice);
            sy = t + one;
        }
        if (kz == 0) {
            cudaMemcpy(t + 2 * one, z, n * es, cudaMemcpyHostToDevice);
            sz = t + 2 * one;
        }
        t += 3 * one;
    }
    float2 *xy32 = reinterpret_cast<float2 *>(t);
    t += align256(np * sizeof(float2));
    float *z32 = reinterpret_cast<float *>(t);
    t += align256(np * sizeof(float));
    uint32_t *keys = reinterpret_cast<uint32_t *>(t);
    t += align256(np * sizeof(uint32_t));
    uint32_t *perm = reinterpret_cast<uint32_t *>(t);
    t += align256(np * sizeof(uint32_t));
    void *sort_tmp = t;
    t += align256(radix_scratch_bytes(n_pad));
    uint32_t *box_scratch = reinterpret_cast<uint32_t *>(t);
    t += 256;
    auto *check = reinterpret_cast<unsigned long long *>(t);

    char *b = static_cast<char *>(blk);
    float4 *nxy2 = reinterpret_cast<float4 *>(b);
    b += align256(np * sizeof(float4));
    float2 *zz = reinterpret_cast<float2 *>(b);
    b += align256(np * sizeof(float2));
    int32_t *orig = reinterpret_cast<int32_t *>(b);
    b += align256(np * sizeof(int32_t));
    double2 *xy64 = reinterpret_cast<double2 *>(b);
    b += align256(np * sizeof(double2));
    double *z64 = reinterpret_cast<double *>(b);
    b += align256(np * sizeof(double));
    float4 *tbox = reinterpret_cast<float4 *>(b);
    b += align256(ntiles * sizeof(float4));
    float4 *sbox = reinterpret_cast<float4 *>(b);
    b += align256(nsub * sizeof(float4));
    float4 *upbox = reinterpret_cast<float4 *>(b);
    b += align256(nsuper * sizeof(float4));
    float4 *box = reinterpret_cast<float4 *>(b);

    int rc = AIDW_OK;
    cudaMemset(check, 0, 2 * sizeof(unsigned long long));
    const int threads = 256;
    const int blocks = static_cast<int>(std::min<int64_t>((n_pad + threads - 1) / threads,
                                                          ctx->sm_count * 8));
    if (dtype == AIDW_DTYPE_F64)
        convert_dataset_kernel<double><<<blocks, threads>>>(
            static_cast<const double *>(sx), static_cast<const double *>(sy),
            static_cast<const double *>(sz), n, n_pad, xy32, z32, xy64, z64, check);
    else
        convert_dataset_kernel<float><<<blocks, threads>>>(
            static_cast<const float *>(sx), static_cast<const float *>(sy),
            static_cast<const float *>(sz), n, n_pad, xy32, z32, xy64, z64, check);
    // Order the FP32 copy along the curve and box every tile. Non-finite inputs go through like any
    // others; the count of them is looked at once, at the end.
    unsigned long long seen[2] = {0, 0};  // non-finite inputs, largest and smallest |z|
    int log_n = 0;
    while ((int64_t(1) << log_n) < n)
        ++log_n;
    bool ok = cudaGetLastError() == cudaSuccess;
    ok = ok && bbox_of(xy32, n, box_scratch, box, 0) == cudaSuccess;
    ok = ok && curve_keys(nullptr, nullptr, xy32, n, n_pad, box, keys, perm, 0) == cudaSuccess;
    ok = ok && radix_sort_pairs(keys, perm, n_pad, sort_tmp, 0) == cudaSuccess;
    if (ok) {
        gather_dataset_kernel<<<blocks, threads>>>(xy32, z32, perm, n, n_pad,
                                                   reinterpret_cast<uint32_t *>(check + 1),
                                                   log_n, nxy2, zz, orig);
        ok = cudaGetLastError() == cudaSuccess;
    }
    ok = ok && tile_boxes(nxy2, ntiles, tbox, 0) == cudaSuccess;
    ok = ok && sub_tile_boxes(nxy2, nsub, sbox, 0) == cudaSuccess;
    ok = ok && super_tile_boxes(tbox, ntiles, nsuper, upbox, 0) == cudaSuccess;
    ok = ok && cudaMemcpy(seen, check, sizeof(seen), cudaMemcpyDeviceToHost) == cudaSuccess;
    ok = ok && cudaDeviceSynchronize() == cudaSuccess;
    if (!ok) {
        cudaGetLastError();
        rc = AIDW_ERR_CUDA;
    } else if (seen[0]) {
        rc = AIDW_ERR_INVALID_ARG;
    }
    dataset_free(tmp, tmp_pooled);
    if (rc) {
        dataset_free(blk, blk_pooled);
        unreserve();
    }
    if (ctx->budget)
        pool_trim(ctx, kPoolKeepBytes);
    if (rc)
        return rc;
    DatasetRec rec;
    rec.dev.nxy2 = nxy2;
    rec.dev.zz = zz;
    rec.dev.orig = orig;
    rec.dev.tile_box = tbox;
    rec.dev.sub_box = sbox;
    rec.dev.super_box = upbox;
    rec.dev.box = box;
    rec.dev.xy64 = xy64;
    rec.dev.z64 = z64;
    rec.dev.n = n;
    rec.dev.n_pad = n_pad;
    const auto from_bits = [](uint32_t b) {
        float f;
        std::memcpy(&f, &b, sizeof(f));
        return f;
    };
    const uint32_t z_bits = static_cast<uint32_t>(seen[1]);
    const uint32_t zn = static_cast<uint32_t>(seen[1] >> 32);
    const int z_exp = value_exponent(z_bits, log_n);
    rec.dev.z_max = from_bits(z_bits) * from_bits(pow2_bits(z_exp));
    rec.dev.z_min = zn ? from_bits(~zn) * from_bits(pow2_bits(z_exp)) : INFINITY;
    rec.dev.z_unscale = from_bits(pow2_bits(-z_exp));
    rec.block = blk;
    rec.pooled = blk_pooled;
    rec.bytes = bytes;
    rec.area = area;
    rec.r_exp = 1.0 / (2.0 * std::sqrt(static_cast<double>(n) / area));  // Eq. 2
    std::lock_guard<std::mutex> g(ctx->mu);
    const int64_t id = ctx->next_ds++;
    ctx->datasets.emplace(id, rec);
    *out = id;
    return AIDW_OK;
}

int aidw_destroy_dataset(aidw_ctx *ctx, aidw_dataset ds)
{
    if (!ctx)
        return AIDW_ERR_INVALID_ARG;
    DatasetRec rec;
    {
        std::lock_guard<std::mutex> g(ctx->mu);
        auto it = ctx->datasets.find(ds);
        if (it == ctx->datasets.end())
            return AIDW_ERR_NOT_FOUND;
        rec = it->second;
        ctx->datasets.erase(it);
    }
    cudaSetDevice(ctx->device);
    cudaDeviceSynchronize();
    dataset_free(rec.block, rec.pooled);
    {
        std::lock_guard<std::mutex> g(ctx->mu);
        ctx->in_use -= rec.bytes;
    }
    if (rec.pooled)
        pool_trim(ctx, kPoolKeepBytes);
    return AIDW_OK;
}

int aidw_dataset_info(aidw_ctx *ctx, aidw_dataset ds, int64_t *n, size_t *device_bytes)
{
    if (!ctx)
        return AIDW_ERR_INVALID_ARG;
    DatasetRec r;
    if (!ctx_dataset_copy(ctx, ds, &r))
        return AIDW_ERR_NOT_FOUND;
    if (n)
        *n = r.dev.n;
    if (device_bytes)
        *device_bytes = r.bytes;
    return AIDW_OK;
}

int aidw_interpolate(aidw_ctx *ctx, aidw_dataset ds, const void *qx, const void *qy, int64_t m,
                     const aidw_params *p, void *out, float *out_alpha, int32_t *out_knn,
                     void *stream)
{
    if (!ctx)
        return AIDW_ERR_INVALID_ARG;
    return interpolate_impl(ctx, ds, qx, qy, m, p, out, out_alpha, out_knn,
                            static_cast<cudaStream_t>(stream), 0, 0);
}

// Test hook with forced split counts (not part of the public header's contract).
int aidw_debug_interpolate_splits(aidw_ctx *ctx, aidw_dataset ds, const void *qx,
                                  const void *qy, int64_t m, const aidw_params *p, void *out,
                                  float *out_alpha, int32_t *out_knn, void *stream,
                                  int32_t knn_splits, int32_t w_splits)
{
    if (!ctx)
        return AIDW_ERR_INVALID_ARG;
    return interpolate_impl(ctx, ds, qx, qy, m, p, out, out_alpha, out_knn,
                            static_cast<cudaStream_t>(stream), knn_splits, w_splits);
}

int aidw_idw(aidw_ctx *ctx, aidw_dataset ds, const void *qx, const void *qy, int64_t m,
             double alpha, int32_t precision, void *out, void *stream)
{
    if (!ctx)
        return AIDW_ERR_INVALID_ARG;
    // Standard IDW is AIDW with five equal levels: Eq. 6 then returns alpha whatever R is.
    // One neighbour is still found, to normalise the weights and to detect coincidence.
    aidw_params p;
    aidw_params_default(&p);
    p.k = 1;
    p.precision = precision;
    for (int i = 0; i < 5; ++i)
        p.alpha[i] = alpha;
    return interpolate_impl(ctx, ds, qx, qy, m, &p, out, nullptr, nullptr,
                            static_cast<cudaStream_t>(stream), 0, 0);
}

int aidw_check_device_errors(aidw_ctx *ctx)
{
    if (!ctx)
        return AIDW_ERR_INVALID_ARG;
    cudaSetDevice(ctx->device);
    if (cudaDeviceSynchronize() != cudaSuccess)
        return AIDW_ERR_CUDA;
    return consume_device_error(ctx, 0);
}

int aidw_set_profiling(aidw_ctx *ctx, int on)
{
    if (!ctx)
        return AIDW_ERR_INVALID_ARG;
    ctx->profiling = on != 0;
    ctx->last_valid = false;
    return AIDW_OK;
}

int aidw_last_kernel_times(aidw_ctx *ctx, aidw_kernel_times *out)
{
    if (!ctx || !out)
        return AIDW_ERR_INVALID_ARG;
    if (!ctx->last_valid)
        return AIDW_ERR_NOT_FOUND;
    if (cudaEventSynchronize(ctx->ev[4]) != cudaSuccess)
        return AIDW_ERR_CUDA;
    float t[4];
    for (int i = 0; i < 4; ++i)
        cudaEventElapsedTime(&t[i], ctx->ev[i], ctx->ev[i + 1]);
    ctx->last.knn_ms = t[0];
    ctx->last.select_ms = t[1];
    ctx->last.weights_ms = t[2];
    ctx->last.finalize_ms = t[3];
    *out = ctx->last;
    return AIDW_OK;
}

int aidw_measure_pipe_rates(aidw_ctx *ctx, aidw_pipe_rates *out)
{
    if (!ctx || !out)
        return AIDW_ERR_INVALID_ARG;
    cudaSetDevice(ctx->device);
    return run_pipe_probe(ctx->sm_count, out) == cudaSuccess ? AIDW_OK : AIDW_ERR_CUDA;
}

int aidw_debug_fail_alloc_after(aidw_ctx *ctx, int64_t after)
{
    if (!ctx)
        return AIDW_ERR_INVALID_ARG;
    std::lock_guard<std::mutex> g(ctx->mu);
    ctx->fail_after = after < 0 ? -1 : after;
    return AIDW_OK;
}

}  // extern "C"

namespace aidw {
ServingRuntime *&ctx_serving(aidw_ctx *ctx)
{
    return ctx->serving;
}
std::mutex &ctx_mutex(aidw_ctx *ctx)
{
    return ctx->mu;
}
int64_t &ctx_serving_queue_limit(aidw_ctx *ctx)
{
    return ctx->serving_queue_limit;
}
}  // namespace aidw
