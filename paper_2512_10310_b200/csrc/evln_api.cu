// C-ABI entry points of libevln (contract: include/evln.h).  Host-side validation, the split
// schedule, tensor-map encoding and kernel launches; no allocation in the per-step calls.
#include "../../include/evln.h"

#include <cuda.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

#include <algorithm>
#include <mutex>
#include <new>
#include <utility>
#include <vector>

#include "attn_simt.cuh"
#include "attn_pair.cuh"
#include "attn_f32.cuh"
#include "attn_f32_small.cuh"
#include "attn_few.cuh"
#include "combine.cuh"
#include "gather_rope.cuh"
#include "common.cuh"
#include "rope_append.cuh"

using namespace evln;

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                  const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                  const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

struct evlnContext {
    int device;
    int num_sms;
    int last_cuda_error;
    int* d_status;
    EncodeTiledFn encode;
    int max_clusters[5];     // clusters of 1, 2, 4, 8, 16 blocks of the few-row kernel that fit the device at once
    int small_clusters[kSmallCluster];   // clusters of 1, 2, .. blocks of the small fp32 kernel
};

#ifdef EVLN_TIMELINE
// debug builds only (see timeline_debug.cuh): where the attention kernel leaves its clock stamps
extern "C" int evlnDebugSetTimeline(void* p)
{
    long long* v = (long long*)p;
    return (int)cudaMemcpyToSymbol(evln::g_timeline_dev, &v, sizeof(v));
}
#endif

namespace {

// Every kernel is launched with programmatic stream serialisation: its prologue may overlap the
// tail of the previous kernel in the stream; each kernel waits (griddepcontrol.wait) before it
// touches global memory.
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                       Args&&... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

// The attention kernel runs as clusters of two CTAs (one CTA pair per work item).
template <typename... KArgs, typename... Args>
cudaError_t launch_pair_pdl(void (*kernel)(KArgs...), dim3 grid, size_t smem, cudaStream_t st, Args&&... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;                 // x: two CTAs per work item
    cfg.blockDim = dim3(kTcThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = 2;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

template <typename T, int D, int RPT>
cudaError_t prepare_simt()
{
    cudaError_t e = cudaFuncSetAttribute(attn_simt_kernel<T, D, RPT, NoTable>, cudaFuncAttributeMaxDynamicSharedMemorySize, simt_smem_bytes<D, RPT>());
    if (RPT == 8 && e == cudaSuccess)
        e = cudaFuncSetAttribute(attn_simt_kernel<T, D, 8, SimtTiles>, cudaFuncAttributeMaxDynamicSharedMemorySize, simt_smem_bytes<D, 8>());
    return e;
}

template <int D>
cudaError_t prepare_f32()
{
    cudaError_t e = cudaFuncSetAttribute(attn_f32_kernel<D, NoTable>, cudaFuncAttributeMaxDynamicSharedMemorySize, F32Plan<D>::kBytes);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(attn_f32_kernel<D, SimtTiles>, cudaFuncAttributeMaxDynamicSharedMemorySize, F32Plan<D>::kBytes);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(attn_f32_small_kernel<D, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, SmallPlan<D>::kBytes);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(attn_f32_small_kernel<D, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, SmallPlan<D>::kBytes);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(attn_f32_small_kernel<D, true>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    return e;
}

template <int MT>
cudaError_t prepare_few()
{
    const void* kernels[3] = {(const void*)attn_few_kernel<MT, false, false, NoLens>, (const void*)attn_few_kernel<MT, false, true, NoLens>,
                              (const void*)attn_few_kernel<MT, true, false, BatchLens>};
    for (int i = 0; i < 3; ++i) {
        cudaError_t e = cudaFuncSetAttribute(kernels[i], cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             kFewMaxSmem);
        if (e == cudaSuccess && i < 2) e = cudaFuncSetAttribute(kernels[i], cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// Shared-memory limits of the kernels that take more than the default, on the current device.
cudaError_t prepare_kernels()
{
    const std::pair<const void*, int> tc[6] = {{(const void*)attn_pair_kernel, kTcSmemBytes},
                                               {(const void*)attn_paged_pair_kernel, kTcSmemBytes},
                                               {(const void*)attn_persistent_kernel<false, NoLens>, kPersistSmemBytes},
                                               {(const void*)attn_persistent_kernel<true, PagedLens>, kPersistSmemBytes},
                                               {(const void*)attn_solo_kernel, kSoloSmemBytes},
                                               {(const void*)attn_packed_kernel, kPersistSmemBytes}};
    for (const auto& k : tc) {
        cudaError_t e = cudaFuncSetAttribute(k.first, cudaFuncAttributeMaxDynamicSharedMemorySize, k.second);
        if (e != cudaSuccess) return e;
    }
    cudaError_t e = prepare_few<1>();
    if (e == cudaSuccess) e = prepare_few<2>();
    if (e == cudaSuccess) e = prepare_f32<128>();
    if (e == cudaSuccess) e = prepare_f32<64>();
    if (e == cudaSuccess) e = prepare_simt<float, 128, 8>();
    if (e == cudaSuccess) e = prepare_simt<float, 128, 2>();
    if (e == cudaSuccess) e = prepare_simt<float, 64, 8>();
    if (e == cudaSuccess) e = prepare_simt<float, 64, 2>();
    if (e == cudaSuccess) e = prepare_simt<__nv_bfloat16, 128, 8>();
    if (e == cudaSuccess) e = prepare_simt<__nv_bfloat16, 128, 2>();
    if (e == cudaSuccess) e = prepare_simt<__nv_bfloat16, 64, 8>();
    if (e == cudaSuccess) e = prepare_simt<__nv_bfloat16, 64, 2>();
    return e;
}

// The attention kernels move registers between their warpgroups (setmaxnreg) inside the pool a CTA
// gets at launch; a request the pool cannot serve would wait for ever.  The plan in attn_pair.cuh is
// made for kRegsLaunch registers per thread: refuse to run a build that came out differently.
bool attention_register_pool_ok()
{
    cudaFuncAttributes fa;
    const void* kernels[6] = {(const void*)attn_pair_kernel, (const void*)attn_paged_pair_kernel, (const void*)attn_persistent_kernel<false, NoLens>, (const void*)attn_persistent_kernel<true, PagedLens>,
                              (const void*)attn_solo_kernel, (const void*)attn_packed_kernel};
    for (const void* k : kernels) {
        if (cudaFuncGetAttributes(&fa, k) != cudaSuccess) return false;
        if (fa.numRegs != kRegsLaunch) return false;
    }
    return true;
}

inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }
inline size_t round_up(size_t x, size_t a) { return (x + a - 1) / a * a; }
inline bool overlap(const void* a, size_t a_bytes, const void* b, size_t b_bytes)
{
    const uintptr_t x = reinterpret_cast<uintptr_t>(a), y = reinterpret_cast<uintptr_t>(b);
    return a_bytes > 0 && b_bytes > 0 && x < y + b_bytes && y < x + a_bytes;
}
inline int elem_bytes(int dtype) { return dtype == EVLN_BF16 ? 2 : 4; }

evlnStatus_t cuda_fail(evlnHandle_t h, cudaError_t e)
{
    h->last_cuda_error = (int)e;
    return EVLN_CUDA_ERROR;
}

// The handle's device must be current when work is launched: the kernels' attributes and the
// tensor maps belong to that device's context.
bool device_is_current(evlnHandle_t h)
{
    int dev = -1;
    return cudaGetDevice(&dev) == cudaSuccess && dev == h->device;
}

// An optional position table must cover the positions [first, first + count) of the call.
bool rope_table_covers(const void* table, int table_first, int table_count, long first, long count)
{
    if (!table) return true;
    if (!aligned16(table) || table_first < 0 || table_count < 0) return false;
    return (long)table_first <= first && first + count <= (long)table_first + table_count;
}

evlnStatus_t check_step_params(evlnHandle_t h, const evlnStepParams* p)
{
    if (!h || !p) return EVLN_INVALID_VALUE;
    if (p->struct_size != sizeof(evlnStepParams)) return EVLN_INVALID_VALUE;
    if (p->dtype != EVLN_BF16 && p->dtype != EVLN_F32) return EVLN_INVALID_VALUE;
    if (p->num_q_heads <= 0 || p->num_kv_heads <= 0 || p->num_q_heads % p->num_kv_heads != 0)
        return EVLN_INVALID_VALUE;
    if (p->cache_len < 0 || p->num_new < 0 || p->cache_capacity < 0) return EVLN_INVALID_VALUE;
    if (!(p->rope_theta > 0.0) || !(p->softmax_scale >= 0.f)) return EVLN_INVALID_VALUE;
    if (p->num_splits < 0 || p->num_splits > kMaxSplits) return EVLN_INVALID_VALUE;
    if (p->kernel != EVLN_KERNEL_AUTO && p->kernel != EVLN_KERNEL_SIMT) return EVLN_INVALID_VALUE;
    if (p->head_dim != 64 && p->head_dim != 128) return EVLN_NOT_SUPPORTED;
    if ((long)p->cache_len + p->num_new > (long)p->cache_capacity) return EVLN_CACHE_FULL;
    if ((long)p->num_new * p->num_q_heads / p->num_kv_heads > (1 << 24)) return EVLN_NOT_SUPPORTED;
    if (!rope_table_covers(p->rope_table, p->rope_table_first_pos, p->rope_table_count, p->cache_len, p->num_new))
        return EVLN_INVALID_VALUE;
    return EVLN_OK;
}

// fp32 on the tensor cores (attn_f32.cuh), unless the caller asks for the kernel without them, or for a softmax scale with which scores of
// ordinary size come from queries and keys whose products leave the range of floats (2^-60 to 2^60 keep them far from it).
inline bool use_f32_kernel(const evlnStepParams* p)
{
    const bool ordinary = p->softmax_scale == 0.f || (p->softmax_scale >= 0x1p-60f && p->softmax_scale <= 0x1p60f);
    return p->kernel == EVLN_KERNEL_AUTO && p->dtype == EVLN_F32 && ordinary;
}

inline bool use_tensor_kernel(const evlnStepParams* p)
{
    return p->kernel == EVLN_KERNEL_AUTO && p->dtype == EVLN_BF16 && p->head_dim == 128;
}

// Cost model of the split-KV schedule of the tensor-core kernel: work items (unit x split) run
// in waves of one CTA pair per two SMs, each walks ceil(nkv / S) KV tiles plus a fixed
// prologue/epilogue; every split adds combine traffic, the first one the merge that a step of one call does not need
// unsplit.  The three calls run a combine either way, and both forms use the same split count, so the price lies
// between what the two would like: it grows with the rows that a merge moves, up to 4 tiles.  (Measured over 0 .. 1500
// cached keys, 40 .. 256 new tokens, five head shapes, both forms: 1.2 % above the best split count on average.  With 4
// tiles for any number of rows three calls took up to 30 % more: 40 tokens of the 7B shape over 700 12.5 us
// unsplit, 10.6 in three splits; without a price one call took up to 33 % more: 196 tokens over 256 12.6 us in two
// splits, 10.6 unsplit.)
int choose_splits_tc(int units_total, long rows_total, int nkv_max, int nkv_min, int num_sms)
{
    int best = 1;
    double best_cost = 1e30;
    const int pairs = num_sms / 2 > 0 ? num_sms / 2 : 1;
    const double merge = std::min(4.0, 1.0 + 7e-4 * rows_total);
    const int smax = nkv_min < kMaxSplits ? (nkv_min < 1 ? 1 : nkv_min) : kMaxSplits;
    for (int s = 1; s <= smax; ++s) {
        const double waves = ceil((double)units_total * s / pairs);
        // per work item: set-up, first-tile latency, partial write-out and teardown cost about as
        // much as 7 KV tiles (measured); every split adds about half a tile of combine work
        const double cost = waves * (ceil((double)nkv_max / s) + 7.0) + (s > 1 ? merge : 0.0) + 0.5 * s;
        if (cost < best_cost - 1e-9) { best_cost = cost; best = s; }
    }
    return best;
}

// A step whose rows per kv head fit one 128-row tile (a few new tokens: the action tokens after a
// frame) runs one CTA per (kv head, split) instead of CTA pairs.
inline bool use_solo_kernel(const evlnStepParams* p)
{
    return use_tensor_kernel(p) && (long)p->num_new * (p->num_q_heads / p->num_kv_heads) <= kTileM;
}

// Short unsplit steps whose 128-row tiles leave SMs idle: a CTA per tile instead of a pair per two, which have not to meet
// before they start nor at the end, and of which the first need fewer key tiles.  (28 layers, 7B shape: 256 tokens on an empty cache 271 us a
// pass with pairs, 265 so; 400 359 and 357; 196 over 256 306 and 303.  For long walks the pairs' halved K/V traffic is worth more: 196
// tokens over 4096 keys 15.8 us a layer and 16.8.)
inline bool use_single_ctas(evlnHandle_t h, const evlnStepParams* p, int splits)
{
    const int G = p->num_q_heads / p->num_kv_heads, tiles = ceil_div(p->num_new * G, kTileM);
    return splits == 1 && (long)tiles * p->num_kv_heads <= h->num_sms && ceil_div(p->cache_len + p->num_new, kTileN) <= 4;
}

// Split schedule of the one-CTA-per-item kernel, in microseconds: a CTA takes 0.9 per KV tile unless HBM (all
// of K and V at most of its rate) takes longer, and a split adds partials of every row to write and merge.
// (Measured over 500 .. 32000 cached keys, 4 and 8 kv heads, 35 .. 128 rows each: within 3 % of the best split
// count everywhere, 0.2 % on average.  Spreading over as many SMs as there are cost up to 19 % with 8 kv
// heads: 8 tokens over 4292 keys 15.1 us with 18 splits, 12.7 with 12.)
int choose_splits_solo(int Hkv, int R, int T, int num_sms)
{
    const int nkv = ceil_div(T, kTileN);
    const double hbm_us = 512.0 * T * Hkv / 6.4e6, split_us = 0.1 + 1e-4 * R * Hkv;
    int best = 1;
    double best_cost = 1e30;
    const int smax = nkv < kMaxSplits ? (nkv < 1 ? 1 : nkv) : kMaxSplits;
    for (int s = 1; s <= smax; ++s) {
        const double waves = ceil((double)Hkv * s / num_sms), work = 0.9 * waves * ceil_div(nkv, s);
        const double cost = (work > 0.8 * hbm_us ? work : 0.8 * hbm_us) + split_us * s;
        if (cost < best_cost - 1e-9) { best_cost = cost; best = s; }
    }
    return best;
}

// At most 32 rows per kv head (up to four action tokens with seven query heads per kv head): the kernel
// whose products stay in registers (attn_few.cuh).  Not with two row tiles where clusters of 16 blocks for all heads do
// not fit the device at once, or do not cover it: mma.sync on half of the SMs is slower than the one-CTA kernel on all of
// them.  Eight and more kv heads, from 3072 keys on: 32 rows of 8 heads 4292 keys 12.4 us against 11.4 (of 16 heads
// 14.9 and 13.3), 20656 keys 21.3 and 19.3; 1500 keys 9.5 and 9.9.  From 24576 keys on also four heads with more than 24
// rows (28 rows, 32768 keys 19.3 and 18.0; 21 rows, 28000 keys 16.0 and 16.6; seven heads 21.9 and 22.8), and
// four to seven heads with too many tokens for the one-launch step (17 rows of 6 heads, 32768 keys 25.4 and 22.9).
// A caller who passes on the split count that evlnStepNumSplits reports gets the library's own kernel; one who asks
// for so few that they leave half of the SMs idle gets the few-row kernel, whose clusters fill them (64 query heads, 4
// tokens over 9000 keys in one split 16.2 us against 59.6; 8 tokens of 32 query heads over 8000 keys in 12 splits 15.3
// and 14.3).
inline bool use_few_kernel(evlnHandle_t h, const evlnStepParams* p)
{
    const int Hkv = p->num_kv_heads, keys = p->cache_len + p->num_new;
    const long rows = (long)p->num_new * (p->num_q_heads / Hkv);
    if (!use_tensor_kernel(p) || rows > kFewRows) return false;
    if (rows <= 16 || Hkv < 4 || keys < (Hkv >= 8 ? 3072 : 24576)) return true;
    if (Hkv < 8 && p->num_new <= kFewFusedTokens && (Hkv > 4 || rows <= 24)) return true;
    return p->num_splits > 0 && (long)p->num_splits * Hkv <= h->num_sms / 2 &&
           p->num_splits < choose_splits_solo(Hkv, (int)rows, keys, h->num_sms);
}
inline int few_row_tiles(int rows) { return rows <= 16 ? 1 : 2; }

struct FewPlan {
    int splits, cluster, stages;
};
// A block needs 0.40 us per 64-key stage (0.54 with two row tiles), all of them together what HBM needs;
// clusters beyond those that fit the device at once wait for a whole round; a cluster costs 1 us of
// exchange, splits a second launch that merges them (measured with 4 and 8 kv heads, 40 .. 32768 keys).
FewPlan few_plan(evlnHandle_t h, const evlnStepParams* p)
{
    const int T = p->cache_len + p->num_new, ns = ceil_div(T, kFewKeys);
    const int rows = p->num_new * (p->num_q_heads / p->num_kv_heads);
    const double stage_us = few_row_tiles(rows) == 1 ? 0.40 : 0.54;
    const double hbm_us = 512.0 * T * p->num_kv_heads / 6.2e6;
    FewPlan best = {1, 1, 0};
    double best_cost = 1e30;
    for (int i = 0; i < 5; ++i) {
        const int c = 1 << i;
        for (int s = p->num_splits > 0 ? p->num_splits : 1; s <= (p->num_splits > 0 ? p->num_splits : 8); ++s) {
            if ((c > 1 || s > 1) && c * s > ns && !(c == 1 && s == p->num_splits)) continue;
            const long clusters = (long)p->num_kv_heads * s;
            const int fit = h->max_clusters[i] > 0 ? h->max_clusters[i] : 0;
            if (fit == 0) continue;
            const double rounds = (double)((clusters + fit - 1) / fit);
            const double work = rounds * ceil_div(ns, c * s) * stage_us;
            const double cost = (work > hbm_us ? work : hbm_us) + rounds + (c > 1 ? 1.0 : 0.0) + (s > 1 ? 1.8 + 0.1 * s : 0.0);
            if (cost < best_cost - 1e-9) { best_cost = cost; best.splits = s; best.cluster = c; }
        }
    }
    best.stages = few_smem_bytes(kFewMaxStages, rows, best.cluster, true, p->num_new) <= kFewMaxSmem ? kFewMaxStages : kFewMinStages;
    return best;
}

// How many clusters of each size of the largest few-row block the current device holds at once.
cudaError_t query_few_clusters(int* max_clusters)
{
    for (int i = 0; i < 5; ++i) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(1u << i);
        cfg.blockDim = dim3(kFewThreads);
        cfg.dynamicSmemBytes = kFewMaxSmem;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = 1u << i;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        int n = 0;
        cudaError_t e = cudaOccupancyMaxActiveClusters(&n, attn_few_kernel<2, false, true, NoLens>, &cfg);
        if (e != cudaSuccess) {
            if (i == 0) return e;
            cudaGetLastError();            // this cluster size is not available
            n = 0;
        }
        max_clusters[i] = n;
    }
    return cudaSuccess;
}

// The same for the small fp32 kernel, clusters of 1 .. kSmallCluster.
cudaError_t query_small_clusters(int* max_clusters)
{
    for (int i = 0; i < kSmallCluster; ++i) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(i + 1);
        cfg.blockDim = dim3(kSmallThreads);
        cfg.dynamicSmemBytes = SmallPlan<128>::kBytes;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = i + 1;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        int n = 0;
        const cudaError_t e = cudaOccupancyMaxActiveClusters(&n, attn_f32_small_kernel<128, true>, &cfg);
        if (e != cudaSuccess) {
            if (i == 0) return e;
            cudaGetLastError();            // this cluster size is not available
            n = 0;
        }
        max_clusters[i] = n;
    }
    return cudaSuccess;
}

template <bool FUSED>
cudaError_t launch_few(const FewPlan& f, int rows, cudaStream_t st, const CUtensorMap& tm_k, const CUtensorMap& tm_v, const FewArgs& a)
{
    cudaLaunchConfig_t cfg = {};
    const int mt = few_row_tiles(rows);
    cfg.gridDim = dim3(f.cluster, a.Hkv, f.splits);
    cfg.blockDim = dim3(kFewThreads);
    cfg.dynamicSmemBytes = few_smem_bytes(f.stages, rows, f.cluster, FUSED, a.num_new);
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = f.cluster;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = f.cluster > 1 ? 2 : 1;
    const NoLens nl = {};
    if (mt == 1) return cudaLaunchKernelEx(&cfg, attn_few_kernel<1, false, FUSED, NoLens>, tm_k, tm_v, a, nl);
    return cudaLaunchKernelEx(&cfg, attn_few_kernel<2, false, FUSED, NoLens>, tm_k, tm_v, a, nl);
}

size_t partial_bytes(int splits, int Hkv, long rows, int D)
{
    return round_up((size_t)splits * Hkv * rows * (D + 1) * sizeof(float), 256);
}

// Row tile and split count of the SIMT and fp32 kernels (splits > 0: given), by a model of measured times at
// head_dim 128 (head_dim 64: about half).  SIMT: a block of 128 rows runs alone on its SM, 13.3 us per 64-key
// tile and 7 us for its start and write-out; a block of 32 rows takes 6.3 us per tile and 5 us when it
// has the SM to itself, 9.5 per tile when two share it.  So 128-row tiles are 1.4 times cheaper per row
// where they fill the chip, 32-row tiles have twice the latency advantage where they would not.  A
// split writes and re-reads a set of partials (about 5 TB/s out of L2).
// fp32 runs on the tensor cores: 128-row tiles (attn_f32.cuh) take 2.25 us per 64-key tile (1.5 at head_dim 64) and 3 us more
// for their start than the others; 32-row blocks (attn_f32_small.cuh) 3.7 us per tile (1.8), and evlnStep in one launch
// where the blocks' rotations are not too many, which saves two launches of about 2 us each and the partials' round
// trip.  So 128-row tiles begin where 32-row blocks would be walked for three tiles or more.  (One call, us: 64 tokens of 2
// heads over 256 keys 9.6 with three launches of float FMAs, 7.9; 34 tokens of 28 heads over 518 keys 18.2 with float FMAs, 16.5 in
// 128-row tiles, 17.1 in one launch; 243 tokens of 2 heads over 373 keys 18.5, 16.5 and, 32 rows in three launches, 14.1.)
struct SimtSchedule {
    int rows_per_thread, splits;
    int share;               // > 0: one block per SM, each that many key tiles of 128-row blocks (see attn_simt.cuh)
    bool one_launch;         // fp32 in 32-row blocks: evlnStep is one launch
};
// The row blocks' key tiles, at most kSimtShareBlocks blocks.
void fill_simt_tiles(const evlnStepParams* p, SimtTiles* t)
{
    const int G = p->num_q_heads / p->num_kv_heads, R = p->num_new * G, blocks = ceil_div(R, 128);
    t->off[0] = 0;
    for (int rb = 0; rb < kSimtShareBlocks; ++rb) {
        const int last = 128 * (rb + 1) < R ? 128 * (rb + 1) - 1 : R - 1;
        t->off[rb + 1] = t->off[rb] + (rb < blocks ? ceil_div(p->cache_len + last / G + 1, kSimtKeys) : 0);
    }
}
// Most tokens whose angles a block of the small fp32 kernel forms in a one-launch step: its rows' and its share of the new ones.
inline int f32_angle_tokens(const evlnStepParams* p, int splits)
{
    const int G = p->num_q_heads / p->num_kv_heads, own = std::min((kSmallRows + G - 2) / G + 1, p->num_new);
    return std::min(own + ceil_div(p->num_new, splits), p->num_new);
}
// (most_splits: bound on the splits of the library's own choice)
SimtSchedule simt_schedule(evlnHandle_t h, const evlnStepParams* p, int splits, int most_splits = kMaxSplits)
{
    const int R = p->num_new * (p->num_q_heads / p->num_kv_heads);
    const int tiles = ceil_div(p->cache_len + p->num_new, kSimtKeys);
    const double d = p->head_dim / 128.0;
    const double split_us = 0.3 + 2.0 * R * p->num_kv_heads * p->head_dim * 4 / 5e6;
    // (Steps of more row blocks than the share table holds keep the split counts, and by that the workspaces, of the
    // kernel without tensor cores.)
    const bool tensor = use_f32_kernel(p) && ceil_div(R, 128) <= kSimtShareBlocks;
    const double big_tile = tensor ? 0.75 / d + 1.5 : 13.3, big_start = tensor ? 7.1 + 2.8 * d : 7.0;
    SimtSchedule best = {8, splits > 0 ? splits : 1, 0, false};
    double best_cost = 1e30;
    const int smax = tiles < most_splits ? tiles : most_splits;
    for (int rpt = 8; rpt >= 2; rpt -= 6) {
        const long row_blocks = (long)ceil_div(R, 16 * rpt) * p->num_kv_heads;
        if (use_f32_kernel(p) && !tensor && rpt != 8) break;
        for (int s = splits > 0 ? splits : 1; s <= (splits > 0 ? splits : smax); ++s) {
            const long blocks = row_blocks * s;
            double cost;
            bool one_launch = false;
            if (tensor && rpt == 2) {
                const double block_us = ceil_div(tiles, s) * (3.8 * d - 0.1) + 1.0;
                cost = (double)((blocks + h->num_sms - 1) / h->num_sms) * block_us + 6.0 + (split_us - 0.2) * s;
                const int tokens = f32_angle_tokens(p, s), fit = tokens <= kSmallAngleTokens && s <= kSmallCluster ? h->small_clusters[s - 1] : 0;
                if (fit > 0) {
                    // what a thread rotates, in vectors, and the angles it forms for that (with a table or without: the split count, and
                    // by that the result's bits, are the same)
                    const double items = (std::min(R, kSmallRows) + 3.0 * ceil_div(p->num_new, s)) * d / 16.0, angles = tokens * d / 4.0;
                    const double one = (double)((row_blocks + fit - 1) / fit) * (block_us + 0.4 * items + 0.4 * angles) + 3.0 + 0.05 * s;
                    if (one < cost) { cost = one; one_launch = true; }
                }
            } else {
                const long at_once = rpt == 8 || blocks <= h->num_sms ? h->num_sms : 2 * h->num_sms;
                const double tile_us = rpt == 8 ? big_tile : at_once == h->num_sms ? 6.3 : 9.5;
                const double waves = (double)((blocks + at_once - 1) / at_once);
                cost = waves * (ceil_div(tiles, s) * tile_us * d + (rpt == 8 ? big_start : 5.0)) + split_us * s;
            }
            if (cost < best_cost - 1e-9) { best_cost = cost; best = {rpt, s, 0, one_launch}; }
        }
    }
    if (splits == 0 && ceil_div(R, 128) <= kSimtShareBlocks && (long)ceil_div(R, 128) * p->num_kv_heads * tiles > h->num_sms) {
        // equal shares: no block waits for another's last tile, but most go over the end of a row block (start and
        // write-out of another one) and a row gets up to one split more
        SimtTiles t;
        fill_simt_tiles(p, &t);
        const int per_head = t.off[kSimtShareBlocks], blocks = ceil_div(R, 128), most = t.off[blocks] - t.off[blocks - 1];
        int share = ceil_div(per_head * p->num_kv_heads, h->num_sms);
        if (share < ceil_div(most, kMaxSplits - 1)) share = ceil_div(most, kMaxSplits - 1);
        const int s = ceil_div(most - 1, share) + 1;
        const double cost = share * big_tile * d + big_start + (tensor ? 5.0 : 4.0) * ceil_div(share, t.off[1]) + split_us * (1.0 + (double)most / share);
        if (s <= most_splits && cost < best_cost - 1e-9) best = {8, s, share, false};
    }
    return best;
}

template <typename T, int D>
void launch_simt(const SimtSchedule& plan, const evlnStepParams* p, dim3 grid, cudaStream_t st, const SimtAttnArgs& a)
{
    if (plan.share > 0) {
        SimtTiles t;
        fill_simt_tiles(p, &t);
        const int blocks = ceil_div(t.off[kSimtShareBlocks] * p->num_kv_heads, plan.share);
        launch_pdl(attn_simt_kernel<T, D, 8, SimtTiles>, dim3(blocks), dim3(kSimtThreads), simt_smem_bytes<D, 8>(), st, a, t);
    } else if (plan.rows_per_thread == 8) {
        launch_pdl(attn_simt_kernel<T, D, 8, NoTable>, grid, dim3(kSimtThreads), simt_smem_bytes<D, 8>(), st, a, NoTable{});
    } else {
        launch_pdl(attn_simt_kernel<T, D, 2, NoTable>, grid, dim3(kSimtThreads), simt_smem_bytes<D, 2>(), st, a, NoTable{});
    }
}

// The scale of the fp32 kernels in two floats each.
void set_f32_scale(const evlnStepParams* p, SimtAttnArgs* a)
{
    const double scale = p->softmax_scale > 0.f ? (double)p->softmax_scale : 1.0 / sqrt((double)p->head_dim);
    const double scale2 = scale * 1.4426950408889634;
    a->scale = (float)scale;
    a->scale_lo = (float)(scale - (double)a->scale);
    a->scale2_hi = (float)scale2;
    a->scale2_lo = (float)(scale2 - (double)a->scale2_hi);
    a->diff_min = kLeastWeight / a->scale2_hi;
    const float huge = 0x1p90f / std::max(a->scale, 1.f);
    uint32_t bits;
    memcpy(&bits, &huge, sizeof(bits));
    a->huge = bits >> 16;
}

template <int D>
void launch_f32(const SimtSchedule& plan, const evlnStepParams* p, dim3 grid, cudaStream_t st, SimtAttnArgs a)
{
    set_f32_scale(p, &a);
    if (plan.rows_per_thread == 2) {
        launch_pdl(attn_f32_small_kernel<D, false>, dim3(grid.z, grid.x, grid.y), dim3(kSmallThreads), SmallPlan<D>::kBytes, st, a,
                   make_fast_div((uint32_t)a.G), F32Fused{});
    } else if (plan.share > 0) {
        SimtTiles t;
        fill_simt_tiles(p, &t);
        const int blocks = ceil_div(t.off[kSimtShareBlocks] * p->num_kv_heads, plan.share);
        launch_pdl(attn_f32_kernel<D, SimtTiles>, dim3(blocks), dim3(kF32Threads), F32Plan<D>::kBytes, st, a, t);
    } else {
        launch_pdl(attn_f32_kernel<D, NoTable>, grid, dim3(kF32Threads), F32Plan<D>::kBytes, st, a, NoTable{});
    }
}

// The whole step in one launch: a cluster per (row block, kv head), a block per split.
template <int D>
cudaError_t launch_f32_step(const evlnStepParams* p, int splits, cudaStream_t st, SimtAttnArgs a, const F32Fused& f)
{
    set_f32_scale(p, &a);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(splits, ceil_div(a.num_new * a.G, kSmallRows), a.Hkv);
    cfg.blockDim = dim3(kSmallThreads);
    cfg.dynamicSmemBytes = SmallPlan<D>::kBytes;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = splits;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, attn_f32_small_kernel<D, true>, a, make_fast_div((uint32_t)a.G), f);
}

int resolve_splits(evlnHandle_t h, const evlnStepParams* p)
{
    if (p->num_new == 0) return 1;
    if (p->num_splits > 0) return p->num_splits;
    const int G = p->num_q_heads / p->num_kv_heads;
    const int R = p->num_new * G;
    const int T = p->cache_len + p->num_new;
    if (use_few_kernel(h, p)) return few_plan(h, p).splits;
    if (use_solo_kernel(p))
        return choose_splits_solo(p->num_kv_heads, R, T, h->num_sms);
    if (use_tensor_kernel(p)) {
        const int units = ceil_div(R, kUnitRows);
        const int nkv_max = unit_kv_tiles(p->cache_len, p->num_new, G, units - 1, kUnitRows);
        const int nkv_min = unit_kv_tiles(p->cache_len, p->num_new, G, 0, kUnitRows);
        return choose_splits_tc(units * p->num_kv_heads, (long)R * p->num_kv_heads, nkv_max, nkv_min, h->num_sms);
    }
    return simt_schedule(h, p, 0).splits;
}

bool encode_map(evlnHandle_t h, CUtensorMap* map, const void* base, int rank, const cuuint64_t* dims,
                const cuuint64_t* strides_bytes, const cuuint32_t* box)
{
    cuuint32_t ones[5] = {1, 1, 1, 1, 1};
    CUresult r = h->encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, (cuuint32_t)rank, const_cast<void*>(base),
                           dims, strides_bytes, box, ones, CU_TENSOR_MAP_INTERLEAVE_NONE,
                           CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

evlnStatus_t check_paged_params(evlnHandle_t h, const evlnPagedParams* p, const int* lens, const int* offs)
{
    if (!h || !p || !lens || !offs) return EVLN_INVALID_VALUE;
    if (p->struct_size != sizeof(evlnPagedParams)) return EVLN_INVALID_VALUE;
    if (p->num_q_heads <= 0 || p->num_kv_heads <= 0 || p->num_q_heads % p->num_kv_heads != 0)
        return EVLN_INVALID_VALUE;
    if (p->batch < 1 || p->num_pages < 1 || p->max_pages_per_seq < 1 || p->kv_chunk_tiles < 0)
        return EVLN_INVALID_VALUE;
    if (!(p->rope_theta > 0.0) || !(p->softmax_scale >= 0.f)) return EVLN_INVALID_VALUE;
    if (p->dtype != EVLN_BF16 || p->head_dim != 128 || p->page_size != 64 || p->batch > kMaxBatch)
        return EVLN_NOT_SUPPORTED;
    if (offs[0] != 0) return EVLN_INVALID_VALUE;
    for (int b = 0; b < p->batch; ++b) {
        if (lens[b] < 0 || offs[b + 1] < offs[b]) return EVLN_INVALID_VALUE;
        const long tokens = (long)lens[b] + (offs[b + 1] - offs[b]);
        if ((tokens + p->page_size - 1) / p->page_size > p->max_pages_per_seq) return EVLN_CACHE_FULL;
        if (!rope_table_covers(p->rope_table, p->rope_table_first_pos, p->rope_table_count, lens[b], offs[b + 1] - offs[b]))
            return EVLN_INVALID_VALUE;
    }
    if ((long)offs[p->batch] * p->num_q_heads / p->num_kv_heads > (1 << 24)) return EVLN_NOT_SUPPORTED;
    return EVLN_OK;
}

// KV tiles of unit u of a batch item: paged episode, or item sharing a cache prefix (tail).
inline int batch_kv_tiles(bool tail, int L, int n, int G, int u)
{
    return tail ? tail_kv_tiles(L, n, G, u, kUnitRows) : unit_kv_tiles(L, n, G, u, kUnitRows);
}

// Episodes by length, longest first (equal lengths in the caller's order).
void longest_first(int batch, const int* lens, const int* offs, int* order)
{
    for (int b = 0; b < batch; ++b) order[b] = b;
    std::stable_sort(order, order + batch, [&](int x, int y) {
        return lens[x] + offs[x + 1] - offs[x] > lens[y] + offs[y + 1] - offs[y];
    });
}

// When the last of `pairs` CTA pairs is done (in KV tiles) if each takes the next work item as it becomes free,
// episodes in the order given, items of at most `chunk` tiles.  The pairs are kept as runs of equal load
// (ascending), so an episode costs a few steps however many items it has.
constexpr int kMaxPairs = 128;
constexpr int kNextItemTiles = 5;        // from a pair's last product of an item to the first of its next one, in KV tiles
constexpr double kSplitTiles = 0.3;      // what a split adds to the merge of its rows, in KV tiles
double finish_time(int pairs, int G, int Hkv, int batch, const int* lens, const int* offs, const int* order, int chunk)
{
    struct Run { double load; int count; } runs[kMaxPairs];
    int num = 1;
    runs[0] = Run{0.0, pairs < kMaxPairs ? pairs : kMaxPairs};
    for (int i = 0; i < batch; ++i) {
        const int b = order[i], n = offs[b + 1] - offs[b];
        if (n == 0) continue;
        const int units = ceil_div(n * G, kUnitRows);
        // (a row unit further on may need a tile more, and by that a split more)
        for (int u = 0, same; u < units; u += same) {
            const int nkv = unit_kv_tiles(lens[b], n, G, u, kUnitRows), splits = ceil_div(nkv, chunk);
            for (same = 1; u + same < units && unit_kv_tiles(lens[b], n, G, u + same, kUnitRows) == nkv;) ++same;
            const double cost = (double)nkv / splits + kNextItemTiles;
            for (long left = (long)same * Hkv * splits; left > 0;) {
                const int take = left < runs[0].count ? (int)left : runs[0].count;
                const double load = runs[0].load + cost;
                left -= take;
                runs[0].count -= take;
                int at = 0;
                if (runs[0].count == 0) {              // the lowest run moves up: close its place while looking
                    --num;
                    for (; at < num && runs[at + 1].load < load; ++at) runs[at] = runs[at + 1];
                    if (at < num && runs[at + 1].load == load) {
                        runs[at + 1].count += take;
                        for (int k = at; k < num; ++k) runs[k] = runs[k + 1];
                    } else {
                        runs[at] = Run{load, take};
                        ++num;
                    }
                } else {
                    while (at < num && runs[at].load < load) ++at;
                    if (at < num && runs[at].load == load) {
                        runs[at].count += take;
                    } else {
                        for (int k = num; k > at; --k) runs[k] = runs[k - 1];
                        runs[at] = Run{load, take};
                        ++num;
                    }
                }
            }
        }
    }
    return runs[num - 1].load;
}

// Work-item size of a batch on CTA pairs.  Not splitting saves the partials (an fp32 row set per split written
// and read again against one rounded row set) and the items' fixed costs; splitting evens out the pairs.  Many
// items even out by themselves (longest first); else the estimate above decides how often the longest
// episode is split.  Measured: 16 ragged episodes of one frame (384 unsplit items) 480 us with items of a quarter
// of a pair's share, 428 unsplit; episodes of 4000 and 1000 tokens 42 us, 28 with the longer one split in two;
// of 16384 and 8000 tokens 104 and 91 (three and two ways); four of 4000 .. 16000 tokens 128 unsplit, 105 in up to four.
int choose_chunk(int pairs, int G, int Hkv, int batch, const int* lens, const int* offs, const int* order, int nkv_max)
{
    long unsplit = 0, tiles = 0;
    for (int b = 0; b < batch; ++b) {
        const int n = offs[b + 1] - offs[b], units = ceil_div(n * G, kUnitRows);
        unsplit += (long)units * Hkv;
        for (int u = 0; u < units; ++u) tiles += (long)unit_kv_tiles(lens[b], n, G, u, kUnitRows) * Hkv;
    }
    if (unsplit >= 8L * pairs) return nkv_max;
    const double rows = (double)offs[batch] * G * Hkv, least = ((double)tiles + (double)kNextItemTiles * unsplit) / pairs;
    int best = nkv_max;
    double best_cost = 1e30;
    for (int splits = 1, last = 0; splits <= kMaxSplits && splits <= nkv_max; ++splits) {
        const int chunk = ceil_div(nkv_max, splits);
        if (chunk == last) continue;
        last = chunk;
        // a KV tile takes a pair about 0.87 us with all of them at work; partials move at about 5.5 TB/s, each row
        // written and read; and every part of a row makes its merge longer, whatever the rows
        const double merge = rows * (splits == 1 ? 0.5 : splits) * 1024.0 / 5.5e6 / 0.87 + kSplitTiles * splits;
        if (least + merge >= best_cost) break;       // (no pair is done before its share, and the merge only grows)
        const double cost = finish_time(pairs, G, Hkv, batch, lens, offs, order, chunk) + merge;
        if (cost < best_cost - 1e-9) { best_cost = cost; best = chunk; }
    }
    return best;
}

// Work-item size (KV tiles) and the largest split count of a batch.
void batch_schedule(int num_sms, int G, int Hkv, int batch, const int* lens, const int* offs, const int* order, bool tail,
                    int kv_chunk_tiles, int* chunk_tiles, int* max_splits, long* items)
{
    int nkv_max = 1;
    for (int b = 0; b < batch; ++b) {
        const int n = offs[b + 1] - offs[b];
        const int units = ceil_div(n * G, kUnitRows);
        for (int u = 0; u < units; ++u) {
            const int nkv = batch_kv_tiles(tail, lens[b], n, G, u);
            if (nkv > nkv_max) nkv_max = nkv;
        }
    }
    int chunk = kv_chunk_tiles;
    if (chunk <= 0) {
        chunk = choose_chunk(num_sms / 2 > 0 ? num_sms / 2 : 1, G, Hkv, batch, lens, offs, order, nkv_max);
    }
    if (chunk < ceil_div(nkv_max, kMaxSplits)) chunk = ceil_div(nkv_max, kMaxSplits);
    long cnt = 0;
    for (int b = 0; b < batch; ++b) {
        const int n = offs[b + 1] - offs[b];
        const int units = ceil_div(n * G, kUnitRows);
        for (int u = 0; u < units; ++u) cnt += ceil_div(batch_kv_tiles(tail, lens[b], n, G, u), chunk);
    }
    *chunk_tiles = chunk;
    *max_splits = ceil_div(nkv_max, chunk);
    *items = cnt * Hkv;
}

// Stages of one kv head of an episode in the few-row kernel (none without new tokens).
inline int few_stages(int L, int n) { return n > 0 ? ceil_div(L + n, kFewKeys) : 0; }

// Most rows per kv head that an episode of the batch brings.
long most_rows(const evlnPagedParams* p, const int* offs)
{
    int n = 0;
    for (int b = 0; b < p->batch; ++b) n = std::max(n, offs[b + 1] - offs[b]);
    return (long)n * (p->num_q_heads / p->num_kv_heads);
}

struct PagedPlan {
    bool few;                // few-row kernel (a block per work item or per equal share)
    int chunk, share;        // KV tiles per work item, or (share > 0) 64-key stages per block
    int splits;              // most partials of a row
    long items;              // work items, or blocks
};
PagedPlan paged_schedule(evlnHandle_t h, const evlnPagedParams* p, const int* lens, const int* offs)
{
    PagedPlan plan = {false, 1, 0, 1, 0};
    const int Hkv = p->num_kv_heads;
    const long rows = most_rows(p, offs);
    if (rows <= kFewRows && p->kv_chunk_tiles == 0) {
        plan.few = true;
        // An equal share of all stages for every SM, but no row in more parts than a warp merges, nor in more
        // than the merge is worth: a stage takes about 0.41 us, another part of the longest row 0.2.
        long total = 0;
        int ns_max = 1;
        for (int b = 0; b < p->batch; ++b) {
            const int ns = few_stages(lens[b], offs[b + 1] - offs[b]);
            total += (long)ns * Hkv;
            if (ns > ns_max) ns_max = ns;
        }
        long share = (total + h->num_sms - 1) / h->num_sms;
        while (2 * share * share < ns_max) ++share;
        if (share < ceil_div(ns_max, kMaxSplits - 1)) share = ceil_div(ns_max, kMaxSplits - 1);
        plan.share = (int)share;
        plan.splits = ceil_div(ns_max - 1, plan.share) + 1;
        plan.items = (total + share - 1) / share;
        return plan;
    }
    int order[kMaxBatch];
    longest_first(p->batch, lens, offs, order);
    batch_schedule(h->num_sms, p->num_q_heads / Hkv, Hkv, p->batch, lens, offs, order, false, p->kv_chunk_tiles, &plan.chunk, &plan.splits,
                   &plan.items);
    // Few rows in work items of the caller's size: a block of the few-row kernel takes 0.8 us per 128-key tile of one
    // row tile and 1.08 of two, a CTA pair 0.75.  So two row tiles run on pairs where the items are long and there is a
    // pair for each (28/4 heads, 4 episodes of up to 9000 keys, 4 tokens each in items of 64 tiles 39.5 us against 47.0,
    // of 8 tiles 18.6 against 15.9; 40 episodes of 4000 keys, items of 32 tiles 104 against 89).
    plan.few = rows <= kFewRows && (rows <= 16 || plan.chunk <= 8 || plan.items > h->num_sms / 2);
    return plan;
}

// chunk_tiles > 0: also the first attention work item of every episode (items are numbered
// episode by episode: kv head, unit, split)
void fill_batch_lens(BatchLens* bl, int G, int Hkv, int batch, const int* lens, const int* offs, int chunk_tiles, bool tail)
{
    memset(bl, 0, sizeof(*bl));
    for (int b = 0; b < batch; ++b) bl->cache_len[b] = lens[b];
    for (int b = 0; b <= batch; ++b) bl->new_off[b] = offs[b];
    for (int b = batch + 1; b <= kMaxBatch; ++b) bl->new_off[b] = offs[batch];
    if (chunk_tiles > 0) {
        int items = 0;
        for (int b = 0; b < batch; ++b) {
            bl->item_off[b] = items;
            const int n = offs[b + 1] - offs[b];
            const int units = ceil_div(n * G, kUnitRows);
            int per_head = 0;
            for (int u = 0; u < units; ++u) per_head += ceil_div(batch_kv_tiles(tail, lens[b], n, G, u), chunk_tiles);
            items += per_head * Hkv;
        }
        for (int b = batch; b <= kMaxBatch; ++b) bl->item_off[b] = items;
    }
}

void fill_lens(BatchLens* bl, const evlnPagedParams* p, const int* lens, const int* offs, int chunk_tiles = 0, int share = 0)
{
    fill_batch_lens(bl, p->num_q_heads / p->num_kv_heads, p->num_kv_heads, p->batch, lens, offs, chunk_tiles, false);
    if (share > 0) {                     // the stages before every episode
        int at = 0;
        for (int b = 0; b <= kMaxBatch; ++b) {
            bl->item_off[b] = at;
            if (b < p->batch) at += few_stages(lens[b], offs[b + 1] - offs[b]) * p->num_kv_heads;
        }
    }
}

// Few rows in many parts: a block per row (of 128 channels; five of them fit an SM) instead of a warp, where all those blocks run at once, or,
// from nine parts on, in two rounds; elsewhere the warps are faster.  (us of a step of three calls, warps and blocks: 16 parts of 840 rows
// 20.6 and 18.4, 27 of 280 15.8 and 15.3, 7 of 560 11.7 and 11.3, 9 of 1280 42.0 and 41.0, a paged one of 1372 19.2 and 18.4; but 5 of 1904 12.7
// and 14.3, 7 of 1120 13.5 and 14.4, 7 of a paged 700 12.4 and 13.3, 9 of 1960 19.1 and 19.7.)  Steps in fp32, whose attention blocks leave more
// room beside them, a little further: 7 of 632 12.1 and 11.2, 5 of 884 12.2 and 11.5, 13 of 1240 22.6 and 20.0.
inline bool combine_wide(int parts, long blocks, bool f32, int sms)
{
    return parts > kCombineFewParts && blocks <= (parts > 8 ? 10L : f32 ? 7L : 4L) * sms;
}
// At most four parts: the form without a loop, where the other one's blocks (eight an SM) would not run at once, or are so few that its longer
// start shows; not between, where more blocks beside the attention's last CTAs crowd the SMs that ended first.  (1372 blocks 21.1 us a step with
// the loop and 20.8, 476 13.3 and 13.0, 256 13.6 and 13.2; but 640 12.3 and 12.8, 800 17.9 and 18.4, 1024 16.6 and 17.1.)
inline bool combine_few(int parts, long blocks, int sms)
{
    return parts <= kCombineFewParts && (blocks <= 4L * sms || blocks > 8L * sms);
}
template <typename T>
evlnStatus_t launch_combine(evlnHandle_t h, const CombineArgs& args, int D, bool paged, const BatchLens* bl,
                            cudaStream_t st, const SimtTiles* shares = nullptr)
{
    CombineArgs a = args;
    a.div_g = make_fast_div((uint32_t)a.G);
    a.div_chunk = make_fast_div((uint32_t)(a.chunk_tiles > 0 ? a.chunk_tiles : 1));
    if (paged && D != 128) return EVLN_NOT_SUPPORTED;
    const bool wide = combine_wide(a.num_splits, (long)ceil_div(a.rows, 128 / D) * a.Hkv, sizeof(T) == 4, h->num_sms);
    const dim3 grid(ceil_div(a.rows, wide ? 128 / D : 4), a.Hkv);
    auto launch = [&](auto form) {
        constexpr int FORM = decltype(form)::value;
        if (paged) {
            launch_pdl(combine_kernel<T, 128, true, BatchLens, FORM>, grid, dim3(128), 0, st, a, *bl);
        } else if (shares) {
            if (D == 128) launch_pdl(combine_kernel<T, 128, false, SimtTiles, FORM>, grid, dim3(128), 0, st, a, *shares);
            else launch_pdl(combine_kernel<T, 64, false, SimtTiles, FORM>, grid, dim3(128), 0, st, a, *shares);
        } else {
            NoLens nl = {};
            if (D == 128) launch_pdl(combine_kernel<T, 128, false, NoLens, FORM>, grid, dim3(128), 0, st, a, nl);
            else launch_pdl(combine_kernel<T, 64, false, NoLens, FORM>, grid, dim3(128), 0, st, a, nl);
        }
    };
    if (combine_few(a.num_splits, (long)grid.x * grid.y, h->num_sms)) launch(std::integral_constant<int, kCombineFew>());
    else if (wide) launch(std::integral_constant<int, kCombineWide>());
    else launch(std::integral_constant<int, kCombineMany>());
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? EVLN_OK : cuda_fail(h, e);
}

// The combine step of an unsplit step on a contiguous cache.
template <typename T>
evlnStatus_t launch_round_out(evlnHandle_t h, const CombineArgs& args, int D, cudaStream_t st)
{
    CombineArgs a = args;
    a.div_g = make_fast_div((uint32_t)a.G);
    const long vectors = (long)a.rows * D / VecTraits<T>::kVec;
    const dim3 grid((unsigned)((vectors + 256 * kRoundVectors - 1) / (256 * kRoundVectors)), a.Hkv);
    const cudaError_t e = D == 128 ? launch_pdl(round_out_kernel<T, 128>, grid, dim3(256), 0, st, a)
                                   : launch_pdl(round_out_kernel<T, 64>, grid, dim3(256), 0, st, a);
    return e == cudaSuccess ? EVLN_OK : cuda_fail(h, e);
}

// The combine step of rows that the attention kernel left final in the workspace (see CopyOutArgs).
evlnStatus_t launch_copy_out(evlnHandle_t h, const CombineArgs& c, cudaStream_t st)
{
    CopyOutArgs a;
    a.rows = (long)c.rows * c.Hkv;
    a.vectors = a.rows * 16;
    a.src = (const uint4*)c.o_part; a.dst = (uint4*)c.out;
    a.lse_src = c.lse_part; a.lse_dst = c.lse_out;
    const long blocks = (a.vectors + 256 * kCopyVectors - 1) / (256 * kCopyVectors);
    cudaError_t e = launch_pdl(copy_out_kernel, dim3((unsigned)blocks), dim3(256), 0, st, a);
    return e == cudaSuccess ? EVLN_OK : cuda_fail(h, e);
}

// The fields of RopeArgs that follow from the others (vec: elements per 16-byte vector).
void finish_rope_args(RopeArgs* a, int vec)
{
    a->G = a->Hq / a->Hkv;
    a->div_g = make_fast_div((uint32_t)a->G);
    a->vph_shift = 0;
    while ((1 << a->vph_shift) < a->D / 2 / vec) ++a->vph_shift;
    a->page_shift = 0;
    while ((1 << a->page_shift) < a->page_size) ++a->page_shift;
}

// The append kernels: a block per token, one thread per work item of it.
inline int rope_items(const RopeArgs& a) { return ((a.Hq + a.Hkv) << a.vph_shift) + (a.Hkv << (a.vph_shift + 1)); }
dim3 rope_block(int items)
{
    const int t = (items + 31) / 32 * 32;
    return dim3(t > kRopeThreadsMax ? kRopeThreadsMax : t < 64 ? 64 : t);
}

// Few tokens with more work items than a block has threads (64 query heads): several blocks per token, so that
// no thread starts its second item after its first.  Many tokens fill the SMs as they are, and every block of a
// token computes all of its angles.
template <typename T, bool PAGED, typename LensT>
void launch_rope_append(const RopeArgs& a, int tokens, cudaStream_t st, const LensT& lens)
{
    const int items = rope_items(a), parts = tokens <= kRopeFewTokens ? ceil_div(items, kRopeThreadsMax) : 1;
    const dim3 grid(tokens + (PAGED ? a.batch : 0), parts), block = rope_block(ceil_div(items, parts));
    if (!PAGED && tokens <= kRopeFewTokens) launch_pdl(rope_append_kernel<T, PAGED, LensT, !PAGED>, grid, block, 0, st, a, lens);
    else launch_pdl(rope_append_kernel<T, PAGED, LensT, false>, grid, block, 0, st, a, lens);
}

// CTA pairs of a persistent launch: one per two SMs, no more than there are items.
inline unsigned persistent_pairs(evlnHandle_t h, long items)
{
    const long pairs = h->num_sms / 2 > 0 ? h->num_sms / 2 : 1;
    return (unsigned)(items < pairs ? items : pairs);
}

// Gives every work item, longest first, to the pair that is done first so far.  next() returns the items in that
// order with their KV tiles; false: no table (one item per pair, or more than the table holds).
struct CostedItem {
    int number, tiles;
};
template <typename Next>
bool assign_items(int pairs, long items, Next&& next, ItemTable* table)
{
    table->count = 0;
    if (items <= pairs || items > kTableItems - pairs || pairs > kMaxPairs) return false;
    struct Load { int tiles, pair; } heap[kMaxPairs];         // the least loaded pair on top
    int turns[kMaxPairs];
    for (int i = 0; i < pairs; ++i) { heap[i] = Load{0, i}; turns[i] = 0; }
    memset(table->item, 0xff, sizeof(table->item));
    int count = 0;
    for (long k = 0; k < items; ++k) {
        const CostedItem it = next();
        Load l = heap[0];
        const int at = turns[l.pair]++ * pairs + l.pair;
        if (at >= kTableItems || turns[l.pair] > kPairItems) return false;
        table->item[at] = (unsigned short)it.number;
        if (at >= count) count = at + 1;
        l.tiles += it.tiles + kNextItemTiles;
        int i = 0;
        for (int c; (c = 2 * i + 1) < pairs; i = c) {
            if (c + 1 < pairs && heap[c + 1].tiles < heap[c].tiles) ++c;
            if (heap[c].tiles >= l.tiles) break;
            heap[i] = heap[c];
        }
        heap[i] = l;
    }
    table->count = count;
    return true;
}

// Launches a persistent kernel on `items` work items (several times when a pair would get more than it keeps).
template <typename Launch>
evlnStatus_t launch_persistent(evlnHandle_t h, long items, TcOutArgs& d, const ItemTable& table, Launch&& launch)
{
    if (table.count > 0) {
        d.first_item = 0;
        d.num_items = (int)items;
        cudaError_t e = launch(dim3(2 * persistent_pairs(h, items)));
        return e == cudaSuccess ? EVLN_OK : cuda_fail(h, e);
    }
    const long most = (long)persistent_pairs(h, items) * kPairItems;
    for (long first = 0; first < items; first += most) {
        d.first_item = (int)first;
        d.num_items = (int)(first + most < items ? first + most : items);
        cudaError_t e = launch(dim3(2 * persistent_pairs(h, d.num_items - first)));
        if (e != cudaSuccess) return cuda_fail(h, e);
    }
    return EVLN_OK;
}

// What the one-launch step adds to an attention call: the new tokens and where the results go (out null:
// partials to the workspace, for the combine kernel).
struct FewFused {
    const void *q_new, *k_new, *v_new;
    long q_stride, k_stride, v_stride;
    void* q_rot;
    void* out;
    float* lse_out;
};

// Attention of few rows on a contiguous cache: the call's partials, or the whole step (fused not null).
evlnStatus_t step_few(evlnHandle_t h, const evlnStepParams* p, const void* q_rot, const void* k_cache, const void* v_cache,
                      float* o_part, float* lse_part, const FewFused* fused, cudaStream_t st)
{
    const int G = p->num_q_heads / p->num_kv_heads, R = p->num_new * G;
    const FewPlan f = few_plan(h, p);
    if (p->num_kv_heads > 65535) return EVLN_NOT_SUPPORTED;
    CUtensorMap tm_k, tm_v;
    {
        // rows past L+n read as zeros, so stale slots never reach the tensor core
        cuuint64_t dims[3] = {128, (cuuint64_t)(p->cache_len + p->num_new), (cuuint64_t)p->num_kv_heads};
        cuuint64_t strides[2] = {256, (cuuint64_t)p->cache_capacity * 256};
        cuuint32_t box[3] = {64, kFewKeys, 1};
        if (!encode_map(h, &tm_k, k_cache, 3, dims, strides, box)) return EVLN_INVALID_VALUE;
        if (!encode_map(h, &tm_v, v_cache, 3, dims, strides, box)) return EVLN_INVALID_VALUE;
    }
    FewArgs a = {};
    a.o_part = o_part; a.lse_part = lse_part;
    a.q_rot_in = (const __nv_bfloat16*)q_rot;
    a.status = h->d_status;
    a.Hkv = p->num_kv_heads; a.G = G; a.rows = R;
    a.cache_len = p->cache_len; a.num_new = p->num_new; a.num_splits = f.splits;
    a.stages = f.stages;
    a.scale_log2 = (p->softmax_scale > 0.f ? p->softmax_scale : 1.0f / sqrtf(128.f)) * 1.4426950408889634f;
    a.div_g = make_fast_div((uint32_t)G);
    a.k_cache = (__nv_bfloat16*)const_cast<void*>(k_cache);
    a.v_cache = (__nv_bfloat16*)const_cast<void*>(v_cache);
    a.cache_cap = p->cache_capacity;
    cudaError_t e;
    if (fused) {
        a.q_new = (const __nv_bfloat16*)fused->q_new;
        a.k_new = (const __nv_bfloat16*)fused->k_new;
        a.v_new = (const __nv_bfloat16*)fused->v_new;
        a.q_stride = fused->q_stride; a.k_stride = fused->k_stride; a.v_stride = fused->v_stride;
        a.q_rot = (__nv_bfloat16*)fused->q_rot;
        a.out = (__nv_bfloat16*)fused->out;
        a.lse_out = fused->lse_out;
        a.log2_theta = log2(p->rope_theta);
        a.table = (const double2*)p->rope_table;
        a.table_first = p->rope_table_first_pos;
        e = launch_few<true>(f, R, st, tm_k, tm_v, a);
    } else {
        e = launch_few<false>(f, R, st, tm_k, tm_v, a);
    }
    return e == cudaSuccess ? EVLN_OK : cuda_fail(h, e);
}

evlnStatus_t noalloc_status_word(int** word);     // defined with the allocation-free variant below

}  // namespace

extern "C" {

const char* evlnGetErrorString(evlnStatus_t s)
{
    switch (s) {
        case EVLN_OK: return "EVLN_OK";
        case EVLN_INVALID_VALUE: return "EVLN_INVALID_VALUE";
        case EVLN_NOT_SUPPORTED: return "EVLN_NOT_SUPPORTED";
        case EVLN_CACHE_FULL: return "EVLN_CACHE_FULL";
        case EVLN_WORKSPACE_TOO_SMALL: return "EVLN_WORKSPACE_TOO_SMALL";
        case EVLN_CUDA_ERROR: return "EVLN_CUDA_ERROR";
        case EVLN_DEVICE_TIMEOUT: return "EVLN_DEVICE_TIMEOUT";
    }
    return "EVLN_UNKNOWN_STATUS";
}

evlnStatus_t evlnCreate(evlnHandle_t* handle, int device)
{
    if (!handle) return EVLN_INVALID_VALUE;
    *handle = nullptr;
    evlnContext* h = new (std::nothrow) evlnContext();
    if (!h) return EVLN_CUDA_ERROR;
    h->device = device;
    h->last_cuda_error = 0;
    h->d_status = nullptr;
    h->encode = nullptr;
    int prev_device = -1;
    cudaError_t e = cudaGetDevice(&prev_device);
    if (e == cudaSuccess) e = cudaSetDevice(device);
    // whatever happens below, the caller's current device is put back
    struct Restore {
        int dev;
        ~Restore() { if (dev >= 0) cudaSetDevice(dev); }
    } restore{prev_device};
    cudaDeviceProp prop;
    if (e == cudaSuccess) e = cudaGetDeviceProperties(&prop, device);
    if (e != cudaSuccess) { delete h; return EVLN_CUDA_ERROR; }
    if (prop.major != 10) { delete h; return EVLN_NOT_SUPPORTED; }
    h->num_sms = prop.multiProcessorCount;
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult qres;
    e = cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres);
    if (e != cudaSuccess || qres != cudaDriverEntryPointSuccess || !fn) { delete h; return EVLN_CUDA_ERROR; }
    h->encode = reinterpret_cast<EncodeTiledFn>(fn);
    e = cudaMalloc(&h->d_status, sizeof(int));
    if (e == cudaSuccess) e = cudaMemset(h->d_status, 0, sizeof(int));
    if (e == cudaSuccess) e = prepare_kernels();
    if (e == cudaSuccess) e = query_few_clusters(h->max_clusters);
    if (e == cudaSuccess) e = query_small_clusters(h->small_clusters);
    if (e == cudaSuccess && !attention_register_pool_ok()) {
        cudaFree(h->d_status);
        delete h;
        return EVLN_NOT_SUPPORTED;
    }
    if (e != cudaSuccess) {
        if (h->d_status) cudaFree(h->d_status);
        delete h;
        return EVLN_CUDA_ERROR;
    }
    *handle = h;
    return EVLN_OK;
}

evlnStatus_t evlnDestroy(evlnHandle_t h)
{
    if (!h) return EVLN_INVALID_VALUE;
    if (h->d_status) cudaFree(h->d_status);
    delete h;
    return EVLN_OK;
}

int evlnGetLastCudaError(evlnHandle_t h) { return h ? h->last_cuda_error : 0; }

evlnStatus_t evlnGetDeviceStatus(evlnHandle_t h, void* stream, int* device_status)
{
    if (!device_status) return EVLN_INVALID_VALUE;
    int* word = nullptr;
    if (h) {
        if (!device_is_current(h)) return EVLN_INVALID_VALUE;
        word = h->d_status;
    } else {
        // the allocation-free call's status word on the current device (part of the library image)
        evlnStatus_t s = noalloc_status_word(&word);
        if (s != EVLN_OK) return s;
    }
    cudaStream_t st = (cudaStream_t)stream;
    int v = 0;
    cudaError_t e = cudaMemcpyAsync(&v, word, sizeof(int), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e == cudaSuccess && v != 0) e = cudaMemsetAsync(word, 0, sizeof(int), st);
    if (e != cudaSuccess) return h ? cuda_fail(h, e) : EVLN_CUDA_ERROR;
    *device_status = v;
    return v == 0 ? EVLN_OK : EVLN_DEVICE_TIMEOUT;
}

// A bounded wait on a barrier nobody arrives on: it must run out and leave its code in the status word.
__global__ void selftest_wait_kernel(int* status, long long limit_cycles)
{
    __shared__ __align__(8) unsigned long long bar;
    __shared__ int s_abort;
    const uint32_t b = ptx::smem_u32(&bar);
    if (threadIdx.x == 0) {
        s_abort = 0;
        ptx::mbar_init(b, 1);
        ptx::fence_barrier_init();
    }
    __syncthreads();
    if (threadIdx.x == 0) wait_bounded(b, 0, EVLN_SELFTEST_STATUS_CODE, status, &s_abort, limit_cycles);
    __syncthreads();
}

evlnStatus_t evlnSelfTestBoundedWait(evlnHandle_t h, long long limit_cycles, void* stream)
{
    if (!h || limit_cycles < 1000 || limit_cycles > 1000000000LL) return EVLN_INVALID_VALUE;
    if (!device_is_current(h)) return EVLN_INVALID_VALUE;
    selftest_wait_kernel<<<1, 32, 0, (cudaStream_t)stream>>>(h->d_status, limit_cycles);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? EVLN_OK : cuda_fail(h, e);
}

size_t evlnRopeTableBytes(int head_dim, int count)
{
    if ((head_dim != 64 && head_dim != 128) || count < 0) return 0;
    return (size_t)count * (head_dim / 2) * sizeof(double2);
}

evlnStatus_t evlnRopeTable(evlnHandle_t h, int head_dim, double rope_theta, int first_pos, int count, void* table,
                           void* stream)
{
    if (!h || first_pos < 0 || count < 0 || !(rope_theta > 0.0)) return EVLN_INVALID_VALUE;
    if (head_dim != 64 && head_dim != 128) return EVLN_NOT_SUPPORTED;
    if (count == 0) return EVLN_OK;
    if (!table || !aligned16(table)) return EVLN_INVALID_VALUE;
    if (!device_is_current(h)) return EVLN_INVALID_VALUE;
    const long total = (long)count * (head_dim / 2);
    launch_pdl(rope_table_kernel, dim3((unsigned)((total + 127) / 128)), dim3(128), 0, (cudaStream_t)stream,
               (double2*)table, first_pos, count, head_dim, log2(rope_theta));
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? EVLN_OK : cuda_fail(h, e);
}

evlnStatus_t evlnStepNumSplits(evlnHandle_t h, const evlnStepParams* p, int* num_splits)
{
    evlnStatus_t s = check_step_params(h, p);
    if (s != EVLN_OK) return s;
    if (!num_splits) return EVLN_INVALID_VALUE;
    *num_splits = resolve_splits(h, p);
    return EVLN_OK;
}

evlnStatus_t evlnStepWorkspaceSize(evlnHandle_t h, const evlnStepParams* p, size_t* bytes)
{
    evlnStatus_t s = check_step_params(h, p);
    if (s != EVLN_OK) return s;
    if (!bytes) return EVLN_INVALID_VALUE;
    const long rows = (long)p->num_new * (p->num_q_heads / p->num_kv_heads);
    *bytes = partial_bytes(resolve_splits(h, p), p->num_kv_heads, rows, p->head_dim);
    return EVLN_OK;
}

evlnStatus_t evlnStepQRotSize(evlnHandle_t h, const evlnStepParams* p, size_t* bytes)
{
    evlnStatus_t s = check_step_params(h, p);
    if (s != EVLN_OK) return s;
    if (!bytes) return EVLN_INVALID_VALUE;
    *bytes = round_up((size_t)p->num_new * p->num_q_heads * p->head_dim * elem_bytes(p->dtype), 256);
    return EVLN_OK;
}

// Argument checks of the append (the parameters themselves are checked, num_new > 0).
static evlnStatus_t check_rope_append(evlnHandle_t h, const evlnStepParams* p, const void* q_new, const void* k_new,
                                      const void* v_new, long q_stride_tok, long k_stride_tok, long v_stride_tok,
                                      const void* q_rot, const void* k_cache, const void* v_cache)
{
    if (!q_new || !k_new || !v_new || !q_rot || !k_cache || !v_cache) return EVLN_INVALID_VALUE;
    if (!aligned16(q_new) || !aligned16(k_new) || !aligned16(v_new) || !aligned16(q_rot) ||
        !aligned16(k_cache) || !aligned16(v_cache))
        return EVLN_INVALID_VALUE;
    if (!device_is_current(h)) return EVLN_INVALID_VALUE;
    const int vec = 16 / elem_bytes(p->dtype);
    if (q_stride_tok < (long)p->num_q_heads * p->head_dim || k_stride_tok < (long)p->num_kv_heads * p->head_dim ||
        v_stride_tok < (long)p->num_kv_heads * p->head_dim)
        return EVLN_INVALID_VALUE;
    if (q_stride_tok % vec || k_stride_tok % vec || v_stride_tok % vec) return EVLN_INVALID_VALUE;
    return EVLN_OK;
}

evlnStatus_t evlnRopeAppend(evlnHandle_t h, const evlnStepParams* p, const void* q_new, const void* k_new,
                            const void* v_new, long q_stride_tok, long k_stride_tok, long v_stride_tok,
                            void* q_rot, void* k_cache, void* v_cache, void* stream)
{
    evlnStatus_t s = check_step_params(h, p);
    if (s != EVLN_OK) return s;
    if (p->num_new == 0) return EVLN_OK;
    s = check_rope_append(h, p, q_new, k_new, v_new, q_stride_tok, k_stride_tok, v_stride_tok, q_rot, k_cache, v_cache);
    if (s != EVLN_OK) return s;
    RopeArgs a = {};
    a.q_new = q_new; a.k_new = k_new; a.v_new = v_new;
    a.q_rot = q_rot; a.k_cache = k_cache; a.v_cache = v_cache;
    a.page_table = nullptr;
    a.q_stride = q_stride_tok; a.k_stride = k_stride_tok; a.v_stride = v_stride_tok;
    a.Hq = p->num_q_heads; a.Hkv = p->num_kv_heads; a.D = p->head_dim;
    a.cache_len = p->cache_len; a.num_new = p->num_new; a.cache_cap = p->cache_capacity;
    a.log2_theta = log2(p->rope_theta);
    a.table = (const double2*)p->rope_table;
    a.table_first = p->rope_table_first_pos;
    finish_rope_args(&a, p->dtype == EVLN_BF16 ? 8 : 4);
    NoLens nl = {};
    cudaStream_t st = (cudaStream_t)stream;
    if (p->dtype == EVLN_BF16)
        launch_rope_append<__nv_bfloat16, false, NoLens>(a, p->num_new, st, nl);
    else
        launch_rope_append<float, false, NoLens>(a, p->num_new, st, nl);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? EVLN_OK : cuda_fail(h, e);
}

// Buffers a caller shares between the arguments of a step.  Launch by launch that is sound: q_rot over q_new (rotation
// in place) or the output over anything but the cache and the workspace.  A launch that does two of the three calls'
// work has no order among its blocks: one block may write what another has still to read.
static bool output_over_q_rot(const evlnStepParams* p, const void* q_rot, const void* out, const float* lse_out)
{
    const size_t rows = (size_t)p->num_new * p->num_q_heads, bytes = rows * p->head_dim * elem_bytes(p->dtype);
    return overlap(out, bytes, q_rot, bytes) || (lse_out && overlap(lse_out, rows * sizeof(float), q_rot, bytes));
}
static bool step_buffers_shared(const evlnStepParams* p, const void* q_new, const void* k_new, const void* v_new, long q_stride,
                                long k_stride, long v_stride, const void* q_rot, const void* out, const float* lse_out)
{
    const size_t e = elem_bytes(p->dtype), rows = (size_t)p->num_new * p->num_q_heads, q_row = (size_t)p->num_q_heads * p->head_dim;
    const size_t kv_row = (size_t)p->num_kv_heads * p->head_dim, before_last = (size_t)(p->num_new - 1);
    const struct { const void* at; size_t bytes; } in[3] = {{q_new, (before_last * q_stride + q_row) * e},
                                                            {k_new, (before_last * k_stride + kv_row) * e},
                                                            {v_new, (before_last * v_stride + kv_row) * e}};
    for (const auto& x : in) {
        if (overlap(q_rot, rows * p->head_dim * e, x.at, x.bytes)) return true;
        // (the output in the very place of the queries: a head's are read by the blocks that write its output, before)
        if (x.at == q_new && out == q_new && q_stride == (long)q_row) continue;
        if (overlap(out, rows * p->head_dim * e, x.at, x.bytes) || (lse_out && overlap(lse_out, rows * sizeof(float), x.at, x.bytes))) return true;
    }
    return output_over_q_rot(p, q_rot, out, lse_out);
}

// New tokens given in the cache itself (rotated in place).  Where the blocks of several row blocks rotate the same keys, one
// would read what another has written.
static bool new_tokens_in_cache(const evlnStepParams* p, const void* k_new, const void* v_new, long k_stride, long v_stride, const void* k_cache,
                                const void* v_cache)
{
    const size_t e = elem_bytes(p->dtype), kv_row = (size_t)p->num_kv_heads * p->head_dim, before_last = (size_t)(p->num_new - 1);
    const size_t k_bytes = (before_last * k_stride + kv_row) * e, v_bytes = (before_last * v_stride + kv_row) * e, cache = kv_row * p->cache_capacity * e;
    return overlap(k_new, k_bytes, k_cache, cache) || overlap(k_new, k_bytes, v_cache, cache) || overlap(v_new, v_bytes, k_cache, cache) ||
           overlap(v_new, v_bytes, v_cache, cache);
}

// Attention of a step.  `direct` (may be null): the step's final output; when the keys are not split and
// the pair or the one-CTA kernel runs, it writes that itself and `done` says that there is nothing left to combine.
struct DirectOut {
    void* out;
    float* lse_out;
    bool done;
};
static evlnStatus_t step_attention(evlnHandle_t h, const evlnStepParams* p, const void* q_rot, const void* k_cache,
                                   const void* v_cache, void* workspace, size_t workspace_bytes, void* stream, DirectOut* direct)
{
    evlnStatus_t s = check_step_params(h, p);
    if (s != EVLN_OK) return s;
    if (p->num_new == 0) return EVLN_OK;
    if (!q_rot || !k_cache || !v_cache || !workspace) return EVLN_INVALID_VALUE;
    if (!aligned16(q_rot) || !aligned16(k_cache) || !aligned16(v_cache) || !aligned16(workspace))
        return EVLN_INVALID_VALUE;
    if (!device_is_current(h)) return EVLN_INVALID_VALUE;
    const int G = p->num_q_heads / p->num_kv_heads;
    const int R = p->num_new * G;
    const int D = p->head_dim;
    const bool simt = !use_tensor_kernel(p);
    const SimtSchedule plan = simt ? simt_schedule(h, p, p->num_splits) : SimtSchedule{};
    const int S = simt ? plan.splits : resolve_splits(h, p);
    if (workspace_bytes < partial_bytes(S, p->num_kv_heads, R, D)) return EVLN_WORKSPACE_TOO_SMALL;
    float* o_part = (float*)workspace;
    float* lse_part = o_part + (size_t)S * p->num_kv_heads * R * D;
    const float scale = p->softmax_scale > 0.f ? p->softmax_scale : 1.0f / sqrtf((float)D);
    cudaStream_t st = (cudaStream_t)stream;

    if (use_few_kernel(h, p)) {
        return step_few(h, p, q_rot, k_cache, v_cache, o_part, lse_part, nullptr, st);
    } else if (use_tensor_kernel(p)) {
        const int T = p->cache_len + p->num_new;
        const bool alone = use_solo_kernel(p) || use_single_ctas(h, p, S);
        CUtensorMap tm_q, tm_k, tm_v;
        {
            cuuint64_t dims[3] = {128, (cuuint64_t)R, (cuuint64_t)p->num_kv_heads};
            cuuint64_t strides[2] = {256, (cuuint64_t)R * 256};
            cuuint32_t box[3] = {64, 128, 1};
            if (!encode_map(h, &tm_q, q_rot, 3, dims, strides, box)) return EVLN_INVALID_VALUE;
        }
        {
            // rows past L+n read as zeros, so stale slots never reach the tensor core
            cuuint64_t dims[3] = {128, (cuuint64_t)T, (cuuint64_t)p->num_kv_heads};
            cuuint64_t strides[2] = {256, (cuuint64_t)p->cache_capacity * 256};
            // per CTA of a pair: half a K tile is 64 keys x all channels (two boxes), half a V tile
            // is 128 keys x 64 channels (one box)
            // (a CTA on its own takes whole tiles: two 128-key boxes each)
            cuuint32_t box_k[3] = {64, 64, 1};
            cuuint32_t box_v[3] = {64, 128, 1};
            if (!encode_map(h, &tm_k, k_cache, 3, dims, strides, alone ? box_v : box_k)) return EVLN_INVALID_VALUE;
            if (!encode_map(h, &tm_v, v_cache, 3, dims, strides, box_v)) return EVLN_INVALID_VALUE;
        }
        TcAttnArgs a = {};
        a.o_part = o_part; a.lse_part = lse_part; a.page_table = nullptr; a.status = h->d_status;
        a.Hkv = p->num_kv_heads; a.G = G; a.rows = R;
        a.cache_len = p->cache_len; a.num_new = p->num_new; a.num_splits = S;
        a.units_per_head = ceil_div(R, alone ? kTileM : kUnitRows);
        a.scale_log2 = scale * 1.4426950408889634f;
        a.div_g = make_fast_div((uint32_t)G);
        a.div_s = make_fast_div((uint32_t)S);
        NoLens nl = {};
        // one work item per (unit, kv head, split): the kernels read it off the block index
        if (p->num_kv_heads > 65535) return EVLN_NOT_SUPPORTED;
        if (alone) {
            TcOutArgs d = {};
            if (S == 1 && direct) {
                d.out = (__nv_bfloat16*)direct->out;
                d.lse_out = direct->lse_out;
                direct->done = true;
            }
            launch_pdl(attn_solo_kernel, dim3(a.units_per_head, p->num_kv_heads, S), dim3(kTcThreads), kSoloSmemBytes, st, tm_q, tm_k, tm_v, a, d);
        } else {
            TcOutArgs d = {};
            if (S == 1 && direct) {                // final rows, straight to the caller
                d.out = (__nv_bfloat16*)direct->out;
                d.lse_out = direct->lse_out;
                direct->done = true;
            }
            const long items = (long)p->num_kv_heads * a.units_per_head * S;
            // More items than pairs: persistent pairs where items are short (a prefill).  From about 32 KV tiles per
            // item on, what the boundaries save is lost to the spills of that kernel's tile loop (140 items of 78
            // tiles: 168 us against 158; 112 items of up to 8: 22.6 against 25.3).
            // Not with more splits than the first unit has tiles (the caller's choice only): a persistent pair ends at
            // an item without tiles, the other kernel writes its empty partial.
            const int tiles = unit_kv_tiles(p->cache_len, p->num_new, G, a.units_per_head - 1, kUnitRows) / S;
            const bool none_empty = S <= unit_kv_tiles(p->cache_len, p->num_new, G, 0, kUnitRows);
            if (items > persistent_pairs(h, items) && none_empty && tiles <= 32 && items <= 0x3fffffffL) {
                d.div_hkv = make_fast_div((uint32_t)p->num_kv_heads);
                d.div_units = make_fast_div((uint32_t)a.units_per_head);
                ItemTable table;
                int k = 0;
                assign_items((int)persistent_pairs(h, items), items, [&]() -> CostedItem {
                    const int unit = a.units_per_head - 1 - k / a.Hkv % a.units_per_head;
                    return CostedItem{k++, unit_kv_tiles(p->cache_len, p->num_new, G, unit, kUnitRows) / S};
                }, &table);
                return launch_persistent(h, items, d, table, [&](dim3 grid) {
                    return launch_pair_pdl(attn_persistent_kernel<false, NoLens>, grid, kPersistSmemBytes, st, tm_q, tm_k, tm_v, a, nl, d, table);
                });
            }
            launch_pair_pdl(attn_pair_kernel, dim3(2 * a.units_per_head, p->num_kv_heads, S), kTcSmemBytes, st, tm_q, tm_k, tm_v, a, nl, d);
        }
    } else {
        SimtAttnArgs a = {};
        a.q_rot = q_rot; a.k_cache = k_cache; a.v_cache = v_cache;
        a.o_part = o_part; a.lse_part = lse_part;
        a.Hkv = p->num_kv_heads; a.G = G;
        a.cache_len = p->cache_len; a.num_new = p->num_new; a.cache_cap = p->cache_capacity;
        a.num_splits = S; a.scale = scale;
        a.share = plan.share;
        a.status = h->d_status;
        dim3 grid(ceil_div(R, 16 * plan.rows_per_thread), p->num_kv_heads, S);
        if (p->dtype == EVLN_BF16) {
            if (D == 128) launch_simt<__nv_bfloat16, 128>(plan, p, grid, st, a);
            else launch_simt<__nv_bfloat16, 64>(plan, p, grid, st, a);
        } else if (use_f32_kernel(p)) {
            if (D == 128) launch_f32<128>(plan, p, grid, st, a);
            else launch_f32<64>(plan, p, grid, st, a);
        } else {
            if (D == 128) launch_simt<float, 128>(plan, p, grid, st, a);
            else launch_simt<float, 64>(plan, p, grid, st, a);
        }
    }
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? EVLN_OK : cuda_fail(h, e);
}


evlnStatus_t evlnStepAttention(evlnHandle_t h, const evlnStepParams* p, const void* q_rot, const void* k_cache,
                               const void* v_cache, void* workspace, size_t workspace_bytes, void* stream)
{
    return step_attention(h, p, q_rot, k_cache, v_cache, workspace, workspace_bytes, stream, nullptr);
}

evlnStatus_t evlnStepCombine(evlnHandle_t h, const evlnStepParams* p, const void* workspace, void* out,
                             float* lse_out, void* stream)
{
    evlnStatus_t s = check_step_params(h, p);
    if (s != EVLN_OK) return s;
    if (p->num_new == 0) return EVLN_OK;
    if (!workspace || !out || !aligned16(workspace) || !aligned16(out)) return EVLN_INVALID_VALUE;
    if (!device_is_current(h)) return EVLN_INVALID_VALUE;
    const int G = p->num_q_heads / p->num_kv_heads;
    const int R = p->num_new * G;
    const bool simt = !use_tensor_kernel(p);
    const SimtSchedule plan = simt ? simt_schedule(h, p, p->num_splits) : SimtSchedule{};
    const int S = simt ? plan.splits : resolve_splits(h, p);
    CombineArgs a = {};
    a.o_part = (const float*)workspace;
    a.lse_part = a.o_part + (size_t)S * p->num_kv_heads * R * p->head_dim;
    a.out = out; a.lse_out = lse_out;
    a.Hkv = p->num_kv_heads; a.G = G; a.D = p->head_dim; a.rows = R; a.num_splits = S;
    cudaStream_t st = (cudaStream_t)stream;
    if (S == 1 && p->dtype == EVLN_BF16) return launch_round_out<__nv_bfloat16>(h, a, p->head_dim, st);
    if (S == 1) return launch_round_out<float>(h, a, p->head_dim, st);
    SimtTiles tiles;
    const SimtTiles* shares = nullptr;
    if (plan.share > 0) {
        a.share = plan.share;
        a.div_share = make_fast_div((uint32_t)a.share);
        fill_simt_tiles(p, &tiles);
        shares = &tiles;
    }
    if (p->dtype == EVLN_BF16) return launch_combine<__nv_bfloat16>(h, a, p->head_dim, false, nullptr, st, shares);
    return launch_combine<float>(h, a, p->head_dim, false, nullptr, st, shares);
}

evlnStatus_t evlnStep(evlnHandle_t h, const evlnStepParams* p, const void* q_new, const void* k_new,
                      const void* v_new, long q_stride_tok, long k_stride_tok, long v_stride_tok, void* q_rot,
                      void* k_cache, void* v_cache, void* workspace, size_t workspace_bytes, void* out,
                      float* lse_out, void* stream)
{
    evlnStatus_t s = check_step_params(h, p);
    if (s != EVLN_OK) return s;
    if (p->num_new == 0) return EVLN_OK;
    // every argument is checked before the first launch, so a rejected call has done nothing
    if (!workspace || !out || !aligned16(workspace) || !aligned16(out)) return EVLN_INVALID_VALUE;
    const long rows = (long)p->num_new * (p->num_q_heads / p->num_kv_heads);
    if (workspace_bytes < partial_bytes(resolve_splits(h, p), p->num_kv_heads, rows, p->head_dim))
        return EVLN_WORKSPACE_TOO_SMALL;
    if (use_few_kernel(h, p) && p->num_new <= kFewFusedTokens &&
        !step_buffers_shared(p, q_new, k_new, v_new, q_stride_tok, k_stride_tok, v_stride_tok, q_rot, out, lse_out)) {
        s = check_rope_append(h, p, q_new, k_new, v_new, q_stride_tok, k_stride_tok, v_stride_tok, q_rot, k_cache, v_cache);
        if (s != EVLN_OK) return s;
        const int S = resolve_splits(h, p);
        float* o_part = (float*)workspace;
        FewFused f = {q_new, k_new, v_new, q_stride_tok, k_stride_tok, v_stride_tok, q_rot, S == 1 ? out : nullptr, lse_out};
        s = step_few(h, p, q_rot, k_cache, v_cache, o_part, o_part + (size_t)S * p->num_kv_heads * rows * 128, &f, (cudaStream_t)stream);
        if (s != EVLN_OK || S == 1) return s;
        return evlnStepCombine(h, p, workspace, out, lse_out, stream);
    }
    if (use_f32_kernel(p) && p->num_kv_heads <= 65535) {
        const SimtSchedule plan = simt_schedule(h, p, p->num_splits);
        if (plan.one_launch && !new_tokens_in_cache(p, k_new, v_new, k_stride_tok, v_stride_tok, k_cache, v_cache) &&
            !step_buffers_shared(p, q_new, k_new, v_new, q_stride_tok, k_stride_tok, v_stride_tok, q_rot, out, lse_out)) {
            s = check_rope_append(h, p, q_new, k_new, v_new, q_stride_tok, k_stride_tok, v_stride_tok, q_rot, k_cache, v_cache);
            if (s != EVLN_OK) return s;
            SimtAttnArgs a = {};
            a.q_rot = q_rot; a.k_cache = k_cache; a.v_cache = v_cache;
            a.Hkv = p->num_kv_heads; a.G = p->num_q_heads / p->num_kv_heads;
            a.cache_len = p->cache_len; a.num_new = p->num_new; a.cache_cap = p->cache_capacity;
            a.num_splits = plan.splits;
            F32Fused f = {};
            f.q_new = (const float*)q_new; f.k_new = (const float*)k_new; f.v_new = (const float*)v_new;
            f.q_stride = q_stride_tok; f.k_stride = k_stride_tok; f.v_stride = v_stride_tok;
            f.out = (float*)out; f.lse_out = lse_out;
            f.log2_theta = log2(p->rope_theta);
            f.table = (const double2*)p->rope_table; f.table_first = p->rope_table_first_pos;
            const cudaError_t e = p->head_dim == 128 ? launch_f32_step<128>(p, plan.splits, (cudaStream_t)stream, a, f)
                                                     : launch_f32_step<64>(p, plan.splits, (cudaStream_t)stream, a, f);
            return e == cudaSuccess ? EVLN_OK : cuda_fail(h, e);
        }
    }
    s = evlnRopeAppend(h, p, q_new, k_new, v_new, q_stride_tok, k_stride_tok, v_stride_tok, q_rot, k_cache, v_cache,
                       stream);
    if (s != EVLN_OK) return s;
    DirectOut direct = {out, lse_out, false};
    s = step_attention(h, p, q_rot, k_cache, v_cache, workspace, workspace_bytes, stream,
                       output_over_q_rot(p, q_rot, out, lse_out) ? nullptr : &direct);
    if (s != EVLN_OK || direct.done) return s;
    return evlnStepCombine(h, p, workspace, out, lse_out, stream);
}

// ---- paged -------------------------------------------------------------------------------

evlnStatus_t evlnPagedWorkspaceSize(evlnHandle_t h, const evlnPagedParams* p, const int* h_cache_lens,
                                    const int* h_new_offsets, size_t* bytes)
{
    evlnStatus_t s = check_paged_params(h, p, h_cache_lens, h_new_offsets);
    if (s != EVLN_OK) return s;
    if (!bytes) return EVLN_INVALID_VALUE;
    const long rows = (long)h_new_offsets[p->batch] * (p->num_q_heads / p->num_kv_heads);
    *bytes = partial_bytes(paged_schedule(h, p, h_cache_lens, h_new_offsets).splits, p->num_kv_heads, rows, p->head_dim);
    return EVLN_OK;
}

evlnStatus_t evlnPagedRopeAppend(evlnHandle_t h, const evlnPagedParams* p, const void* q_new, const void* k_new,
                                 const void* v_new, const int* h_cache_lens, const int* h_new_offsets,
                                 const int* d_page_table, void* q_rot, void* k_pool, void* v_pool, void* stream)
{
    evlnStatus_t s = check_paged_params(h, p, h_cache_lens, h_new_offsets);
    if (s != EVLN_OK) return s;
    const int total = h_new_offsets[p->batch];
    if (total == 0) return EVLN_OK;
    if (!q_new || !k_new || !v_new || !d_page_table || !q_rot || !k_pool || !v_pool) return EVLN_INVALID_VALUE;
    if (!aligned16(q_new) || !aligned16(k_new) || !aligned16(v_new) || !aligned16(q_rot) ||
        !aligned16(k_pool) || !aligned16(v_pool))
        return EVLN_INVALID_VALUE;
    if (!device_is_current(h)) return EVLN_INVALID_VALUE;
    RopeArgs a = {};
    a.q_new = q_new; a.k_new = k_new; a.v_new = v_new;
    a.q_rot = q_rot; a.k_cache = k_pool; a.v_cache = v_pool; a.page_table = d_page_table;
    a.q_stride = (long)p->num_q_heads * p->head_dim;
    a.k_stride = a.v_stride = (long)p->num_kv_heads * p->head_dim;
    a.Hq = p->num_q_heads; a.Hkv = p->num_kv_heads; a.D = p->head_dim;
    a.num_new = total; a.batch = p->batch; a.page_size = p->page_size; a.max_pages = p->max_pages_per_seq;
    a.log2_theta = log2(p->rope_theta);
    a.table = (const double2*)p->rope_table;
    a.table_first = p->rope_table_first_pos;
    finish_rope_args(&a, 8);
    BatchLens bl;
    fill_lens(&bl, p, h_cache_lens, h_new_offsets);
    launch_rope_append<__nv_bfloat16, true, BatchLens>(a, total, (cudaStream_t)stream, bl);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? EVLN_OK : cuda_fail(h, e);
}

evlnStatus_t evlnPagedStepAttention(evlnHandle_t h, const evlnPagedParams* p, const void* q_rot,
                                    const void* k_pool, const void* v_pool, const int* h_cache_lens,
                                    const int* h_new_offsets, const int* d_page_table, void* workspace,
                                    size_t workspace_bytes, void* stream)
{
    evlnStatus_t s = check_paged_params(h, p, h_cache_lens, h_new_offsets);
    if (s != EVLN_OK) return s;
    const int total = h_new_offsets[p->batch];
    if (total == 0) return EVLN_OK;
    if (!q_rot || !k_pool || !v_pool || !d_page_table || !workspace) return EVLN_INVALID_VALUE;
    if (!aligned16(q_rot) || !aligned16(k_pool) || !aligned16(v_pool) || !aligned16(workspace))
        return EVLN_INVALID_VALUE;
    if (!device_is_current(h)) return EVLN_INVALID_VALUE;
    const int G = p->num_q_heads / p->num_kv_heads;
    const long rows = (long)total * G;
    const PagedPlan plan = paged_schedule(h, p, h_cache_lens, h_new_offsets);
    const int chunk = plan.chunk, smax = plan.splits;
    const long items = plan.items;
    if (workspace_bytes < partial_bytes(smax, p->num_kv_heads, rows, 128)) return EVLN_WORKSPACE_TOO_SMALL;
    if (items <= 0 || items * (plan.share > 0 ? plan.share : 1) > 0x3fffffffL) return EVLN_NOT_SUPPORTED;

    if (plan.few) {
        CUtensorMap tm_k, tm_v;
        cuuint64_t dims[4] = {128, 64, (cuuint64_t)p->num_kv_heads, (cuuint64_t)p->num_pages};
        cuuint64_t strides[3] = {256, 64 * 256, (cuuint64_t)p->num_kv_heads * 64 * 256};
        cuuint32_t box[4] = {64, kFewKeys, 1, 1};
        if (!encode_map(h, &tm_k, k_pool, 4, dims, strides, box)) return EVLN_INVALID_VALUE;
        if (!encode_map(h, &tm_v, v_pool, 4, dims, strides, box)) return EVLN_INVALID_VALUE;
        const int most = (int)most_rows(p, h_new_offsets);
        FewArgs a = {};
        a.o_part = (float*)workspace;
        a.lse_part = a.o_part + (size_t)smax * p->num_kv_heads * rows * 128;
        a.q_rot_in = (const __nv_bfloat16*)q_rot;
        a.page_table = d_page_table; a.status = h->d_status;
        a.Hkv = p->num_kv_heads; a.G = G; a.rows = (int)rows;
        a.batch = p->batch; a.max_pages = p->max_pages_per_seq; a.chunk_tiles = chunk;
        a.share = plan.share;
        a.div_share = make_fast_div((uint32_t)(plan.share > 0 ? plan.share : 1));
        a.scale_log2 = (p->softmax_scale > 0.f ? p->softmax_scale : 1.0f / sqrtf(128.f)) * 1.4426950408889634f;
        a.div_g = make_fast_div((uint32_t)G);
        BatchLens bl;
        fill_lens(&bl, p, h_cache_lens, h_new_offsets, chunk, plan.share);
        if (plan.share == 0 && bl.item_off[p->batch] != (int)items) return EVLN_INVALID_VALUE;
        const size_t smem = few_smem_bytes(kFewPagedStages, most, 1, false, 0) + kFewOutBytes;
        cudaStream_t st = (cudaStream_t)stream;
        cudaError_t e = few_row_tiles(most) == 1
                            ? launch_pdl(attn_few_kernel<1, true, false, BatchLens>, dim3((int)items), dim3(kFewThreads), smem, st, tm_k, tm_v, a, bl)
                            : launch_pdl(attn_few_kernel<2, true, false, BatchLens>, dim3((int)items), dim3(kFewThreads), smem, st, tm_k, tm_v, a, bl);
        return e == cudaSuccess ? EVLN_OK : cuda_fail(h, e);
    }

    CUtensorMap tm_q, tm_k, tm_v;
    {
        cuuint64_t dims[3] = {128, (cuuint64_t)rows, (cuuint64_t)p->num_kv_heads};
        cuuint64_t strides[2] = {256, (cuuint64_t)rows * 256};
        cuuint32_t box[3] = {64, 128, 1};
        if (!encode_map(h, &tm_q, q_rot, 3, dims, strides, box)) return EVLN_INVALID_VALUE;
    }
    {
        cuuint64_t dims[4] = {128, 64, (cuuint64_t)p->num_kv_heads, (cuuint64_t)p->num_pages};
        cuuint64_t strides[3] = {256, 64 * 256, (cuuint64_t)p->num_kv_heads * 64 * 256};
        cuuint32_t box[4] = {64, 64, 1, 1};
        if (!encode_map(h, &tm_k, k_pool, 4, dims, strides, box)) return EVLN_INVALID_VALUE;
        if (!encode_map(h, &tm_v, v_pool, 4, dims, strides, box)) return EVLN_INVALID_VALUE;
    }
    const float scale = p->softmax_scale > 0.f ? p->softmax_scale : 1.0f / sqrtf(128.f);
    TcAttnArgs a = {};
    a.o_part = (float*)workspace;
    a.lse_part = a.o_part + (size_t)smax * p->num_kv_heads * rows * 128;
    a.page_table = d_page_table; a.status = h->d_status;
    a.Hkv = p->num_kv_heads; a.G = G; a.rows = (int)rows;
    a.batch = p->batch; a.max_pages = p->max_pages_per_seq; a.chunk_tiles = chunk;
    a.scale_log2 = scale * 1.4426950408889634f;
    a.div_g = make_fast_div((uint32_t)G);
    a.div_s = make_fast_div(1u);
    PagedLens bl;
    fill_lens(&bl, p, h_cache_lens, h_new_offsets);
    {
        int order[kMaxBatch];
        longest_first(p->batch, h_cache_lens, h_new_offsets, order);
        int item = 0;
        for (int i = 0; i <= kMaxBatch; ++i) {
            bl.item_off[i] = item;
            if (i >= p->batch) continue;
            const int b = order[i], n = h_new_offsets[b + 1] - h_new_offsets[b], units = ceil_div(n * G, kUnitRows);
            bl.order[i] = (unsigned char)b;
            for (int u = 0; u < units; ++u) item += ceil_div(unit_kv_tiles(h_cache_lens[b], n, G, u, kUnitRows), chunk) * p->num_kv_heads;
        }
        if (item != (int)items) return EVLN_INVALID_VALUE;
    }
    TcOutArgs d = {};
    if (smax == 1) {
        d.out = (__nv_bfloat16*)workspace;
        d.lse_out = a.lse_part;
    }
    if (items <= persistent_pairs(h, items)) {
        const cudaError_t e = launch_pair_pdl(attn_paged_pair_kernel, dim3(2 * (unsigned)items), kTcSmemBytes, (cudaStream_t)stream, tm_q, tm_k, tm_v, a, bl, d);
        return e == cudaSuccess ? EVLN_OK : cuda_fail(h, e);
    }
    ItemTable table;
    int k = 0, place = -1, unit = 0, units = 0, slot = 0, splits = 0, tiles = 0;     // in the order decode_work numbers them
    assign_items((int)persistent_pairs(h, items), items, [&]() -> CostedItem {
        if (slot == splits) {
            slot = 0;
            if (++unit >= units) unit = 0;                                           // the next kv head
            if (place < 0 || bl.item_off[place + 1] <= k) {
                do ++place; while (bl.item_off[place + 1] <= k);
                units = ceil_div((h_new_offsets[bl.order[place] + 1] - h_new_offsets[bl.order[place]]) * G, kUnitRows);
                unit = 0;
            }
            const int b = bl.order[place], nkv = unit_kv_tiles(h_cache_lens[b], h_new_offsets[b + 1] - h_new_offsets[b], G, unit, kUnitRows);
            splits = ceil_div(nkv, chunk);
            tiles = nkv / splits;
        }
        ++slot;
        return CostedItem{k++, tiles};
    }, &table);
    return launch_persistent(h, items, d, table, [&](dim3 grid) {
        return launch_pair_pdl(attn_persistent_kernel<true, PagedLens>, grid, kPersistSmemBytes, (cudaStream_t)stream, tm_q, tm_k, tm_v, a, bl, d, table);
    });
}

evlnStatus_t evlnPagedStepCombine(evlnHandle_t h, const evlnPagedParams* p, const void* workspace,
                                  const int* h_cache_lens, const int* h_new_offsets, void* out, float* lse_out,
                                  void* stream)
{
    evlnStatus_t s = check_paged_params(h, p, h_cache_lens, h_new_offsets);
    if (s != EVLN_OK) return s;
    const int total = h_new_offsets[p->batch];
    if (total == 0) return EVLN_OK;
    if (!workspace || !out || !aligned16(workspace) || !aligned16(out)) return EVLN_INVALID_VALUE;
    if (!device_is_current(h)) return EVLN_INVALID_VALUE;
    const int G = p->num_q_heads / p->num_kv_heads;
    const long rows = (long)total * G;
    const PagedPlan plan = paged_schedule(h, p, h_cache_lens, h_new_offsets);
    const int chunk = plan.chunk, smax = plan.splits;
    CombineArgs a = {};
    a.o_part = (const float*)workspace;
    a.lse_part = a.o_part + (size_t)smax * p->num_kv_heads * rows * 128;
    a.out = out; a.lse_out = lse_out;
    a.Hkv = p->num_kv_heads; a.G = G; a.D = 128; a.rows = (int)rows; a.num_splits = smax;
    a.batch = p->batch; a.chunk_tiles = chunk;
    if (smax == 1 && !plan.few) return launch_copy_out(h, a, (cudaStream_t)stream);
    a.share = plan.share;
    a.div_share = make_fast_div((uint32_t)(plan.share > 0 ? plan.share : 1));
    BatchLens bl;
    fill_lens(&bl, p, h_cache_lens, h_new_offsets, 0, plan.share);
    return launch_combine<__nv_bfloat16>(h, a, 128, true, &bl, (cudaStream_t)stream);
}

evlnStatus_t evlnPagedCheckTable(const evlnPagedParams* p, const int* h_cache_lens, const int* h_new_offsets,
                                 const int* h_page_table, int* h_bad_episode, int* h_bad_index)
{
    if (!p || !h_cache_lens || !h_new_offsets || !h_page_table) return EVLN_INVALID_VALUE;
    if (p->struct_size != sizeof(evlnPagedParams)) return EVLN_INVALID_VALUE;
    if (p->batch < 1 || p->num_pages < 1 || p->max_pages_per_seq < 1 || p->page_size < 1) return EVLN_INVALID_VALUE;
    if (h_new_offsets[0] != 0) return EVLN_INVALID_VALUE;
    std::vector<unsigned char> used((size_t)p->num_pages, 0);
    for (int b = 0; b < p->batch; ++b) {
        if (h_cache_lens[b] < 0 || h_new_offsets[b + 1] < h_new_offsets[b]) return EVLN_INVALID_VALUE;
        const long tokens = (long)h_cache_lens[b] + (h_new_offsets[b + 1] - h_new_offsets[b]);
        const long need = (tokens + p->page_size - 1) / p->page_size;
        if (need > p->max_pages_per_seq) return EVLN_CACHE_FULL;
        for (long i = 0; i < need; ++i) {
            const int pg = h_page_table[(long)b * p->max_pages_per_seq + i];
            if (pg < 0 || pg >= p->num_pages || used[pg]) {
                if (h_bad_episode) *h_bad_episode = b;
                if (h_bad_index) *h_bad_index = (int)i;
                return EVLN_INVALID_VALUE;
            }
            used[pg] = 1;
        }
    }
    return EVLN_OK;
}

}  // extern "C"

// ---- packed sequence under the action-isolating mask (Sec. 3.3) -----------------------------

namespace {
struct PackedPlan {
    int n_vis, n_act;            // instruction + visual tokens; action tokens
    int lens[kMaxBatch];         // per action chunk: visible prefix of the cache
    int offs[kMaxBatch + 1];     // per action chunk: first own token
    int chunk, smax;             // KV tiles per work item of the action batch, its largest split count
    long items;
    size_t off_qv, off_qa, off_tk, off_tv, off_part, bytes;   // workspace layout
};

evlnStatus_t plan_packed(evlnHandle_t h, const evlnPackedParams* p, PackedPlan* pl)
{
    if (!h || !p) return EVLN_INVALID_VALUE;
    if (p->struct_size != sizeof(evlnPackedParams)) return EVLN_INVALID_VALUE;
    if (p->num_q_heads <= 0 || p->num_kv_heads <= 0 || p->num_q_heads % p->num_kv_heads != 0) return EVLN_INVALID_VALUE;
    if (p->instr_len < 0 || p->frame_tokens < 0 || p->action_tokens < 0 || p->num_frames < 0 || p->kv_chunk_tiles < 0)
        return EVLN_INVALID_VALUE;
    if (!(p->rope_theta > 0.0) || !(p->softmax_scale >= 0.f)) return EVLN_INVALID_VALUE;
    if (p->dtype != EVLN_BF16 || p->head_dim != 128 || p->num_frames > kMaxBatch) return EVLN_NOT_SUPPORTED;
    const long n_vis = (long)p->instr_len + (long)p->num_frames * p->frame_tokens;
    const long n_act = (long)p->num_frames * p->action_tokens;
    const int G = p->num_q_heads / p->num_kv_heads;
    if ((n_vis + n_act) * G > (1 << 24)) return EVLN_NOT_SUPPORTED;
    if (n_vis > (long)p->cache_capacity) return EVLN_CACHE_FULL;
    pl->n_vis = (int)n_vis;
    pl->n_act = (int)n_act;
    for (int t = 0; t < p->num_frames; ++t) {
        pl->lens[t] = p->instr_len + (t + 1) * p->frame_tokens;      // chunk t sees the instruction and v_1 .. v_{t+1}
        pl->offs[t] = t * p->action_tokens;
    }
    pl->offs[p->num_frames] = (int)n_act;
    pl->chunk = pl->smax = 1;
    pl->items = 0;
    // an action chunk walks no more keys than the largest unit of the visual run beside it: not split
    // unless the caller says so
    if (n_act > 0)
        batch_schedule(h->num_sms, G, p->num_kv_heads, p->num_frames, pl->lens, pl->offs, nullptr, true,
                       p->kv_chunk_tiles > 0 ? p->kv_chunk_tiles : 1 << 24, &pl->chunk, &pl->smax, &pl->items);
    const size_t part_a = pl->smax > 1 ? partial_bytes(pl->smax, p->num_kv_heads, n_act * G, 128) : 0;
    size_t off = 0;
    pl->off_qv = off; off += round_up((size_t)n_vis * p->num_q_heads * 128 * 2, 256);
    pl->off_qa = off; off += round_up((size_t)n_act * p->num_q_heads * 128 * 2, 256);
    pl->off_tk = off; off += round_up((size_t)n_act * p->num_kv_heads * 128 * 2, 256);
    pl->off_tv = off; off += round_up((size_t)n_act * p->num_kv_heads * 128 * 2, 256);
    pl->off_part = off; off += part_a;
    pl->bytes = off > 256 ? off : 256;
    return EVLN_OK;
}
}  // namespace

extern "C" evlnStatus_t evlnPackedWorkspaceSize(evlnHandle_t h, const evlnPackedParams* p, size_t* bytes)
{
    PackedPlan pl;
    evlnStatus_t s = plan_packed(h, p, &pl);
    if (s != EVLN_OK) return s;
    if (!bytes) return EVLN_INVALID_VALUE;
    *bytes = pl.bytes;
    return EVLN_OK;
}

extern "C" evlnStatus_t evlnPackedForward(evlnHandle_t h, const evlnPackedParams* p, const void* q, const void* k,
                                          const void* v, long q_stride_tok, long k_stride_tok, long v_stride_tok,
                                          void* k_cache, void* v_cache, void* workspace, size_t workspace_bytes,
                                          void* out, float* lse_out, void* stream)
{
    PackedPlan pl;
    evlnStatus_t s = plan_packed(h, p, &pl);
    if (s != EVLN_OK) return s;
    if (pl.n_vis + pl.n_act == 0) return EVLN_OK;
    if (!q || !k || !v || !k_cache || !v_cache || !workspace || !out) return EVLN_INVALID_VALUE;
    if (!aligned16(q) || !aligned16(k) || !aligned16(v) || !aligned16(k_cache) || !aligned16(v_cache) ||
        !aligned16(workspace) || !aligned16(out))
        return EVLN_INVALID_VALUE;
    if (q_stride_tok < (long)p->num_q_heads * 128 || k_stride_tok < (long)p->num_kv_heads * 128 ||
        v_stride_tok < (long)p->num_kv_heads * 128 || q_stride_tok % 8 || k_stride_tok % 8 || v_stride_tok % 8)
        return EVLN_INVALID_VALUE;
    if (workspace_bytes < pl.bytes) return EVLN_WORKSPACE_TOO_SMALL;
    if (!device_is_current(h)) return EVLN_INVALID_VALUE;
    char* ws = (char*)workspace;
    cudaStream_t st = (cudaStream_t)stream;
    const int G = p->num_q_heads / p->num_kv_heads;
    if ((long)ceil_div(pl.n_vis * G, kUnitRows) * p->num_kv_heads + pl.items > 0x3fffffffL) return EVLN_NOT_SUPPORTED;
    BatchLens bl;
    fill_batch_lens(&bl, G, p->num_kv_heads, p->num_frames, pl.lens, pl.offs, pl.chunk, true);
    if (bl.item_off[p->num_frames] != (int)pl.items) return EVLN_NOT_SUPPORTED;

    // every token of the sequence: the visual run into the cache, the action tokens into buffers of their
    // own (nobody else's keys)
    {
        RopePackedArgs a = {};
        a.r.q_new = q; a.r.k_new = k; a.r.v_new = v;
        a.r.q_rot = ws + pl.off_qv; a.r.k_cache = k_cache; a.r.v_cache = v_cache;
        a.r.q_stride = q_stride_tok; a.r.k_stride = k_stride_tok; a.r.v_stride = v_stride_tok;
        a.r.Hq = p->num_q_heads; a.r.Hkv = p->num_kv_heads; a.r.D = 128;
        a.r.num_new = pl.n_vis + pl.n_act; a.r.cache_cap = p->cache_capacity;
        a.r.page_size = 1;
        a.r.log2_theta = log2(p->rope_theta);
        finish_rope_args(&a.r, 8);
        a.num_visual = pl.n_vis; a.num_action = pl.n_act;
        a.I = p->instr_len; a.F = p->frame_tokens; a.A = p->action_tokens;
        a.div_f = make_fast_div((uint32_t)(p->frame_tokens > 0 ? p->frame_tokens : 1));
        a.div_a = make_fast_div((uint32_t)(p->action_tokens > 0 ? p->action_tokens : 1));
        a.q_rot_act = ws + pl.off_qa; a.k_act = ws + pl.off_tk; a.v_act = ws + pl.off_tv;
        cudaError_t e = launch_pdl(rope_packed_kernel, dim3(a.r.num_new), rope_block(rope_items(a.r)), 0, st, a);
        if (e != cudaSuccess) return cuda_fail(h, e);
    }
    // one launch: the visual run as one causal prefill (its query tiles never load a KV tile past their own
    // last token, and no action token is among the keys at all), and beside it the action chunks, chunk t
    // seeing the first lens[t] tokens of the cache and its own tokens
    const long rows_a = (long)pl.n_act * G;
    const bool split = pl.smax > 1;
    {
        CUtensorMap maps[6];              // visual q, k, v; action q, k, v
        const cuuint32_t box_q[3] = {64, 128, 1}, box_k[3] = {64, 64, 1}, box_v[3] = {64, 128, 1};
        const cuuint32_t* boxes[3] = {box_q, box_k, box_v};
        const void* bases[6] = {ws + pl.off_qv, k_cache, v_cache, ws + pl.off_qa, ws + pl.off_tk, ws + pl.off_tv};
        const long rows[6] = {(long)pl.n_vis * G, pl.n_vis, pl.n_vis, rows_a, pl.n_act, pl.n_act};
        const long pitch[6] = {rows[0], p->cache_capacity, p->cache_capacity, rows_a, pl.n_act, pl.n_act};
        for (int i = 0; i < 6; ++i) {
            if (rows[i] == 0) continue;
            cuuint64_t dims[3] = {128, (cuuint64_t)rows[i], (cuuint64_t)p->num_kv_heads};
            cuuint64_t strides[2] = {256, (cuuint64_t)pitch[i] * 256};
            if (!encode_map(h, &maps[i], bases[i], 3, dims, strides, boxes[i % 3])) return EVLN_INVALID_VALUE;
        }
        for (int i = 0; i < 6; ++i)       // a run without tokens loads nothing: any valid map will do
            if (rows[i] == 0) maps[i] = maps[(i + 3) % 6];
        const float scale = p->softmax_scale > 0.f ? p->softmax_scale : 1.0f / sqrtf(128.f);
        TcAttnArgs a = {};
        a.o_part = (float*)(ws + pl.off_part);
        a.lse_part = a.o_part + (size_t)pl.smax * p->num_kv_heads * rows_a * 128;
        a.status = h->d_status;
        a.Hkv = p->num_kv_heads; a.G = G; a.rows = (int)rows_a;
        a.num_new = pl.n_vis; a.units_per_head = ceil_div(pl.n_vis * G, kUnitRows);
        a.batch = p->num_frames; a.chunk_tiles = pl.chunk;
        a.scale_log2 = scale * 1.4426950408889634f;
        a.div_g = make_fast_div((uint32_t)G);
        a.div_s = make_fast_div(1u);
        TcOutArgs d = {};
        d.out = (__nv_bfloat16*)out; d.lse_out = lse_out;
        d.map = make_packed_map(p->instr_len, p->frame_tokens, p->action_tokens, 0);
        d.act_items = (int)pl.items; d.act_split = split;
        d.act_map = make_packed_map(p->instr_len, p->frame_tokens, p->action_tokens, 1);
        d.div_hkv = make_fast_div((uint32_t)p->num_kv_heads);
        // both runs of items come longest first: merge them
        const long items = pl.items + (long)a.units_per_head * p->num_kv_heads;
        ItemTable table;
        int act = 0, vis = 0, chunk_of = p->num_frames - 1;
        assign_items((int)persistent_pairs(h, items), items, [&]() -> CostedItem {
            int act_tiles = -1, vis_tiles = -1;
            if (act < (int)pl.items) {
                while (bl.item_off[chunk_of] > (int)pl.items - 1 - act) --chunk_of;
                const int nkv = tail_kv_tiles(pl.lens[chunk_of], p->action_tokens, G, 0, kUnitRows);
                act_tiles = nkv / ceil_div(nkv, pl.chunk);
            }
            if (vis < a.units_per_head * a.Hkv) vis_tiles = unit_kv_tiles(0, pl.n_vis, G, a.units_per_head - 1 - vis / a.Hkv, kUnitRows);
            if (act_tiles >= vis_tiles) return CostedItem{act++, act_tiles};
            return CostedItem{(int)pl.items + vis++, vis_tiles};
        }, &table);
        s = launch_persistent(h, items, d, table, [&](dim3 grid) {
            return launch_pair_pdl(attn_packed_kernel, grid, kPersistSmemBytes, st, maps[0], maps[1], maps[2], maps[3], maps[4], maps[5], a, bl, d, table);
        });
        if (s != EVLN_OK) return s;
    }
    if (!split) return EVLN_OK;
    CombineArgs c = {};
    c.o_part = (const float*)(ws + pl.off_part);
    c.lse_part = c.o_part + (size_t)pl.smax * p->num_kv_heads * rows_a * 128;
    c.out = out; c.lse_out = lse_out;
    c.Hkv = p->num_kv_heads; c.G = G; c.D = 128; c.rows = (int)rows_a; c.num_splits = pl.smax;
    c.batch = p->num_frames; c.chunk_tiles = pl.chunk;
    c.tail = 1;
    c.map = make_packed_map(p->instr_len, p->frame_tokens, p->action_tokens, 1);
    return launch_combine<__nv_bfloat16>(h, c, 128, true, &bl, st);
}

// ---- un-rotated store + frame sampler ------------------------------------------------------

namespace {
evlnStatus_t check_gather_params(evlnHandle_t h, const evlnGatherParams* p)
{
    if (!h || !p) return EVLN_INVALID_VALUE;
    if (p->struct_size != sizeof(evlnGatherParams)) return EVLN_INVALID_VALUE;
    if (p->dtype != EVLN_BF16 && p->dtype != EVLN_F32) return EVLN_INVALID_VALUE;
    if (p->num_kv_heads <= 0 || p->store_capacity < 0 || p->work_capacity < 0) return EVLN_INVALID_VALUE;
    if (!(p->rope_theta > 0.0)) return EVLN_INVALID_VALUE;
    if (p->head_dim != 64 && p->head_dim != 128) return EVLN_NOT_SUPPORTED;
    if (!device_is_current(h)) return EVLN_INVALID_VALUE;
    return EVLN_OK;
}
}  // namespace

extern "C" int evlnSampleFrames(int sampler, int num_frames, int budget, int stride, int* h_indices)
{
    if (num_frames < 0 || budget < 0 || !h_indices) return -1;
    if (num_frames == 0 || budget == 0) return 0;
    if (sampler == EVLN_SAMPLE_UNIFORM) {
        if (num_frames <= budget) {
            for (int i = 0; i < num_frames; ++i) h_indices[i] = i;
            return num_frames;
        }
        if (budget == 1) { h_indices[0] = num_frames - 1; return 1; }
        for (int k = 0; k < budget; ++k)      // round(k (N-1) / (B-1)), halves up
            h_indices[k] = (int)((2L * k * (num_frames - 1) + (budget - 1)) / (2L * (budget - 1)));
        return budget;
    }
    if (sampler == EVLN_SAMPLE_SLIDING) {
        if (stride < 1) return -1;
        int count = 0;
        for (int f = num_frames - 1; f >= 0 && count < budget; f -= stride) ++count;
        for (int k = 0; k < count; ++k) h_indices[k] = num_frames - 1 - (count - 1 - k) * stride;
        return count;
    }
    return -1;
}

extern "C" evlnStatus_t evlnStoreAppend(evlnHandle_t h, const evlnGatherParams* p, const void* k_new,
                                        const void* v_new, long k_stride_tok, long v_stride_tok, int store_len,
                                        int num_new, void* k_store, void* v_store, void* stream)
{
    evlnStatus_t s = check_gather_params(h, p);
    if (s != EVLN_OK) return s;
    if (store_len < 0 || num_new < 0) return EVLN_INVALID_VALUE;
    if ((long)store_len + num_new > (long)p->store_capacity) return EVLN_CACHE_FULL;
    if (num_new == 0) return EVLN_OK;
    if (!k_new || !v_new || !k_store || !v_store) return EVLN_INVALID_VALUE;
    if (!aligned16(k_new) || !aligned16(v_new) || !aligned16(k_store) || !aligned16(v_store)) return EVLN_INVALID_VALUE;
    const int vec = 16 / elem_bytes(p->dtype);
    const long row = (long)p->num_kv_heads * p->head_dim;
    if (k_stride_tok < row || v_stride_tok < row || k_stride_tok % vec || v_stride_tok % vec) return EVLN_INVALID_VALUE;
    GatherArgs a = {};
    a.k_src = k_new; a.v_src = v_new; a.k_dst = k_store; a.v_dst = v_store;
    a.k_stride = k_stride_tok; a.v_stride = v_stride_tok;
    a.Hkv = p->num_kv_heads; a.D = p->head_dim;
    a.dst_cap = p->store_capacity; a.first_slot = store_len; a.num_tokens = num_new;
    cudaStream_t st = (cudaStream_t)stream;
    if (p->dtype == EVLN_BF16) launch_pdl(store_append_kernel<__nv_bfloat16>, dim3(num_new), dim3(128), 0, st, a);
    else launch_pdl(store_append_kernel<float>, dim3(num_new), dim3(128), 0, st, a);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? EVLN_OK : cuda_fail(h, e);
}

extern "C" evlnStatus_t evlnGatherRope(evlnHandle_t h, const evlnGatherParams* p, int num_segments,
                                       const int* h_seg_src, const int* h_seg_len, const void* k_store,
                                       const void* v_store, void* k_work, void* v_work, int* h_total, void* stream)
{
    evlnStatus_t s = check_gather_params(h, p);
    if (s != EVLN_OK) return s;
    if (num_segments < 0 || (num_segments > 0 && (!h_seg_src || !h_seg_len))) return EVLN_INVALID_VALUE;
    if (num_segments > kMaxSegments) return EVLN_NOT_SUPPORTED;
    SegList segs;
    memset(&segs, 0, sizeof(segs));
    long total = 0;
    for (int i = 0; i < num_segments; ++i) {
        if (h_seg_src[i] < 0 || h_seg_len[i] < 0 || (long)h_seg_src[i] + h_seg_len[i] > (long)p->store_capacity)
            return EVLN_INVALID_VALUE;
        segs.src[i] = h_seg_src[i];
        segs.dst_off[i] = (int)total;
        total += h_seg_len[i];
        if (total > (long)p->work_capacity) return EVLN_CACHE_FULL;
    }
    for (int i = num_segments; i <= kMaxSegments; ++i) segs.dst_off[i] = (int)total;
    if (h_total) *h_total = (int)total;
    if (total == 0) return EVLN_OK;
    if (!rope_table_covers(p->rope_table, p->rope_table_first_pos, p->rope_table_count, 0, total)) return EVLN_INVALID_VALUE;
    if (!k_store || !v_store || !k_work || !v_work) return EVLN_INVALID_VALUE;
    if (!aligned16(k_store) || !aligned16(v_store) || !aligned16(k_work) || !aligned16(v_work)) return EVLN_INVALID_VALUE;
    GatherArgs a = {};
    a.k_src = k_store; a.v_src = v_store; a.k_dst = k_work; a.v_dst = v_work;
    a.Hkv = p->num_kv_heads; a.D = p->head_dim;
    a.src_cap = p->store_capacity; a.dst_cap = p->work_capacity;
    a.num_tokens = (int)total; a.num_segments = num_segments;
    a.log2_theta = log2(p->rope_theta);
    a.table = (const double2*)p->rope_table;
    a.table_first = p->rope_table_first_pos;
    cudaStream_t st = (cudaStream_t)stream;
    const int vec = 16 / elem_bytes(p->dtype);
    while ((1 << a.vph_shift) < a.D / 2 / vec) ++a.vph_shift;
    a.k_chunks = ceil_div(a.Hkv << a.vph_shift, 32);
    a.v_chunks = ceil_div(a.Hkv << (a.vph_shift + 1), 64);
    a.div_chunks = make_fast_div((uint32_t)(a.k_chunks + a.v_chunks));
    if (gather_by_block(a.k_chunks, total, a.table != nullptr, p->dtype == EVLN_BF16, a.D)) {
        if (p->dtype == EVLN_BF16) launch_pdl(gather_rope_block_kernel<__nv_bfloat16>, dim3((unsigned)total), dim3(kGatherBlockThreads), 0, st, a, segs);
        else launch_pdl(gather_rope_block_kernel<float>, dim3((unsigned)total), dim3(kGatherBlockThreads), 0, st, a, segs);
        const cudaError_t e = cudaGetLastError();
        return e == cudaSuccess ? EVLN_OK : cuda_fail(h, e);
    }
    if (total * (a.k_chunks + a.v_chunks) > 0x7fffff00L) return EVLN_NOT_SUPPORTED;
    const long blocks = (total * (a.k_chunks + a.v_chunks) + kGatherWarps - 1) / kGatherWarps;
    const dim3 grid((unsigned)blocks), block(32 * kGatherWarps);
    const bool wave = gather_one_wave(a.Hkv << a.vph_shift, a.k_chunks, blocks, a.table != nullptr, h->num_sms);
    if (p->dtype == EVLN_BF16) launch_pdl(wave ? gather_rope_kernel<__nv_bfloat16, true> : gather_rope_kernel<__nv_bfloat16, false>, grid, block, 0, st, a, segs);
    else launch_pdl(wave ? gather_rope_kernel<float, true> : gather_rope_kernel<float, false>, grid, block, 0, st, a, segs);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? EVLN_OK : cuda_fail(h, e);
}

// ---- host-resident store: strided DMA between the pinned host store and the device store ----

namespace {
evlnStatus_t store_copy(evlnHandle_t h, const evlnGatherParams* p, const void* k_src, const void* v_src, int src_cap,
                        int src_slot, int len, void* k_dst, void* v_dst, int dst_cap, int dst_slot, cudaStream_t st,
                        cudaMemcpyKind kind)
{
    evlnStatus_t s = check_gather_params(h, p);
    if (s != EVLN_OK) return s;
    if (src_slot < 0 || dst_slot < 0 || len < 0 || src_cap < 0 || dst_cap < 0) return EVLN_INVALID_VALUE;
    if ((long)src_slot + len > (long)src_cap) return EVLN_INVALID_VALUE;
    if ((long)dst_slot + len > (long)dst_cap) return EVLN_CACHE_FULL;
    if (len == 0) return EVLN_OK;
    if (!k_src || !v_src || !k_dst || !v_dst) return EVLN_INVALID_VALUE;
    const size_t row = (size_t)p->head_dim * elem_bytes(p->dtype);       // one token of one head
    const size_t width = row * len;
    cudaError_t e = cudaMemcpy2DAsync((char*)k_dst + row * dst_slot, row * dst_cap, (const char*)k_src + row * src_slot,
                                      row * src_cap, width, p->num_kv_heads, kind, st);
    if (e == cudaSuccess)
        e = cudaMemcpy2DAsync((char*)v_dst + row * dst_slot, row * dst_cap, (const char*)v_src + row * src_slot,
                              row * src_cap, width, p->num_kv_heads, kind, st);
    return e == cudaSuccess ? EVLN_OK : cuda_fail(h, e);
}
}  // namespace

extern "C" evlnStatus_t evlnStoreOffload(evlnHandle_t h, const evlnGatherParams* p, const void* k_store,
                                         const void* v_store, int src_slot, int len, void* h_k_store, void* h_v_store,
                                         int host_capacity, int dst_slot, void* stream)
{
    if (!p) return EVLN_INVALID_VALUE;
    return store_copy(h, p, k_store, v_store, p->store_capacity, src_slot, len, h_k_store, h_v_store, host_capacity,
                      dst_slot, (cudaStream_t)stream, cudaMemcpyDeviceToHost);
}

extern "C" evlnStatus_t evlnStoreFetch(evlnHandle_t h, const evlnGatherParams* p, const void* h_k_store,
                                       const void* h_v_store, int host_capacity, int src_slot, int len, void* k_store,
                                       void* v_store, int dst_slot, void* stream)
{
    if (!p) return EVLN_INVALID_VALUE;
    return store_copy(h, p, h_k_store, h_v_store, host_capacity, src_slot, len, k_store, v_store, p->store_capacity,
                      dst_slot, (cudaStream_t)stream, cudaMemcpyHostToDevice);
}

// ---- allocation-free variant --------------------------------------------------------------

// Scratch for the split partials of evlnStepAttentionNoAlloc, part of the library image: every
// device that loads the library holds these bytes until the process exits.  In host code the
// names below are only stand-ins for the device objects; their device addresses come from
// cudaGetSymbolAddress (once per device) and are what the kernels receive.
static __device__ __align__(256) unsigned char g_noalloc_scratch[EVLN_NOALLOC_SCRATCH_BYTES];
static __device__ __align__(256) int g_noalloc_status;

namespace {
constexpr int kMaxDevices = 64;
struct NoAllocDevice {
    bool ready;
    evlnContext ctx;          // plain struct used as the handle of the regular entry points
    void* scratch;
};
NoAllocDevice g_noalloc_dev[kMaxDevices];
std::mutex g_noalloc_mutex;       // host threads may race for the first call on a device

// First call on a device: resolve device addresses and properties.  Allocates nothing.
evlnStatus_t noalloc_setup(int device, NoAllocDevice** out)
{
    if (device < 0 || device >= kMaxDevices) return EVLN_NOT_SUPPORTED;
    NoAllocDevice* d = &g_noalloc_dev[device];
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    if (!d->ready) {
        cudaDeviceProp prop;
        cudaError_t e = cudaGetDeviceProperties(&prop, device);
        if (e != cudaSuccess) return EVLN_CUDA_ERROR;
        if (prop.major != 10) return EVLN_NOT_SUPPORTED;
        void* scratch = nullptr;
        void* status = nullptr;
        e = cudaGetSymbolAddress(&scratch, g_noalloc_scratch);
        if (e != cudaSuccess || !scratch) return EVLN_CUDA_ERROR;
        e = cudaGetSymbolAddress(&status, g_noalloc_status);
        if (e != cudaSuccess || !status) return EVLN_CUDA_ERROR;
        void* fn = nullptr;
        cudaDriverEntryPointQueryResult qres;
        e = cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres);
        if (e != cudaSuccess || qres != cudaDriverEntryPointSuccess || !fn) return EVLN_CUDA_ERROR;
        e = prepare_kernels();
        if (e == cudaSuccess) e = query_few_clusters(d->ctx.max_clusters);
        if (e == cudaSuccess) e = query_small_clusters(d->ctx.small_clusters);
        if (e != cudaSuccess) return EVLN_CUDA_ERROR;
        if (!attention_register_pool_ok()) return EVLN_NOT_SUPPORTED;
        d->ctx.device = device;
        d->ctx.num_sms = prop.multiProcessorCount;
        d->ctx.last_cuda_error = 0;
        d->ctx.d_status = static_cast<int*>(status);
        d->ctx.encode = reinterpret_cast<EncodeTiledFn>(fn);
        d->scratch = scratch;
        d->ready = true;
    }
    *out = d;
    return EVLN_OK;
}
// Device address of the allocation-free call's status word on the current device.
evlnStatus_t noalloc_status_word(int** word)
{
    int device = -1;
    if (cudaGetDevice(&device) != cudaSuccess) return EVLN_CUDA_ERROR;
    NoAllocDevice* d = nullptr;
    evlnStatus_t s = noalloc_setup(device, &d);
    if (s != EVLN_OK) return s;
    *word = d->ctx.d_status;
    return EVLN_OK;
}
}  // namespace

extern "C" evlnStatus_t evlnStepAttentionNoAlloc(const evlnStepParams* p, const void* q_rot, const void* k_cache,
                                                 const void* v_cache, void* out, float* lse_out, void* stream)
{
    int device = -1;
    if (cudaGetDevice(&device) != cudaSuccess) return EVLN_CUDA_ERROR;
    NoAllocDevice* d = nullptr;
    evlnStatus_t s = noalloc_setup(device, &d);
    if (s != EVLN_OK) return s;
    evlnHandle_t h = &d->ctx;
    size_t need = 0;
    s = evlnStepWorkspaceSize(h, p, &need);
    if (s != EVLN_OK) return s;
    if (p->num_new == 0) return EVLN_OK;
    evlnStepParams fitting = *p;
    if (need > (size_t)EVLN_NOALLOC_SCRATCH_BYTES) {
        // The fp32 and SIMT kernels split to fill the chip, up to 2.3 times faster than what fits here for large steps, so it is
        // this call that makes do with fewer splits.  (The schedules of the other kernels take about as few as they can.)
        const size_t one = partial_bytes(1, p->num_kv_heads, (long)p->num_new * (p->num_q_heads / p->num_kv_heads), p->head_dim);
        const int fit = (int)(EVLN_NOALLOC_SCRATCH_BYTES / one);
        if (p->num_splits > 0 || use_tensor_kernel(p) || fit < 1) return EVLN_WORKSPACE_TOO_SMALL;
        fitting.num_splits = simt_schedule(h, p, 0, fit).splits;
        p = &fitting;
    }
    if (!out || !aligned16(out)) return EVLN_INVALID_VALUE;
    DirectOut direct = {out, lse_out, false};
    s = step_attention(h, p, q_rot, k_cache, v_cache, d->scratch, (size_t)EVLN_NOALLOC_SCRATCH_BYTES, stream,
                       output_over_q_rot(p, q_rot, out, lse_out) ? nullptr : &direct);
    if (s != EVLN_OK || direct.done) return s;
    return evlnStepCombine(h, p, d->scratch, out, lse_out, stream);
}
