// Step attention of a few new tokens (at most 32 packed query rows per kv head; bf16, head_dim 128):
// the action tokens decoded after a frame (Sec. 3.1), contiguous cache or a batch of paged episodes.
//
// Bound: reading K and V once from HBM, and below a few MB the chain of latencies of a step.  With so
// few rows a 128-row tcgen05 tile is padding, and its round trips through tensor memory are the longest
// part of the chain, so the products run on mma.sync (16-row tiles, fed by ldmatrix): scores, exponentials
// and P stay in the registers of one warp and no two warps wait for each other before the final merge.
//
// A block: 8 compute warps and a producer warp.  K and V come through a ring of 64-key stages (16 KB +
// 16 KB, TMA, 128-byte swizzle; a 64-token page is exactly one stage).  With MT 16-row tiles of queries
// (1 or 2), four warps share a stage (16 MT keys x 16 rows each) and the two groups of four take the stages
// in turn; every warp keeps a running maximum, sum and output of its own.
// The warps' results are merged in shared memory.  Paged: one block per SM, each with an equal share of the
// batch's stages, walked in episode order; a share goes through the ends of units (episode, kv head) with the
// ring running on, and a unit is split where the shares meet.  (One block per work item of a quarter of an
// SM's share, until then: 16 ragged episodes of one token 61.6 us, 8 episodes of up to 4096 tokens 22.4.  Items
// in whole numbers left SMs idle at the end, and every item paid a start of about 3 us.)  Contiguous caches spread a kv head's keys over a
// cluster of up to 16 blocks, which send each row to the block that merges it (distributed shared memory,
// st.async on that block's barrier: one way, no cluster-wide meeting at the end), so that a whole
// step leaves one (normalised) result per head, or per split when the caller asks for splits.
//
// FUSED: the block also does the append kernel's work for its own keys: it rotates the queries straight
// into shared memory (and, once per head, into q_rot), rotates the new keys that fall into its range,
// writes them with the values to the cache and into the stage they belong to, and the cluster writes the
// final output: evlnStep is one launch.  Same bits as the three calls: same rotation, same order.
#pragma once

#include <cuda.h>

#include "attn_pair.cuh"
#include "common.cuh"
#include "ptx_sm100.cuh"
#include "rope_append.cuh"

namespace evln {

constexpr int kFewRows = 32;                  // most packed query rows per kv head
constexpr int kFewFusedTokens = 16;           // most new tokens of a fused step
constexpr int kFewWarps = 8;                  // compute warps
constexpr int kFewThreads = 32 * (kFewWarps + 1);
constexpr int kFewStageBytes = 2 * kFewKeys * 256;
constexpr int kFewGroups = 2;                 // groups of warps that take the stages in turn
// Ring depth: a multiple of the number of groups, so that a slot is always consumed by the same group.
// (A group that met another group's slot could find its barrier a whole phase behind, which a wait by
// parity cannot tell from complete.)  Six where they fit: a block keeps 192 KB in flight, which is what
// 64 blocks need to draw the full HBM rate (with four, 71 GB/s per SM).
constexpr int kFewMaxStages = 6, kFewMinStages = 4;
static_assert(kFewMaxStages % kFewGroups == 0 && kFewMinStages % kFewGroups == 0, "a slot belongs to one group");
// Paged: four, beside them the warps' outputs have a place of their own, so that the ring goes on filling while a
// unit's results are merged.  148 blocks draw the full HBM rate with half of that.
constexpr int kFewPagedStages = 4;
constexpr int kFewMaxCluster = 16;
constexpr int kFewOStride = 132;              // floats per row of a warp's output in shared memory

struct FewArgs {
    float* o_part;            // [S, Hkv, rows, 128]
    float* lse_part;          // [S, Hkv, rows]
    const __nv_bfloat16* q_rot_in;
    const int* page_table;    // paged only
    int* status;              // device status word
    int Hkv, G;
    int rows;                 // packed rows per kv head over the whole call
    int cache_len, num_new;   // contiguous only
    int num_splits;           // contiguous only
    int stages;               // ring depth
    int batch, max_pages, chunk_tiles;   // paged only
    int share;                // paged only: stages per block, 0: work items of chunk_tiles tiles
    FastDiv div_share;
    float scale_log2;         // softmax scale * log2(e)
    FastDiv div_g;            // division by G
    // contiguous only: the cache, for the fused append
    __nv_bfloat16* k_cache;
    __nv_bfloat16* v_cache;
    int cache_cap;
    // fused only
    const __nv_bfloat16* q_new;
    const __nv_bfloat16* k_new;
    const __nv_bfloat16* v_new;
    long q_stride, k_stride, v_stride;
    __nv_bfloat16* q_rot;
    __nv_bfloat16* out;       // final output [n, Hq, 128], null: partials go to o_part / lse_part
    float* lse_out;
    double log2_theta;
    const double2* table;
    int table_first;
};

// Shared memory, from a 1024-byte boundary: stages | Q [16 MT][256 B] | barriers | weights | rows the cluster's
// blocks send here | fused: angles, new K/V rows.  After the last stage has been consumed the ring holds
// the warps' outputs (paged: they lie behind the weights).
constexpr int kFewBarBytes = 256;
constexpr int kFewStatBytes = 2 * kFewWarps * kFewRows * 4;
constexpr int kFewRowBytes = kFewOStride * 4;           // a row in flight: 128 channels, reference, sum
constexpr int kFewAngleBytes = Rotation<__nv_bfloat16>::kAngles * 16;
constexpr int kFewMaxSmem = 227 * 1024;
constexpr int kFewOutBytes = kFewWarps * 16 * kFewOStride * 4;      // the warps' outputs (paged: behind the statistics)
__host__ __device__ inline int few_cluster_bytes(int rows, int cluster)
{
    return cluster > 1 ? (rows + cluster - 1) / cluster * cluster * kFewRowBytes : 0;
}
inline int few_smem_bytes(int stages, int rows, int cluster, bool fused, int num_new)
{
    return 1024 + stages * kFewStageBytes + (rows + 15) / 16 * 16 * 256 + kFewBarBytes + kFewStatBytes + few_cluster_bytes(rows, cluster) +
           (fused ? num_new * (kFewAngleBytes + 512) : 0);
}
static_assert(kFewMinStages * kFewStageBytes >= kFewOutBytes, "the outputs fit the stages");

// Bytes of (row, 16-byte chunk) in a 64-channel block of 128-byte swizzled rows.
__device__ __forceinline__ uint32_t swz(int row, int chunk) { return (uint32_t)(row * 128 + ((chunk ^ (row & 7)) << 4)); }

// A finished row (lane: channels 4 lane .. + 3; output and sum relative to the reference M): the final
// output, or the split's partial.
__device__ __forceinline__ void few_write_row(const FewArgs& a, const float4& acc, float M, float sum, int g, int slot, int row_base,
                                              int r, int lane)
{
    const float inv = sum > 0.f ? 1.f / sum : 0.f;
    const float lse = sum > 0.f ? (M + log2f(sum)) * 0.6931471805599453f : -INFINITY;
    if (a.out) {
        const int tok = (int)fast_div((uint32_t)r, a.div_g);
        const long at = (long)tok * a.Hkv * a.G + g * a.G + (r - tok * a.G);
        reinterpret_cast<uint2*>(a.out + at * 128)[lane] =
            make_uint2(ptx::pack_bf16x2(acc.x * inv, acc.y * inv), ptx::pack_bf16x2(acc.z * inv, acc.w * inv));
        if (a.lse_out && lane == 0) a.lse_out[at] = lse;
    } else {
        const long prow = ((long)slot * a.Hkv + g) * a.rows + row_base + r;
        reinterpret_cast<float4*>(a.o_part + prow * 128)[lane] = make_float4(acc.x * inv, acc.y * inv, acc.z * inv, acc.w * inv);
        if (lane == 0) a.lse_part[prow] = lse;
    }
}

// MT: 16-row tiles of the queries.  Contiguous cache: grid (cluster, kv heads, splits);
// PAGED: one block per share of the stages, or per work item, numbered as in the pair kernel.
template <int MT, bool PAGED, bool FUSED, typename LensT>
__global__ void __launch_bounds__(kFewThreads)
attn_few_kernel(const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_v, const FewArgs a,
                const __grid_constant__ LensT lens)
{
    static_assert(!(PAGED && FUSED), "the paged calls come one by one");
    constexpr int WK = kFewWarps / MT;                 // warps that share a row tile: 16 MT keys of a stage each,
    constexpr int kShare = 16 * MT;                    //   every second stage
    extern __shared__ uint8_t smem_raw[];
    const uint32_t smem_base = (ptx::smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* smem_gen = smem_raw + (smem_base - ptx::smem_u32(smem_raw));
    const int stages = PAGED ? kFewPagedStages : a.stages;
    const int q_off = stages * kFewStageBytes, bar_off = q_off + MT * 16 * 256, stat_off = bar_off + kFewBarBytes;
    const uint32_t bar_full = smem_base + bar_off, bar_empty = bar_full + 8 * kFewMaxStages;
    volatile int* s_abort = reinterpret_cast<volatile int*>(smem_gen + bar_off + 16 * kFewMaxStages);
    float* s_m = reinterpret_cast<float*>(smem_gen + stat_off);            // [kFewWarps][kFewRows] reference of each warp's rows
    float* s_l = s_m + kFewWarps * kFewRows;                               // ... and their sums
    float* s_in = s_l + kFewWarps * kFewRows;                              // [rows this block merges][cluster][kFewOStride]
    uint8_t* s_tail = smem_gen + stat_off + kFewStatBytes + (PAGED ? 0 : few_cluster_bytes(a.num_new * a.G, gridDim.x));
    float4* s_cs = reinterpret_cast<float4*>(s_tail);                      // fused: [n][kAngles]
    uint8_t* s_new = s_tail + (FUSED ? a.num_new * kFewAngleBytes : 0);              // fused: [n][K 256 B | V 256 B]
    const uint32_t bar_in = bar_full + 16 * kFewMaxStages + 8;             // the rows sent here have arrived

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    // ---- the block's share: keys of stages [st0, st1) ----
    int g, slot, L, n, row_base = 0, b = 0, st0, st1;
    int left = 0;                                      // paged: stages of the block's share behind this unit
    uint32_t rank = 0, csize = 1;
    auto episode = [&](int e) {
        if constexpr (PAGED) {
            b = e;
            L = lens.cache_len[b];
            n = lens.new_off[b + 1] - lens.new_off[b];
            row_base = lens.new_off[b] * a.G;
        }
    };
    if (!PAGED) {
        csize = gridDim.x;                             // the cluster spans x
        rank = blockIdx.x;
        g = (int)blockIdx.y;
        slot = (int)blockIdx.z;
        L = a.cache_len;
        n = a.num_new;
        const int ns = (L + n + kFewKeys - 1) / kFewKeys;
        const int lo = slot * ns / a.num_splits, len = (slot + 1) * ns / a.num_splits - lo;
        st0 = lo + (int)rank * len / (int)csize;
        st1 = lo + ((int)rank + 1) * len / (int)csize;
    } else {
        if constexpr (PAGED) {
            const int item = (int)blockIdx.x, first = a.share > 0 ? item * a.share : item;
            int lo = 0, hi = a.batch;                  // largest b with item_off[b] <= first
            while (hi - lo > 1) {
                const int mid = (lo + hi) >> 1;
                if (lens.item_off[mid] <= first) lo = mid; else hi = mid;
            }
            episode(lo);
            const int end = lens.item_off[a.batch], rem = first - lens.item_off[b];
            if (first >= end || n <= 0) return;
            const int ns = (L + n + kFewKeys - 1) / kFewKeys;
            if (a.share > 0) {
                g = (int)((unsigned)rem / (unsigned)ns);
                st0 = rem - g * ns;
                left = min(a.share, end - first);
                st1 = min(ns, st0 + left);
                left -= st1 - st0;
                slot = item - (int)fast_div((uint32_t)(first - st0), a.div_share);      // shares that the unit met before
            } else {
                const int per_head = (int)((unsigned)(lens.item_off[b + 1] - lens.item_off[b]) / (unsigned)a.Hkv);    // one row unit: the split count
                g = (int)((unsigned)rem / (unsigned)per_head);
                slot = rem - g * per_head;
                const int nkv = (L + n + kTileN - 1) / kTileN;                           // work items are cut at 128-key tiles
                st0 = 2 * (int)((unsigned)slot * (unsigned)nkv / (unsigned)per_head);
                st1 = min(2 * (int)((unsigned)(slot + 1) * (unsigned)nkv / (unsigned)per_head), ns);
            }
        }
    }
    auto next_unit = [&]() {                           // the share goes on at the start of the next (episode, kv head)
        if constexpr (PAGED) {
            if (++g == a.Hkv) {
                g = 0;
                int e = b;
                do ++e; while (lens.new_off[e + 1] == lens.new_off[e]);
                episode(e);
            }
            slot = st0 = 0;
            st1 = min((L + n + kFewKeys - 1) / kFewKeys, left);
            left -= st1;
        }
    };
    int rows = n * a.G;
    int count = st1 - st0;

    if (tid == 0) {
        for (int i = 0; i < stages; ++i) {
            ptx::mbar_init(bar_full + 8 * i, 1);
            ptx::mbar_init(bar_empty + 8 * i, kFewWarps / kFewGroups);
        }
        ptx::mbar_init(bar_in, 1);
        ptx::fence_barrier_init();
        *s_abort = 0;
        // this block merges the rows rank, rank + csize, ...: each comes from every block of the cluster
        if (csize > 1 && (int)rank < rows)
            ptx::mbar_expect_tx(bar_in, (uint32_t)((rows - (int)rank + (int)csize - 1) / (int)csize) * csize * 520u);
        ptx::prefetch_tensormap(&tm_k);
        ptx::prefetch_tensormap(&tm_v);
    }
    __syncthreads();
    if (csize > 1) ptx::cluster_arrive_relaxed();      // (waited for before the first row is sent)
    ptx::grid_launch_dependents();
    ptx::grid_dependency_wait();

    // stages are taken from the last key backwards: the new tokens' stage is the first to land
    auto load_stage = [&](int i, int at, int pg) {
        const int s = st1 - 1 - i;
        const uint32_t dst = smem_base + at * kFewStageBytes, bar = bar_full + 8 * at;
        ptx::mbar_expect_tx(bar, kFewStageBytes);
        if (PAGED) {
            ptx::tma_load_4d(dst, &tm_k, bar, 0, 0, g, pg);
            ptx::tma_load_4d(dst + 8192, &tm_k, bar, 64, 0, g, pg);
            ptx::tma_load_4d(dst + 16384, &tm_v, bar, 0, 0, g, pg);
            ptx::tma_load_4d(dst + 24576, &tm_v, bar, 64, 0, g, pg);
        } else {
            const int key0 = s * kFewKeys;
            ptx::tma_load_3d(dst, &tm_k, bar, 0, key0, g);
            ptx::tma_load_3d(dst + 8192, &tm_k, bar, 64, key0, g);
            ptx::tma_load_3d(dst + 16384, &tm_v, bar, 0, key0, g);
            ptx::tma_load_3d(dst + 24576, &tm_v, bar, 64, key0, g);
        }
    };
    if (!PAGED && warp == kFewWarps && lane == 0)
        for (int i = 0; i < count && i < stages; ++i) load_stage(i, i, 0);
    bool ok = true;
    if (PAGED && warp == kFewWarps) {
        // ================= producer =================
        // (the whole warp: a page number costs a round trip to L2, so the lanes fetch 32 of them at once)
        int at = 0;
        uint32_t phase = 1;                            // of the ring's first turn: its slots are free
        for (;;) {
            const int* pages = a.page_table + (long)b * a.max_pages + st1 - 1;
            int pg = 0;
            for (int i = 0; i < st1 - st0 && ok; ++i) {
                if ((i & 31) == 0) pg = i + lane < st1 - st0 ? pages[-(i + lane)] : 0;
                const int page = __shfl_sync(0xffffffffu, pg, i & 31);
                if (lane == 0) {
                    ok = wait_bounded(bar_empty + 8 * at, phase, kDevTimeoutProducer, a.status, s_abort);
                    if (ok) load_stage(i, at, page);
                }
                ok = __shfl_sync(0xffffffffu, (int)ok, 0) != 0;
                if (++at == stages) { at = 0; phase ^= 1; }
            }
            if (!ok || left == 0) break;
            next_unit();
        }
        if (lane == 0 && (!ok || *s_abort)) {
            const long long t0 = clock64();            // loads in flight land before the block may leave
            while (clock64() - t0 < 400000) { }
        }
        return;
    }
    // the compute warps of a paged block go from unit to unit on a barrier of their own
    auto sync = [&]() {
        if (PAGED) asm volatile("bar.sync 1, %0;" :: "n"(32 * kFewWarps) : "memory");
        else __syncthreads();
    };
    constexpr int kTeam = kFewWarps + (PAGED ? 0 : 1);                     // warps that share the work around the products
    constexpr int kQPer = (MT * 16 * 16 + 32 * kTeam - 1) / (32 * kTeam);
    constexpr bool kAhead = PAGED && MT == 1;          // the next unit's are requested before this one is merged (two row
                                                       // tiles leave no registers for them: 69 us against 64)
    uint4 qx[kQPer];                                   // the unit's queries on their way to shared memory
    auto load_q = [&]() {
#pragma unroll
        for (int k = 0; k < kQPer; ++k) {
            const int i = tid + k * 32 * kTeam, r = i >> 4;
            qx[k] = make_uint4(0u, 0u, 0u, 0u);
            if (i < MT * 16 * 16 && r < n * a.G) qx[k] = reinterpret_cast<const uint4*>(a.q_rot_in + ((long)g * a.rows + row_base + r) * 128)[i & 15];
        }
    };
    int i0 = 0;                                        // ring index of the unit's first stage
    for (;;) {

    // ---- queries into shared memory (rows past the last one are zeros) ----
    auto q_slot = [&](int r, int chunk) -> uint4* {    // 16-byte chunk 0..15 of row r: two 64-channel blocks
        return reinterpret_cast<uint4*>(smem_gen + q_off + (chunk >> 3) * (MT * 16 * 128) + swz(r, chunk & 7));
    };
    if (!FUSED) {
        if (!kAhead || i0 == 0) load_q();
#pragma unroll
        for (int k = 0; k < kQPer; ++k) {
            const int i = tid + k * 32 * kTeam;
            if (i < MT * 16 * 16) *q_slot(i >> 4, i & 15) = qx[k];
        }
    } else {
        // a warp per head vector, two channel pairs per lane: rows 0 .. rows-1 are queries, then the new
        // keys and the new values
        const bool own_new = st1 * kFewKeys > L && count > 0;     // new tokens in this block's range
        const int items = rows + (own_new ? 2 * n : 0);
        auto source = [&](int it) -> const __nv_bfloat16* {
            if (it < rows) {
                const int tok = (int)fast_div((uint32_t)it, a.div_g);
                return a.q_new + tok * a.q_stride + (long)(g * a.G + it - tok * a.G) * 128;
            }
            const int e = it - rows;
            return e < n ? a.k_new + e * a.k_stride + (long)g * 128 : a.v_new + (e - n) * a.v_stride + (long)g * 128;
        };
        uint32_t lo = 0, hi = 0;
        if (warp < items) {
            const uint32_t* src = reinterpret_cast<const uint32_t*>(source(warp));
            lo = src[lane];
            hi = src[lane + 32];
        }
        for (int i = tid; i < n * 64; i += kFewThreads) {
            const int tok = i >> 6, j = i & 63;
            Rotation<__nv_bfloat16>::put(s_cs + tok * Rotation<__nv_bfloat16>::kAngles, j,
                                         a.table ? a.table[((long)L + tok - a.table_first) * 64 + j] : rope_cos_sin((long)L + tok, j, 128, a.log2_theta));
        }
        for (int i = rows * 16 + tid; i < MT * 16 * 16; i += kFewThreads) *q_slot(i >> 4, i & 15) = make_uint4(0u, 0u, 0u, 0u);
        __syncthreads();
        for (int it = warp; it < items; it += kFewWarps + 1) {
            if (it != warp) {
                const uint32_t* src = reinterpret_cast<const uint32_t*>(source(it));
                lo = src[lane];
                hi = src[lane + 32];
            }
            const bool is_q = it < rows, is_v = it >= rows + n;
            const int tok = is_q ? (int)fast_div((uint32_t)it, a.div_g) : is_v ? it - rows - n : it - rows;
            uint32_t x = lo, y = hi;
            if (!is_v) {
                typedef Rotation<__nv_bfloat16> R;
                const float4* cs = s_cs + tok * R::kAngles + R::place(lane);
                R::turn_pair(cs[0], cs[1], lo, hi, x, y);
            }
            if (is_q) {
                reinterpret_cast<uint32_t*>(q_slot(it, lane >> 2))[lane & 3] = x;
                reinterpret_cast<uint32_t*>(q_slot(it, 8 + (lane >> 2)))[lane & 3] = y;
                if (rank == 0 && slot == 0) {
                    uint32_t* dst = reinterpret_cast<uint32_t*>(a.q_rot + ((long)g * a.rows + it) * 128);
                    dst[lane] = x;
                    dst[lane + 32] = y;
                }
            } else {
                const int key = L + tok;
                if (key < st0 * kFewKeys || key >= st1 * kFewKeys) continue;
                uint32_t* dst = reinterpret_cast<uint32_t*>((is_v ? a.v_cache : a.k_cache) + ((long)g * a.cache_cap + key) * 128);
                dst[lane] = x;
                dst[lane + 32] = y;
                uint32_t* keep = reinterpret_cast<uint32_t*>(s_new + tok * 512 + (is_v ? 256 : 0));
                keep[lane] = x;
                keep[lane + 32] = y;
            }
        }
        if (own_new) {
            // the new rows into the stages they belong to, once the loads of those stages have landed
            // (the first stages of the ring; n <= 16 tokens touch at most two)
            __syncthreads();
            const int first = max(L, st0 * kFewKeys);
            const int touched = st1 - first / kFewKeys;
            bool ok = true;
            for (int i = 0; i < touched && ok; ++i)
                ok = wait_bounded(bar_full + 8 * i, 0, kDevTimeoutMmaKV, a.status, s_abort);
            const int own = min(L + n, st1 * kFewKeys) - first;
            for (int i = tid; i < own * 32 && ok; i += kFewThreads) {
                const int key = first + (i >> 5), c = i & 31;            // 16 chunks of K, 16 of V
                const int at = st1 - 1 - key / kFewKeys;
                uint8_t* dst = smem_gen + at * kFewStageBytes + (c >> 3) * 8192 + swz(key & 63, c & 7);
                *reinterpret_cast<uint4*>(dst) = reinterpret_cast<const uint4*>(s_new + (key - L) * 512)[c];
            }
            ptx::fence_proxy_async();                  // a later load into these stages comes after these writes
        }
    }
    sync();

    if (!PAGED && warp == kFewWarps) {
        // ================= producer =================
        if (lane == 0) {
            for (int i = stages; i < count && ok; ++i) {
                ok = wait_bounded(bar_empty + 8 * (i % stages), ((i / stages) & 1) ^ 1, kDevTimeoutProducer, a.status, s_abort);
                if (ok) load_stage(i, i % stages, 0);
            }
            if (!ok || *s_abort) {
                const long long t0 = clock64();        // loads in flight land before the block may leave
                while (clock64() - t0 < 400000) { }
            }
        }
        __syncwarp();
    }

    // ================= compute warps =================
    const int mt = warp % MT, share = (warp & 3) / MT, group = warp >> 2;   // (the producer warp computes nothing)
    float o[16][4];                                    // 16 rows x 128 channels: 8-channel tiles
    float m[2] = {-INFINITY, -INFINITY}, l[2] = {0.f, 0.f};      // of rows lane / 4 and + 8; m in score units
#pragma unroll
    for (int t = 0; t < 16; ++t)
#pragma unroll
        for (int e = 0; e < 4; ++e) o[t][e] = 0.f;

    if (warp < kFewWarps) {
        // lane addresses of ldmatrix: matrix i = lane / 8, row lane % 8 of it
        const int mi = lane >> 3, mr = lane & 7;
        uint32_t q[8][4];
        {
            const int r = mt * 16 + (mi & 1) * 8 + mr;
#pragma unroll
            for (int ks = 0; ks < 8; ++ks)
                ptx::ldmatrix_x4(q[ks], smem_base + q_off + (ks >> 2) * (MT * 16 * 128) + swz(r, (ks & 3) * 2 + (mi >> 1)));
        }
        int bound[2];                                  // last visible key of the thread's two rows
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int r = mt * 16 + h * 8 + (lane >> 2);
            bound[h] = r < rows ? L + (int)fast_div((uint32_t)r, a.div_g) : 0x3fffffff;      // padding rows: nothing to mask
        }
        const int k0 = share * kShare;
        const int k_row = k0 + (mi >> 1) * 8 + mr, k_chunk = mi & 1;      // scores: key, channel half
        const int v_row = k0 + (mi & 1) * 8 + mr, v_chunk = mi >> 1;      // products: key, channel half
        const float headroom = 8.f / a.scale_log2;

        uint32_t kf[MT][8][4], vf[8][4];
        auto load_k = [&](int at) {
            const uint32_t base = smem_base + at * kFewStageBytes;
#pragma unroll
            for (int ks = 0; ks < 8; ++ks)
#pragma unroll
                for (int kk = 0; kk < MT; ++kk)
                    ptx::ldmatrix_x4(kf[kk][ks], base + (ks >> 2) * 8192 + kk * 16 * 128 + swz(k_row, (ks & 3) * 2 + k_chunk));
        };
        auto load_v = [&](int at, int kk) {
            const uint32_t base = smem_base + at * kFewStageBytes + 16384 + kk * 16 * 128;
#pragma unroll
            for (int t = 0; t < 8; ++t)
                ptx::ldmatrix_x4_trans(vf[t], base + (t >> 2) * 8192 + swz(v_row, (t & 3) * 2 + v_chunk));
        };
        // Two warps per scheduler: an iteration is a chain of latencies (barrier, fragments, scores,
        // exponentials, products), so all fragments are requested ahead of the products that need them.
        const int skip = (group ^ i0) & 1;             // slots belong to the groups, whichever stage they hold
        int at = PAGED ? (i0 + skip) % kFewPagedStages : group;            // slot of stage i, and its phase
        uint32_t phase = PAGED ? ((i0 + skip) / kFewPagedStages) & 1 : 0;
        for (int i = skip; i < count && ok; i += kFewGroups) {
            ok = wait_bounded(bar_full + 8 * at, phase, kDevTimeoutMmaKV, a.status, s_abort);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            load_k(at);
            load_v(at, 0);
            float s[MT][2][2][4];                      // [16 keys][channel parity][8-key tile]
#pragma unroll
            for (int kk = 0; kk < MT; ++kk)
#pragma unroll
                for (int t = 0; t < 4; ++t)
#pragma unroll
                    for (int e = 0; e < 4; ++e) s[kk][t >> 1][t & 1][e] = 0.f;
#pragma unroll
            for (int ks = 0; ks < 8; ++ks)
#pragma unroll
                for (int kk = 0; kk < MT; ++kk) {
                    ptx::mma_bf16(s[kk][ks & 1][0], q[ks], kf[kk][ks][0], kf[kk][ks][1]);
                    ptx::mma_bf16(s[kk][ks & 1][1], q[ks], kf[kk][ks][2], kf[kk][ks][3]);
                }
            float x[2 * MT][4];                        // 8-key tiles
#pragma unroll
            for (int t = 0; t < 2 * MT; ++t)
#pragma unroll
                for (int e = 0; e < 4; ++e) x[t][e] = s[t >> 1][0][t & 1][e] + s[t >> 1][1][t & 1][e];
            const int key0 = (st1 - 1 - i) * kFewKeys + k0;
            if (key0 + kShare - 1 > L) {               // (every row sees the keys up to L)
#pragma unroll
                for (int t = 0; t < 2 * MT; ++t)
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        if (key0 + t * 8 + (lane & 3) * 2 + (e & 1) > bound[e >> 1]) x[t][e] = -INFINITY;
            }
            // a row's reference moves only when a score exceeds it by 2^8 (the final division by the
            // row sum makes any reference exact)
            float mx[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                mx[h] = fmaxf(x[0][2 * h], x[0][2 * h + 1]);
#pragma unroll
                for (int t = 1; t < 2 * MT; ++t) mx[h] = ptx::max3(mx[h], x[t][2 * h], x[t][2 * h + 1]);
            }
            if (__any_sync(0xffffffffu, mx[0] > m[0] + headroom || mx[1] > m[1] + headroom)) {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    float y = mx[h];
                    y = fmaxf(y, __shfl_xor_sync(0xffffffffu, y, 1));
                    y = fmaxf(y, __shfl_xor_sync(0xffffffffu, y, 2));
                    const float m_new = fmaxf(m[h], y);
                    const float alpha = m_new == -INFINITY ? 1.f : ptx::ex2((m[h] - m_new) * a.scale_log2);
                    m[h] = m_new;
                    l[h] *= alpha;
#pragma unroll
                    for (int t = 0; t < 16; ++t) {
                        o[t][2 * h] *= alpha;
                        o[t][2 * h + 1] *= alpha;
                    }
                }
            }
            const float n0 = m[0] == -INFINITY ? 0.f : -m[0] * a.scale_log2, n1 = m[1] == -INFINITY ? 0.f : -m[1] * a.scale_log2;
            uint32_t p[MT][4];                         // 16 keys each
#pragma unroll
            for (int t = 0; t < 2 * MT; ++t) {
                const float p0 = ptx::ex2(fmaf(x[t][0], a.scale_log2, n0)), p1 = ptx::ex2(fmaf(x[t][1], a.scale_log2, n0));
                const float p2 = ptx::ex2(fmaf(x[t][2], a.scale_log2, n1)), p3 = ptx::ex2(fmaf(x[t][3], a.scale_log2, n1));
                l[0] += p0 + p1;
                l[1] += p2 + p3;
                p[t >> 1][(t & 1) * 2] = ptx::pack_bf16x2(p0, p1);
                p[t >> 1][(t & 1) * 2 + 1] = ptx::pack_bf16x2(p2, p3);
            }
#pragma unroll
            for (int kk = 0; kk < MT; ++kk) {
                if (kk > 0) load_v(at, kk);
#pragma unroll
                for (int t = 0; t < 8; ++t) {
                    ptx::mma_bf16(o[2 * t], p[kk], vf[t][0], vf[t][1]);
                    ptx::mma_bf16(o[2 * t + 1], p[kk], vf[t][2], vf[t][3]);
                }
            }
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(bar_empty + 8 * at);
            at += kFewGroups;
            if (at >= stages) { at -= stages; phase ^= 1; }
        }
        m[0] *= a.scale_log2;                          // (log2 units from here on)
        m[1] *= a.scale_log2;
    }

    // ---- the warps' results into shared memory (not paged: where the ring was, every stage has been consumed) ----
    if (!PAGED) __syncthreads();
    const int done_g = g, done_slot = slot, done_base = row_base;
    const bool more = PAGED && left > 0;
    if (more) {
        i0 += count;
        next_unit();
        if (kAhead) load_q();
    }
    float* s_o = reinterpret_cast<float*>(PAGED ? s_tail : smem_gen);                 // [kFewWarps][16][kFewOStride]
    if (warp < kFewWarps) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            if (mt * 16 + h * 8 >= rows) break;        // padding rows only
            float sum = l[h];
            sum += __shfl_xor_sync(0xffffffffu, sum, 1);
            sum += __shfl_xor_sync(0xffffffffu, sum, 2);
            const int r = h * 8 + (lane >> 2);
            if ((lane & 3) == 0) {
                s_m[(warp / MT) * kFewRows + mt * 16 + r] = m[h];
                s_l[(warp / MT) * kFewRows + mt * 16 + r] = sum;
            }
            float* dst = s_o + (warp * 16 + r) * kFewOStride + (lane & 3) * 2;
#pragma unroll
            for (int t = 0; t < 16; ++t) *reinterpret_cast<float2*>(dst + t * 8) = make_float2(o[t][2 * h], o[t][2 * h + 1]);
        }
    }
    if (csize > 1) ptx::cluster_wait();                // every block of the cluster has set up its barriers
    sync();
    // merge the WK shares of every row: a warp per row, 4 channels per lane
    for (int r = warp; r < rows; r += kTeam) {
        float M = -INFINITY;
#pragma unroll
        for (int w = 0; w < WK; ++w) M = fmaxf(M, s_m[w * kFewRows + r]);
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
        float sum = 0.f;
#pragma unroll
        for (int w = 0; w < WK; ++w) {
            const float mw = s_m[w * kFewRows + r];
            const float f = mw == -INFINITY ? 0.f : ptx::ex2(mw - M);
            sum = fmaf(f, s_l[w * kFewRows + r], sum);
            const float4 v = *reinterpret_cast<const float4*>(s_o + ((w * MT + (r >> 4)) * 16 + (r & 15)) * kFewOStride + lane * 4);
            acc.x = fmaf(f, v.x, acc.x); acc.y = fmaf(f, v.y, acc.y);
            acc.z = fmaf(f, v.z, acc.z); acc.w = fmaf(f, v.w, acc.w);
        }
        if (csize > 1) {
            // to the block that merges this row, into the place of this block's contribution
            const uint32_t owner = (uint32_t)r % csize;
            const uint32_t at = ptx::smem_u32(s_in + (((uint32_t)r / csize) * csize + rank) * kFewOStride);
            const uint32_t bar = ptx::map_to_cta(bar_in, owner);
            ptx::st_async_f32x4(ptx::map_to_cta(at + lane * 16, owner), acc, bar);
            if (lane == 0) ptx::st_async_f32x2(ptx::map_to_cta(at + 512, owner), M, sum, bar);
        } else {
            few_write_row(a, acc, M, sum, done_g, done_slot, done_base, r, lane);
        }
    }
    if (more) {
        rows = n * a.G;
        count = st1 - st0;
        continue;
    }
    if (csize > 1 && (int)rank < rows) {
        // merge the cluster's contributions to this block's rows
        const bool all = __syncthreads_and(wait_bounded(bar_in, 0, kDevTimeoutSoftmaxX, a.status, s_abort)) != 0;
        if (!all) {
            // gave up: stay until no block of the cluster can send any more (they arrive here or have left)
            ptx::cluster_arrive_relaxed();
            ptx::cluster_wait();
            return;
        }
        for (int k = warp; (int)rank + k * (int)csize < rows; k += kFewWarps + 1) {
            const float* in = s_in + k * (int)csize * kFewOStride;
            float mc = -INFINITY, lc = 0.f;
            if (lane < (int)csize) {
                const float2 ml = *reinterpret_cast<const float2*>(in + lane * kFewOStride + 128);
                mc = ml.x;
                lc = ml.y;
            }
            float M = mc;
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, off));
            const float f = mc == -INFINITY ? 0.f : ptx::ex2(mc - M);
            float sum = f * lc;
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
            float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int c = 0; c < kFewMaxCluster; ++c) {
                const float fc = __shfl_sync(0xffffffffu, f, c);
                if (c < (int)csize) {
                    const float4 v = *reinterpret_cast<const float4*>(in + c * kFewOStride + lane * 4);
                    acc.x = fmaf(fc, v.x, acc.x); acc.y = fmaf(fc, v.y, acc.y);
                    acc.z = fmaf(fc, v.z, acc.z); acc.w = fmaf(fc, v.w, acc.w);
                }
            }
            few_write_row(a, acc, M, sum, g, slot, row_base, (int)rank + k * (int)csize, lane);
        }
    }
    break;
    }
}

}  // namespace evln
