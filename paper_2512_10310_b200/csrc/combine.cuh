// Split-reduction combine kernel: merges the per-split partial outputs of the step attention.
//
//   M = max_s lse_s,  w_s = e^{lse_s - M},  O = sum_s w_s O_s / sum_s w_s,  lse = M + log sum_s w_s
//
// One warp per packed query row (or per 32 channels of one: see the forms below): lane s holds lse_s (at most 32 splits), the maximum and the
// weight sum are warp-shuffle reductions, then each lane merges D/32 contiguous channels with
// vector loads.  The row is rounded once to the storage dtype and written to its place in the
// token-major [n, Hq, D] output.  HBM/L2-bound: S*(D+1) floats in, D elements out per row.
#pragma once

#include <type_traits>

#include "common.cuh"

namespace evln {

struct CombineArgs {
    const float* o_part;     // [S, Hkv, R, D]
    const float* lse_part;   // [S, Hkv, R]
    void* out;               // [n, Hq, D]
    float* lse_out;          // [n, Hq] or null
    int Hkv, G, D;
    int rows;                // R = (total) new tokens * G
    int num_splits;          // contiguous: S for every row
    // batches: per-episode split counts are derived from the lengths
    int batch, chunk_tiles;
    int tail;                // batch of items sharing a cache prefix (own tokens tiled separately)
    FastDiv div_g;           // division by G, by the work-item size in KV tiles (chunk_tiles, at least 1):
    FastDiv div_chunk;       //   a row's warp decodes its place with multiplications (an integer division costs
                             //   as much as the rest of the merge)
    int share;               // fp32 kernel: key tiles per block of equal shares; batches whose blocks took equal shares of the 64-key stages (item_off counts them):
    FastDiv div_share;       //   the shares that met a row's keys are its splits; 0: work items of chunk_tiles
    PackedMap map;           // where output token m goes (identity unless the call serves a packed sequence)
};

// Forms of the kernel, by the most parts of a row and by the rows; the sums keep the order of the parts in all of them, and
// all of them leave out the parts from kCombineFewParts on whose weight is 0 (an infinite value at a key of no weight is then
// not multiplied by 0), so the bits are the same.
//   few   at most kCombineFewParts: no loop behind the first loads, so that the kernel keeps 38 registers and a step of
//         1400 blocks is one wave (196 tokens of the 7B shape: 64 registers and 1.2 waves before)
//   many  a loop over the rest, eight parts at a time; bounded to the 64 registers of eight blocks an SM
//   wide  few rows in many parts: a row's D / 32 warps take 32 channels each, a lane one float of each part, so that up to
//         16 parts are on their way at once, on four times as many SMs
constexpr int kCombineFew = 0, kCombineMany = 1, kCombineWide = 2;
constexpr int kCombineFewParts = 4;

template <typename T, int D, bool PAGED, typename LensT, int FORM>
__global__ void __launch_bounds__(128, FORM == kCombineFew ? 12 : FORM == kCombineMany ? 8 : 1)
combine_kernel(const CombineArgs a, const __grid_constant__ LensT lens)
{
    constexpr bool WIDE = FORM == kCombineWide;
    constexpr int kWarps = WIDE ? D / 32 : 1;                   // warps per row
    constexpr int C = WIDE ? 1 : D / 32;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int col = WIDE ? (warp % kWarps) * 32 + lane : lane * C;      // the lane's first channel
    const uint32_t row = (blockIdx.x * 4u + (uint32_t)warp) / kWarps;   // packed row within kv head (< 2^24, checked on the host)
    const int g = blockIdx.y;
    if (row >= (uint32_t)a.rows) return;
    const uint32_t row_tok = fast_div(row, a.div_g);            // its token among the call's new tokens ...
    const int row_head = (int)(row - row_tok * (uint32_t)a.G);  // ... and its query head within the group

    int S = a.num_splits;
    if constexpr (PAGED) {
        const int tok = (int)row_tok;
        int lo = 0, hi = a.batch;
        while (hi - lo > 1) {
            int mid = (lo + hi) >> 1;
            if (lens.new_off[mid] <= tok) lo = mid; else hi = mid;
        }
        const int b = lo;
        const int n_b = lens.new_off[b + 1] - lens.new_off[b];
        if (a.share > 0) {
            const uint32_t ns = (uint32_t)(lens.cache_len[b] + n_b + kFewKeys - 1) / kFewKeys, at = (uint32_t)lens.item_off[b] + g * ns;
            S = (int)(fast_div(at + ns - 1, a.div_share) - fast_div(at, a.div_share)) + 1;
        } else {
            const int local_row = (int)row - lens.new_off[b] * a.G;
            const int unit = local_row / kUnitRows;                  // (a power of two)
            const int nkv = a.tail ? tail_kv_tiles_fast(lens.cache_len[b], n_b, a.div_g, unit, kUnitRows)
                                   : unit_kv_tiles_fast(lens.cache_len[b], n_b, a.div_g, unit, kUnitRows);
            S = (int)fast_div((uint32_t)(nkv + a.chunk_tiles - 1), a.div_chunk);
        }
    }

    if constexpr (std::is_same<LensT, SimtTiles>::value) {
        const int rb = (int)row >> 7;
        const uint32_t at = (uint32_t)(g * lens.off[kSimtShareBlocks] + lens.off[rb]), tiles = (uint32_t)(lens.off[rb + 1] - lens.off[rb]);
        S = (int)(fast_div(at + tiles - 1, a.div_share) - fast_div(at, a.div_share)) + 1;
    }

    const long stride_s = (long)a.Hkv * a.rows;           // rows between consecutive splits
    const long prow0 = (long)g * a.rows + row;
    // (so far launch parameters only: a row's warp knows its place before the partials exist)
    asm volatile("griddepcontrol.wait;" ::: "memory");          // programmatic dependent launch: inputs ready
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    constexpr int kPre = WIDE ? 16 : kCombineFewParts;
    // (Letting every lane read all log-sum-exps of a row with few splits, so that the maximum and
    // the weights need no shuffles, was measured slower: 3.85 against 3.45 us at the 7B step.)
    float my_lse = (lane < S) ? a.lse_part[prow0 + lane * stride_s] : -INFINITY;
    // the first partial rows do not depend on the weights: their loads go out with the lse load
    float pre[kPre][C];
#pragma unroll
    for (int s = 0; s < kPre; ++s) {
        if (s < S) {
            const float* op = a.o_part + (prow0 + s * stride_s) * D + col;
            if (C == 4) {
                float4 x = *reinterpret_cast<const float4*>(op);
                pre[s][0] = x.x; pre[s][1] = x.y; pre[s][2] = x.z; pre[s][3] = x.w;
            } else {
#pragma unroll
                for (int c = 0; c < C; ++c) pre[s][c] = op[c];
            }
        } else {
#pragma unroll
            for (int c = 0; c < C; ++c) pre[s][c] = 0.f;
        }
    }
    float M = my_lse;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, off));
    float w = (my_lse == -INFINITY) ? 0.f : expf(my_lse - M);    // M = -inf only if all are
    float wsum = w;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) wsum += __shfl_xor_sync(0xffffffffu, wsum, off);

    float acc[C];
#pragma unroll
    for (int c = 0; c < C; ++c) acc[c] = 0.f;
#pragma unroll
    for (int s = 0; s < kPre; ++s) {
        const float ws = __shfl_sync(0xffffffffu, w, s);      // 0 for s >= S and for empty splits
        if (s < kCombineFewParts || ws != 0.f) {              // (see the forms above)
#pragma unroll
            for (int c = 0; c < C; ++c) acc[c] = fmaf(ws, pre[s][c], acc[c]);
        }
    }
    // the remaining splits, kBatch at a time: their loads are in flight together, the sums keep the
    // order of the splits
    constexpr int kBatch = WIDE ? 16 : 8;
    for (int s0 = kPre; FORM != kCombineFew && s0 < S; s0 += kBatch) {
        float v[kBatch][C];
#pragma unroll
        for (int k = 0; k < kBatch; ++k) {
            const int s = s0 + k;
            if (s < S) {
                const float* op = a.o_part + (prow0 + s * stride_s) * D + col;
                if (C == 4) {
                    float4 x = *reinterpret_cast<const float4*>(op);
                    v[k][0] = x.x; v[k][1] = x.y; v[k][2] = x.z; v[k][3] = x.w;
                } else {
#pragma unroll
                    for (int c = 0; c < C; ++c) v[k][c] = op[c];
                }
            } else {
#pragma unroll
                for (int c = 0; c < C; ++c) v[k][c] = 0.f;
            }
        }
#pragma unroll
        for (int k = 0; k < kBatch; ++k) {
            const float ws = (s0 + k < S) ? __shfl_sync(0xffffffffu, w, s0 + k) : 0.f;   // 0 for empty splits too
            if (ws != 0.f) {                                                            // uniform across the warp
#pragma unroll
                for (int c = 0; c < C; ++c) acc[c] = fmaf(ws, v[k][c], acc[c]);
            }
        }
    }
    const float inv = (wsum > 0.f) ? 1.f / wsum : 0.f;

    const long tok = packed_row(a.map, (int)row_tok);
    const int h = g * a.G + row_head;
    const int Hq = a.Hkv * a.G;
    T* dst = (T*)a.out + (tok * Hq + h) * D + col;
    __align__(16) T y[C];
#pragma unroll
    for (int c = 0; c < C; ++c) from_float(acc[c] * inv, y[c]);
    constexpr int kBytes = C * (int)sizeof(T);
    if constexpr (kBytes == 16) *reinterpret_cast<uint4*>(dst) = *reinterpret_cast<const uint4*>(y);
    else if constexpr (kBytes == 8) *reinterpret_cast<uint2*>(dst) = *reinterpret_cast<const uint2*>(y);
    else if constexpr (kBytes == 4) *reinterpret_cast<uint32_t*>(dst) = *reinterpret_cast<const uint32_t*>(y);
    else *dst = y[0];
    if (a.lse_out && col == 0) a.lse_out[tok * Hq + h] = (wsum > 0.f) ? M + logf(wsum) : -INFINITY;
}

// The combine step of rows whose keys were not split: the one partial of a row is its output, rounded and put in its
// place.  Same bits as the merge above (weight and sum are 1), without its chain of loads and shuffles.  Bound by the
// boundary between two launches and then by L2.
constexpr int kRoundVectors = 2;      // 16-byte vectors of the output per thread, all in flight

template <typename T, int D>
__global__ void __launch_bounds__(256)
round_out_kernel(const CombineArgs a)
{
    constexpr int V = VecTraits<T>::kVec, kPerRow = D / V;
    const int g = blockIdx.y;
    const uint32_t i0 = blockIdx.x * (256u * kRoundVectors) + threadIdx.x;      // (rows per kv head are at most 2^24)
    const float* part = a.o_part + (long)g * a.rows * D;
    const int Hq = a.Hkv * a.G;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    float4 x[kRoundVectors][V / 4];
    float lse[kRoundVectors];
#pragma unroll
    for (int k = 0; k < kRoundVectors; ++k) {
        const uint32_t i = i0 + 256u * k, row = i / kPerRow;
        if (row >= (uint32_t)a.rows) continue;
#pragma unroll
        for (int c = 0; c < V / 4; ++c) x[k][c] = *reinterpret_cast<const float4*>(part + (long)i * V + 4 * c);
        if (a.lse_out && i % kPerRow == 0) lse[k] = a.lse_part[(long)g * a.rows + row];
    }
#pragma unroll
    for (int k = 0; k < kRoundVectors; ++k) {
        const uint32_t i = i0 + 256u * k, row = i / kPerRow;
        if (row >= (uint32_t)a.rows) continue;
        const uint32_t tok = fast_div(row, a.div_g);
        const long at = (long)tok * Hq + g * a.G + (int)(row - tok * (uint32_t)a.G);
        __align__(16) T y[V];
#pragma unroll
        for (int c = 0; c < V / 4; ++c) {
            from_float(x[k][c].x, y[4 * c]);
            from_float(x[k][c].y, y[4 * c + 1]);
            from_float(x[k][c].z, y[4 * c + 2]);
            from_float(x[k][c].w, y[4 * c + 3]);
        }
        *reinterpret_cast<uint4*>((T*)a.out + at * D + (i % kPerRow) * V) = *reinterpret_cast<const uint4*>(y);
        if (a.lse_out && i % kPerRow == 0) a.lse_out[at] = lse[k];
    }
}

// Unsplit paged batches: the rows are final (rounded, in output order) in the workspace: n * Hq rows of
// 16-byte vectors and their log-sum-exps go to the caller's buffers.  HBM/L2-bound: a third of the bytes
// that one set of fp32 partials would move.
struct CopyOutArgs {
    const uint4* src;
    uint4* dst;
    const float* lse_src;
    float* lse_dst;          // or null
    long vectors, rows;
};
constexpr int kCopyVectors = 4;      // per thread, all in flight

__global__ void __launch_bounds__(256)
copy_out_kernel(const CopyOutArgs a)
{
    const long i0 = (long)blockIdx.x * (256 * kCopyVectors) + threadIdx.x;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    uint4 v[kCopyVectors];
#pragma unroll
    for (int k = 0; k < kCopyVectors; ++k)
        if (i0 + 256 * k < a.vectors) v[k] = a.src[i0 + 256 * k];
#pragma unroll
    for (int k = 0; k < kCopyVectors; ++k)
        if (i0 + 256 * k < a.vectors) a.dst[i0 + 256 * k] = v[k];
    if (a.lse_dst) {                 // 16 vectors per row
        const long r = (long)blockIdx.x * (256 * kCopyVectors / 16) + threadIdx.x;
        if (threadIdx.x < 256 * kCopyVectors / 16 && r < a.rows) a.lse_dst[r] = a.lse_src[r];
    }
}

}  // namespace evln
