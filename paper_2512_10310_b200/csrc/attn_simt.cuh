// SIMT step attention in float FMAs (no tensor cores): bf16 with head_dim 64, and, when the caller asks for
// it (EVLN_KERNEL_SIMT), any type as an on-device cross-check of the tensor-core kernels.
//
// Bound: the FMA pipes (4 D flop per visible pair; 128 FMA per SM and cycle).  A block of 256 threads
// owns a tile of 16 * RPT packed query rows of one kv head and walks its split's keys 64 at a time:
//   thread (ty, tx) = (tid / 16, tid % 16) holds rows ty, ty + 16, ... (RPT of them), scores the keys
//   tx, tx + 16, tx + 32, tx + 48 of the tile, and accumulates channels 4 tx .. 4 tx + 3 (and + 64).
//   Everything it multiplies comes out of shared memory as 16-byte vectors and is used RPT (or 4)
//   times; products go two at a time (packed FMAs over channel pairs).  Rows of Q, K and P are padded
//   so that neither the 16 keys nor the two rows a warp touches at once meet in a bank.
//   One K and one V tile are resident: the next K tile is fetched (cp.async) while the products with V
//   run, the next V tile while the next scores run.
// RPT = 8 (128 rows): each vector from shared memory feeds 8 rows, the FMA pipes are the limit.
// RPT = 2 (32 rows): a quarter of the work per block, for calls whose 128-row tiles would leave SMs
// idle; shared-memory reads bound it at about the same rate per row (K and V vectors feed 2 rows).
// TilesT = SimtTiles (RPT = 8): one block per SM with an equal share of all visible (row block, key tile)
// pairs instead of (row block, kv head, split) blocks, whose whole numbers left SMs idle (196 tokens of the 7B
// shape over 1024 cached: 44 row blocks in three splits kept 132 SMs busy for up to 7 tiles each, now 148 for
// 6: 108.5 and 96.4 us a step).  A share goes through the ends of row blocks; a row is split where two shares meet.
#pragma once

#include <type_traits>

#include "common.cuh"
#include "ptx_sm100.cuh"

namespace evln {

struct SimtAttnArgs {
    const void* q_rot;     // [Hkv, R, D]
    const void* k_cache;   // [Hkv, cap, D]
    const void* v_cache;
    float* o_part;         // [S, Hkv, R, D]
    float* lse_part;       // [S, Hkv, R]
    int Hkv, G;
    int cache_len, num_new, cache_cap;
    int num_splits;
    int share;             // key tiles per block, 0: a block per (row block, kv head, split)
    float scale;
    // attn_f32.cuh only:
    float scale_lo;                 // rest of the scale
    float scale2_hi, scale2_lo;     // scale * log2(e) in two parts
    float diff_min;                 // difference of scores whose weight is 0
    uint32_t huge;                  // magnitude (a bf16 number's bits) from which on a query or key is not split
    int* status;                    // device status word
};

constexpr int kSimtThreads = 256;
constexpr int kSimtKeys = 64;                           // keys per tile
constexpr int kSimtPStride = kSimtKeys + 16;            // two neighbouring rows 16 banks apart
template <int D, int RPT> constexpr int simt_smem_bytes()
{
    return (16 * RPT * (D + 4) + kSimtKeys * (D + 4) + kSimtKeys * D + 16 * RPT * kSimtPStride) * (int)sizeof(float);
}

// Row `row` of a tile to shared memory, 4 channels at `d`; rows at or past `rows` read as zeros.
template <typename T>
__device__ __forceinline__ void simt_fetch(float* dst, const T* base, int row, int rows, int D, int d)
{
    if constexpr (sizeof(T) == 4) {
        ptx::cp_async16(ptx::smem_u32(dst), base + (row < rows ? (long)row * D + d : 0), row < rows);
    } else {
        uint2 raw = make_uint2(0u, 0u);
        if (row < rows) raw = *reinterpret_cast<const uint2*>(base + (long)row * D + d);
        *reinterpret_cast<float4*>(dst) = make_float4(__uint_as_float(raw.x << 16), __uint_as_float(raw.x & 0xffff0000u),
                                                      __uint_as_float(raw.y << 16), __uint_as_float(raw.y & 0xffff0000u));
    }
}

// One row over the `keys` keys from kb / vb on that it sees, by one warp, key after key: see the end of the kernel.
// (Out of line and with plain arguments, so that the tile loop keeps its registers: inlined, 97.2 us instead of
// 94.9 for 196 tokens of the 7B shape over 1024 cached.)
template <typename T, int D>
__device__ __noinline__ void simt_row(const T* q, const T* kb, const T* vb, float* op, float* lp, float scale, int keys)
{
    constexpr int C = D / 32;
    const int lane = threadIdx.x & 31;
    q += lane * C;
    float m = -INFINITY, l = 0.f, o[C];
#pragma unroll
    for (int c = 0; c < C; ++c) o[c] = 0.f;
    for (int t = 0; t < keys; ++t) {
        float s = 0.f;
#pragma unroll
        for (int c = 0; c < C; ++c) s = fmaf(to_float(q[c]), to_float(kb[(long)t * D + lane * C + c]), s);
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
        s *= scale;
        const float m_new = fmaxf(m, s), ref = (m_new == -INFINITY) ? 0.f : m_new;
        const float alpha = expf(m - ref), p = expf(s - ref);
        m = m_new;
        l = l * alpha + p;
#pragma unroll
        for (int c = 0; c < C; ++c) o[c] = fmaf(p, to_float(vb[(long)t * D + lane * C + c]), o[c] * alpha);
    }
    const float inv = (l > 0.f) ? 1.f / l : 0.f;
#pragma unroll
    for (int c = 0; c < C; ++c) op[lane * C + c] = o[c] * inv;
    if (lane == 0) *lp = (l > 0.f) ? m + logf(l) : -INFINITY;
}

// (RPT = 2: three blocks an SM; left to itself the compiler takes 64 registers at head_dim 64, for four that never meet, and
// keeps too few loads in flight: 4 query heads, 239 tokens over 1403 keys 42.8 us against 34.5)
template <typename T, int D, int RPT, typename TilesT>
__global__ void __launch_bounds__(kSimtThreads, RPT == 2 ? 3 : 1)
attn_simt_kernel(const SimtAttnArgs a, const __grid_constant__ TilesT tiles)
{
    constexpr bool SHARE = std::is_same<TilesT, SimtTiles>::value;
    constexpr int NT = kSimtThreads;
    constexpr int TY = NT / 16, BM = TY * RPT, BN = kSimtKeys, QS = D + 4, PS = kSimtPStride;
    constexpr int kUnrollQ = RPT >= 8 ? 4 : 8, kUnrollV = RPT >= 8 ? 2 : 4;   // loads in flight ahead of the products
    constexpr int NV = D / 64;                          // 4-channel groups of O per thread
    constexpr int kVec = D / 4;                         // 16-byte vectors per row
    extern __shared__ __align__(16) float simt_smem[];
    float* s_q = simt_smem;                             // [BM][QS]
    float* s_k = s_q + BM * QS;                         // [BN][QS]
    float* s_v = s_k + BN * QS;                         // [BN][D]
    float* s_p = s_v + BN * D;                          // [BM][PS]

    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int R = a.num_new * a.G;
    const int total = a.cache_len + a.num_new;
    int rb, g, split, j_lo, j_hi;                       // the row block and its key tiles
    int left = 0;                                       // tiles of the block's share behind them
    if constexpr (SHARE) {
        const int per_head = tiles.off[kSimtShareBlocks], first = blockIdx.x * a.share;
        g = first / per_head;
        const int rem = first - g * per_head;
        rb = 0;
        while (tiles.off[rb + 1] <= rem) ++rb;
        j_lo = rem - tiles.off[rb];
        left = min(a.share, per_head * a.Hkv - first);
        j_hi = min(tiles.off[rb + 1] - tiles.off[rb], j_lo + left);
        left -= j_hi - j_lo;
        split = blockIdx.x - (first - j_lo) / a.share;  // shares that the row block met before
    } else {
        rb = blockIdx.x;
        g = blockIdx.y;
        split = blockIdx.z;
        const int all_tiles = (total + BN - 1) / BN;    // splits are whole key tiles
        j_lo = (int)((long)split * all_tiles / a.num_splits);
        j_hi = (int)((long)(split + 1) * all_tiles / a.num_splits);
    }

    ptx::grid_dependency_wait();                        // programmatic dependent launch: inputs ready
    ptx::grid_launch_dependents();
    for (;;) {
    const int row0 = rb * BM;
    const int t_lo = j_lo * BN;
    // keys past the row block's last token are visible to none of its rows
    const int last_row = min(row0 + BM, R) - 1;
    const int t_hi = min(min(total, j_hi * BN), a.cache_len + last_row / a.G + 1);
    int bound[RPT];                                     // last visible key of the thread's rows
#pragma unroll
    for (int r = 0; r < RPT; ++r) bound[r] = a.cache_len + (row0 + r * TY + ty) / a.G;

    const T* qb = (const T*)a.q_rot + ((long)g * R + row0) * D;
    const T* kb = (const T*)a.k_cache + ((long)g * a.cache_cap + t_lo) * D;
    const T* vb = (const T*)a.v_cache + ((long)g * a.cache_cap + t_lo) * D;
    const int keys = t_hi - t_lo, ntiles = keys > 0 ? (keys + BN - 1) / BN : 0;

    auto fetch_k = [&](int j) {
        for (int i = tid; i < BN * kVec; i += NT)
            simt_fetch(s_k + (i / kVec) * QS + (i % kVec) * 4, kb, j * BN + i / kVec, keys, D, (i % kVec) * 4);
    };
    auto fetch_v = [&](int j) {
        for (int i = tid; i < BN * kVec; i += NT)
            simt_fetch(s_v + (i / kVec) * D + (i % kVec) * 4, vb, j * BN + i / kVec, keys, D, (i % kVec) * 4);
    };

    if (ntiles > 0) {
        for (int i = tid; i < BM * kVec; i += NT)
            simt_fetch(s_q + (i / kVec) * QS + (i % kVec) * 4, qb, i / kVec, R - row0, D, (i % kVec) * 4);
        fetch_k(0);
    }
    ptx::cp_async_commit();
    if (ntiles > 0) fetch_v(0);
    ptx::cp_async_commit();

    float m[RPT], l[RPT];
    uint64_t o[RPT][2 * NV];                            // channel pairs
#pragma unroll
    for (int r = 0; r < RPT; ++r) {
        m[r] = -INFINITY;
        l[r] = 0.f;
#pragma unroll
        for (int c = 0; c < 2 * NV; ++c) o[r][c] = 0ull;
    }

    for (int j = 0; j < ntiles; ++j) {
        ptx::cp_async_wait<1>();
        __syncthreads();                                // Q and K_j are there
        float s[RPT][4];
        {
            uint64_t acc[RPT][4];
#pragma unroll
            for (int r = 0; r < RPT; ++r)
#pragma unroll
                for (int c = 0; c < 4; ++c) acc[r][c] = 0ull;
#pragma unroll kUnrollQ
            for (int d = 0; d < D; d += 4) {
                ulonglong2 k[4];
#pragma unroll
                for (int c = 0; c < 4; ++c) k[c] = *reinterpret_cast<const ulonglong2*>(s_k + (tx + 16 * c) * QS + d);
#pragma unroll
                for (int r = 0; r < RPT; ++r) {
                    const ulonglong2 q = *reinterpret_cast<const ulonglong2*>(s_q + (r * TY + ty) * QS + d);
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        acc[r][c] = ptx::fma2(q.x, k[c].x, acc[r][c]);
                        acc[r][c] = ptx::fma2(q.y, k[c].y, acc[r][c]);
                    }
                }
            }
#pragma unroll
            for (int r = 0; r < RPT; ++r)
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    float lo, hi;
                    ptx::unpack2(acc[r][c], lo, hi);
                    s[r][c] = (lo + hi) * a.scale;
                }
        }
        __syncthreads();                                // everyone is done with K_j
        if (j + 1 < ntiles) fetch_k(j + 1);
        ptx::cp_async_commit();

        const int key0 = t_lo + j * BN + tx;
#pragma unroll
        for (int r = 0; r < RPT; ++r) {
            float mx = -INFINITY;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                if (key0 + 16 * c > bound[r] || key0 + 16 * c >= t_hi) s[r][c] = -INFINITY;
                mx = fmaxf(mx, s[r][c]);
            }
#pragma unroll
            for (int off = 8; off > 0; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
            const float m_new = fmaxf(m[r], mx);
            const float ref = (m_new == -INFINITY) ? 0.f : m_new;      // a row that has seen no key yet: every p is 0
            const float alpha = expf(m[r] - ref);                       // m = -inf: 0
            m[r] = m_new;
            float sum = 0.f;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const float p = expf(s[r][c] - ref);
                sum += p;
                s_p[(r * TY + ty) * PS + tx + 16 * c] = p;
            }
            l[r] = l[r] * alpha + sum;
            const uint64_t alpha2 = ptx::pack2(alpha, alpha);
#pragma unroll
            for (int c = 0; c < 2 * NV; ++c) o[r][c] = ptx::mul2(o[r][c], alpha2);
        }
        ptx::cp_async_wait<1>();
        __syncthreads();                                // V_j is there (a row's P stays within its warp)
        // (Small blocks stop at the tile's last key: 3 tokens on an empty cache 9.5 us, 7.4 so.  For 128 rows the loop's fixed
        // length is worth more: 95.1 us against 98.8 for the 7B shape over 1024 keys.)
        const int k_end = RPT >= 8 ? BN : min(BN, keys - j * BN);
#pragma unroll kUnrollV
        for (int k = 0; k < k_end; k += 4) {
            float4 p[RPT];
#pragma unroll
            for (int r = 0; r < RPT; ++r) p[r] = *reinterpret_cast<const float4*>(s_p + (r * TY + ty) * PS + k);
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) {
                ulonglong2 v[NV];
#pragma unroll
                for (int c = 0; c < NV; ++c) v[c] = *reinterpret_cast<const ulonglong2*>(s_v + (k + kk) * D + c * 64 + tx * 4);
#pragma unroll
                for (int r = 0; r < RPT; ++r) {
                    const float x = kk == 0 ? p[r].x : kk == 1 ? p[r].y : kk == 2 ? p[r].z : p[r].w;
                    const uint64_t x2 = ptx::pack2(x, x);
#pragma unroll
                    for (int c = 0; c < NV; ++c) {
                        o[r][2 * c] = ptx::fma2(x2, v[c].x, o[r][2 * c]);
                        o[r][2 * c + 1] = ptx::fma2(x2, v[c].y, o[r][2 * c + 1]);
                    }
                }
            }
        }
        __syncthreads();                                // everyone is done with V_j
        if (j + 1 < ntiles) fetch_v(j + 1);
        ptx::cp_async_commit();
    }

    // A masked key's probability is 0, but 0 times an infinite or undefined value is not: a row block whose results
    // are not all finite is done again row by row, each over the keys it sees.
    uint64_t zero = 0ull;                               // ... or undefined
#pragma unroll
    for (int r = 0; r < RPT; ++r)
#pragma unroll
        for (int c = 0; c < 2 * NV; ++c) zero = ptx::fma2(o[r][c], 0ull, zero);
    float z0, z1;
    ptx::unpack2(zero, z0, z1);
    if (__syncthreads_and(z0 + z1 == 0.f)) {
#pragma unroll
        for (int r = 0; r < RPT; ++r) {
            float sum = l[r];
#pragma unroll
            for (int off = 8; off > 0; off >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
            const int row = row0 + r * TY + ty;
            if (row >= R) continue;
            const long prow = ((long)split * a.Hkv + g) * R + row;
            const float inv = (sum > 0.f) ? 1.f / sum : 0.f;
#pragma unroll
            for (int c = 0; c < NV; ++c) {
                float4 v;
                ptx::unpack2(o[r][2 * c], v.x, v.y);
                ptx::unpack2(o[r][2 * c + 1], v.z, v.w);
                *reinterpret_cast<float4*>(a.o_part + prow * D + c * 64 + tx * 4) = make_float4(v.x * inv, v.y * inv, v.z * inv, v.w * inv);
            }
            if (tx == 0) a.lse_part[prow] = (sum > 0.f) ? m[r] + logf(sum) : -INFINITY;
        }
    } else {
        for (int row = row0 + (tid >> 5); row <= last_row; row += NT / 32)
        {
            const long prow = ((long)split * a.Hkv + g) * R + row;
            simt_row<T, D>(qb + (long)(row - row0) * D, kb, vb, a.o_part + prow * D, a.lse_part + prow, a.scale, min(keys, a.cache_len + row / a.G + 1 - t_lo));
        }
    }
    // (everyone is done with the tiles in shared memory since the last key tile's final meeting)
    if constexpr (SHARE) {
        if (left > 0) {
            if (tiles.off[rb + 1] == tiles.off[kSimtShareBlocks]) {       // the kv head's last row block
                rb = 0;
                ++g;
            } else {
                ++rb;
            }
            split = j_lo = 0;
            j_hi = min(tiles.off[rb + 1] - tiles.off[rb], left);
            left -= j_hi;
            continue;
        }
    }
    break;
    }
}

}  // namespace evln
