// fp32 step attention of little work: the same three bf16 parts per float as attn_f32.cuh on mma.sync, for
// steps that are a chain of latencies.  A 128-row tcgen05 tile takes about 9 K cycles from its operands to its
// outputs whatever it holds; here 32 rows x 64 keys stay in the registers of 8 warps.
//
// A block: 32 packed query rows of one kv head (two 16-row tiles) and a split of its keys, 64 at a time.  All warps split
// the K and V tiles into their parts (registers to swizzled shared memory, the next tile's loads in flight); then warp
// (w % 2, w / 2) has 16 rows and 16 of the tile's keys to itself: scores, probabilities and a running maximum, sum and
// output of its own.  The large parts' product of every 16 channels and every tile's product with V start from zero and are
// added in registers, the small parts of a score are a sum of their own, so that the tensor core cuts off even less than in attn_f32.cuh.  The four warps of a row are merged in shared memory.
//
// FUSED: evlnStep as one launch.  The splits of a row block are a cluster.  Its blocks rotate the row block's queries (each
// all of them, into q_rot and its own shared memory) and the new keys (a share each, into the cache with the values; blocks of
// other rows write the same numbers), meet, and at the end merge the splits out of each other's shared memory with the
// combine kernel's arithmetic: the bits of the three calls.
#pragma once

#include "attn_f32.cuh"
#include "rope_append.cuh"

namespace evln {

// What the one-launch step adds: the new tokens and where the results go.
struct F32Fused {
    const float* q_new;
    const float* k_new;
    const float* v_new;
    long q_stride, k_stride, v_stride;
    float* out;              // [n, Hq, D]
    float* lse_out;          // [n, Hq] or null
    double log2_theta;
    const double2* table;
    int table_first;
};

constexpr int kSmallThreads = 256, kSmallRows = 32;
constexpr int kSmallCluster = 16;                     // most splits of a one-launch step
constexpr int kSmallAngleTokens = 80;                 // most tokens whose angles a block of a one-launch step holds

template <int D> struct SmallPlan {
    static constexpr int kBlk = 64 * 128, kPart = kBlk * (D / 64);         // one part of a K or V tile, 64-channel blocks
    static constexpr int kQBlk = kSmallRows * 128, kQPart = kQBlk * (D / 64);
    static constexpr int kKOff = 0, kVOff = 3 * kPart, kQOff = 6 * kPart;
    static constexpr int kStride = D + 4;                                  // floats per row of an output
    static constexpr int kStatOff = kQOff + 3 * kQPart;                    // float [2][8][16]: the warps' maxima and sums
    static constexpr int kLseOff = kStatOff + 2 * 8 * 16 * 4;              // float [32]
    static constexpr int kHugeOff = kLseOff + kSmallRows * 4;              // int
    static constexpr int kBytes = kHugeOff + 16 + 1024;
    static constexpr int kAngles = D / 2 + D / 16;                         // places of a token's angles
    static_assert(8 * 16 * kStride * 4 <= 6 * kPart, "the warps' outputs fit the tiles");
    static_assert(kSmallRows * kStride * 4 <= 3 * kQPart, "the rows to merge fit the queries");
    static_assert(kSmallAngleTokens * kAngles * 16 <= 6 * kPart, "the angles fit the tiles");
};

template <int D, bool FUSED>
__global__ void __launch_bounds__(kSmallThreads, 1)
attn_f32_small_kernel(const SimtAttnArgs a, const FastDiv div_g, const __grid_constant__ F32Fused f)
{
    using Plan = SmallPlan<D>;
    constexpr int NT = kSmallThreads, kVecs = 64 * D / 4 / NT, kHalf = D / 2, kT = D / 8;
    extern __shared__ uint8_t small_smem_raw[];
    const uint32_t base = (ptx::smem_u32(small_smem_raw) + 1023u) & ~1023u;
    uint8_t* smem = small_smem_raw + (base - ptx::smem_u32(small_smem_raw));
    float* s_stat = reinterpret_cast<float*>(smem + Plan::kStatOff);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int R = a.num_new * a.G, total = a.cache_len + a.num_new;
    const int split = blockIdx.x, g = blockIdx.z, row0 = blockIdx.y * kSmallRows, rows = min(kSmallRows, R - row0);
    const int all_tiles = (total + 63) / 64;
    const int j_lo = (int)((unsigned)split * (unsigned)all_tiles / (unsigned)a.num_splits);
    const int j_hi = (int)((unsigned)(split + 1) * (unsigned)all_tiles / (unsigned)a.num_splits);
    const int tok0 = (int)fast_div((uint32_t)row0, div_g), tok1 = (int)fast_div((uint32_t)(row0 + rows - 1), div_g);   // the rows' tokens
    const int t_lo = j_lo * 64, keys = min(min(total, j_hi * 64), a.cache_len + tok1 + 1) - t_lo;
    const int ntiles = keys > 0 ? (keys + 63) / 64 : 0;
    const float* kb = (const float*)a.k_cache + ((long)g * a.cache_cap + t_lo) * D;
    const float* vb = (const float*)a.v_cache + ((long)g * a.cache_cap + t_lo) * D;

    ptx::grid_dependency_wait();
    ptx::grid_launch_dependents();

    // a tile of K or V: 4 channels of a key per vector
    constexpr int kRowStep = NT / (D / 4);
    static_assert(kRowStep % 8 == 0, "a thread's keys have the same place in the swizzle");
    const int t_row = tid / (D / 4), t_vec = tid % (D / 4);
    const uint32_t t_place = (t_vec >> 4) * Plan::kBlk + t_row * 128 + ((((t_vec & 15) >> 1) ^ (t_row & 7)) << 4) + (t_vec & 1) * 8;
    ulonglong2 kx[kVecs], vx[kVecs];
    auto zero_tile = [&](ulonglong2 (&x)[kVecs]) {
#pragma unroll
        for (int i = 0; i < kVecs; ++i) x[i] = make_ulonglong2(0ull, 0ull);
    };
    auto load_rows = [&](ulonglong2 (&x)[kVecs], const float* from, int lo, int hi) {     // rows lo .. hi-1 of the tile
#pragma unroll
        for (int i = 0; i < kVecs; ++i) {
            const int r = t_row + i * kRowStep;
            if (r >= lo && r < hi) x[i] = *reinterpret_cast<const ulonglong2*>(from + tid * 4 + i * (NT * 4));
        }
    };
    int* s_huge = reinterpret_cast<int*>(smem + Plan::kHugeOff);
    if (tid == 0) *s_huge = 0;
    uint32_t top = 0;                                        // largest query and key parts
    auto store_tile = [&](const ulonglong2 (&x)[kVecs], uint8_t* to, bool is_k) {
#pragma unroll
        for (int i = 0; i < kVecs; ++i) {
            uint2 p[3];
            split3(x[i].x, p[0].x, p[1].x, p[2].x);
            split3(x[i].y, p[0].y, p[1].y, p[2].y);
            if (is_k) top = ptx::max_abs_bf16x2(ptx::max_abs_bf16x2(top, p[0].x), p[0].y);
#pragma unroll
            for (int y = 0; y < 3; ++y) *reinterpret_cast<uint2*>(to + t_place + i * (kRowStep * 128) + y * Plan::kPart) = p[y];
        }
    };
    // 4 channels at 4 c of query row r, three parts
    auto store_q = [&](int r, int c, const ulonglong2& x) {
        uint2 p[3];
        split3(x.x, p[0].x, p[1].x, p[2].x);
        split3(x.y, p[0].y, p[1].y, p[2].y);
        top = ptx::max_abs_bf16x2(ptx::max_abs_bf16x2(top, p[0].x), p[0].y);
        uint8_t* at = smem + Plan::kQOff + (c >> 4) * Plan::kQBlk + r * 128 + ((((c & 15) >> 1) ^ (r & 7)) << 4) + (c & 1) * 8;
#pragma unroll
        for (int y = 0; y < 3; ++y) *reinterpret_cast<uint2*>(at + y * Plan::kQPart) = p[y];
    };

    zero_tile(kx);
    zero_tile(vx);
    const int cached = FUSED ? a.cache_len - t_lo : keys;    // rows of the split's keys that are there before this launch
    load_rows(kx, kb, 0, min(keys, cached));
    load_rows(vx, vb, 0, min(keys, cached));
    if constexpr (FUSED) {
        constexpr int kPairs = kHalf / 4;
        // the new tokens that the row block sees, this block's share of them; angles of those and of its queries' tokens
        // (one run of tokens where the two meet)
        const int seen = tok1 + 1;
        const int k_first = (int)((unsigned)split * (unsigned)seen / (unsigned)a.num_splits);
        const int k_end = (int)((unsigned)(split + 1) * (unsigned)seen / (unsigned)a.num_splits), nk = k_end - k_first;
        const bool meet = nk == 0 || k_end >= tok0;
        const int first = meet && nk > 0 ? min(tok0, k_first) : tok0;            // (a share ends at tok1 at most)
        const int run = seen - first, count = run + (meet ? 0 : nk);             // tokens first .. tok1, then the share
        double2* angles = reinterpret_cast<double2*>(smem);
        // a work item: 4 + 4 channels of a query (in both halves of the head), of a new key, or 4 of a new value
        const int q_items = rows * kPairs, k_items = nk * kPairs, items = q_items + k_items + nk * (D / 4);
        auto load_item = [&](int it, uint4& lo, uint4& hi) {
            if (it < q_items + k_items) {
                const int e = it < q_items ? it : it - q_items, r = e / kPairs, k = e % kPairs;
                const int tok = it < q_items ? (int)fast_div((uint32_t)(row0 + r), div_g) : k_first + r;
                const float* src = it < q_items ? f.q_new + tok * f.q_stride + (long)(g * a.G + row0 + r - tok * a.G) * D : f.k_new + tok * f.k_stride + (long)g * D;
                lo = *reinterpret_cast<const uint4*>(src + 4 * k);
                hi = *reinterpret_cast<const uint4*>(src + kHalf + 4 * k);
            } else {
                const int e = it - q_items - k_items;
                lo = *reinterpret_cast<const uint4*>(f.v_new + (k_first + e / (D / 4)) * f.v_stride + (long)g * D + e % (D / 4) * 4);
            }
        };
        auto finish_item = [&](int it, const uint4& lo, const uint4& hi) {
            if (it < q_items + k_items) {
                const bool is_q = it < q_items;
                const int e = is_q ? it : it - q_items, r = e / kPairs, k = e % kPairs;
                const int tok = is_q ? (int)fast_div((uint32_t)(row0 + r), div_g) : k_first + r;
                uint4 out_lo, out_hi;
                Rotation<float>::turn(angles + (is_q || meet ? tok - first : run + r) * Plan::kAngles, k, lo, hi, out_lo, out_hi);
                float* dst = is_q ? (float*)a.q_rot + ((long)g * R + row0 + r) * D : (float*)a.k_cache + ((long)g * a.cache_cap + a.cache_len + tok) * D;
                if (!is_q || split == 0) {
                    *reinterpret_cast<uint4*>(dst + 4 * k) = out_lo;
                    *reinterpret_cast<uint4*>(dst + kHalf + 4 * k) = out_hi;
                }
                if (is_q) {
                    store_q(r, k, *reinterpret_cast<const ulonglong2*>(&out_lo));
                    store_q(r, k + kPairs, *reinterpret_cast<const ulonglong2*>(&out_hi));
                }
            } else {
                const int e = it - q_items - k_items;
                *reinterpret_cast<uint4*>((float*)a.v_cache + ((long)g * a.cache_cap + a.cache_len + k_first + e / (D / 4)) * D + e % (D / 4) * 4) = lo;
            }
        };
        // the first items are on their way while the angles are formed, four at a time (a sine is one long chain)
        constexpr int kAhead = 3;
        uint4 lo[kAhead], hi[kAhead];
#pragma unroll
        for (int u = 0; u < kAhead; ++u)
            if (tid + u * NT < items) load_item(tid + u * NT, lo[u], hi[u]);
        {
            constexpr int kStep = NT / kHalf;
            const int j = tid & (kHalf - 1);
            const double omega = f.table ? 0.0 : rope_omega(j, D, f.log2_theta);
            for (int i0 = tid / kHalf; i0 < count; i0 += 4 * kStep) {
                double2 cs[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int i = min(i0 + u * kStep, count - 1);
                    const long pos = (long)a.cache_len + (i < run ? first + i : k_first + i - run);
                    cs[u] = f.table ? f.table[(pos - f.table_first) * kHalf + j] : rope_cos_sin_at(pos, omega);
                }
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (i0 + u * kStep < count) Rotation<float>::put(angles + (i0 + u * kStep) * Plan::kAngles, j, cs[u]);
            }
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < kAhead; ++u)
            if (tid + u * NT < items) finish_item(tid + u * NT, lo[u], hi[u]);
        for (int it = tid + kAhead * NT; it < items; it += NT) {
            load_item(it, lo[0], hi[0]);
            finish_item(it, lo[0], hi[0]);
        }
        for (int it = q_items * 2 + tid; it < kSmallRows * (D / 4); it += NT) store_q(it / (D / 4), it % (D / 4), make_ulonglong2(0ull, 0ull));
        // the new keys and values are in the cache when all blocks of the cluster are here
        __syncwarp();
        ptx::cluster_arrive();
        ptx::cluster_wait();
        load_rows(kx, kb, max(0, cached), keys);
        load_rows(vx, vb, max(0, cached), keys);
    } else {
        for (int it = tid; it < kSmallRows * (D / 4); it += NT) {
            const int r = it / (D / 4), c = it % (D / 4);
            ulonglong2 x = make_ulonglong2(0ull, 0ull);
            if (r < rows) x = *reinterpret_cast<const ulonglong2*>((const float*)a.q_rot + ((long)g * R + row0 + r) * D + 4 * c);
            store_q(r, c, x);
        }
    }

    const int rt = warp & 1, kg = warp >> 1;                 // row tile and 16 keys of the tile
    const int mi = lane >> 3, mr = lane & 7;                 // ldmatrix: matrix, row of it
    const int q_row = rt * 16 + (mi & 1) * 8 + mr, q_chunk = mi >> 1;
    const int k_row = kg * 16 + (mi >> 1) * 8 + mr, k_chunk = mi & 1;
    const int v_row = kg * 16 + (mi & 1) * 8 + mr, v_chunk = mi >> 1;
    float o[kT][4];                                          // 16 rows x D channels: 8-channel tiles
    float m[2] = {-INFINITY, -INFINITY}, l[2] = {0.f, 0.f};  // of rows lane / 4 and + 8; unscaled maximum
    int bound[2];                                            // last visible key of the split
#pragma unroll
    for (int h = 0; h < 2; ++h) bound[h] = a.cache_len + (int)fast_div((uint32_t)(row0 + rt * 16 + h * 8 + (lane >> 2)), div_g) - t_lo;
#pragma unroll
    for (int t = 0; t < kT; ++t)
#pragma unroll
        for (int e = 0; e < 4; ++e) o[t][e] = 0.f;
    auto swz_at = [](int row, int chunk, int blk) -> uint32_t {          // 16-byte chunk of a row, 64-channel blocks
        return (uint32_t)((chunk >> 3) * blk + row * 128 + (((chunk & 7) ^ (row & 7)) << 4));
    };

    for (int j = 0; j < ntiles; ++j) {
        __syncthreads();                                     // everyone is done with tile j - 1 (and the angles)
        store_tile(kx, smem + Plan::kKOff, true);
        store_tile(vx, smem + Plan::kVOff, false);
        __syncthreads();
        if (j + 1 < ntiles) {
            zero_tile(kx);
            zero_tile(vx);
            load_rows(kx, kb + (long)(j + 1) * 64 * D, 0, keys - (j + 1) * 64);
            load_rows(vx, vb + (long)(j + 1) * 64 * D, 0, keys - (j + 1) * 64);
        }
        const int key0 = j * 64 + kg * 16;
        if (rt * 16 >= rows || key0 >= keys) continue;
        float big[2][4], small[2][4];                        // [8 keys]
#pragma unroll
        for (int t = 0; t < 2; ++t)
#pragma unroll
            for (int e = 0; e < 4; ++e) big[t][e] = small[t][e] = 0.f;
#pragma unroll
        for (int ks = 0; ks < D / 16; ++ks) {
            uint32_t q[3][4], k[3][4];
#pragma unroll
            for (int y = 0; y < 3; ++y) {
                ptx::ldmatrix_x4(q[y], base + Plan::kQOff + y * Plan::kQPart + swz_at(q_row, 2 * ks + q_chunk, Plan::kQBlk));
                ptx::ldmatrix_x4(k[y], base + Plan::kKOff + y * Plan::kPart + swz_at(k_row, 2 * ks + k_chunk, Plan::kBlk));
            }
#pragma unroll
            for (int t = 0; t < 2; ++t) {
                ptx::mma_bf16(small[t], q[2], k[0][2 * t], k[0][2 * t + 1]);
                ptx::mma_bf16(small[t], q[0], k[2][2 * t], k[2][2 * t + 1]);
                ptx::mma_bf16(small[t], q[1], k[1][2 * t], k[1][2 * t + 1]);
                ptx::mma_bf16(small[t], q[1], k[0][2 * t], k[0][2 * t + 1]);
                ptx::mma_bf16(small[t], q[0], k[1][2 * t], k[1][2 * t + 1]);
                float u[4] = {0.f, 0.f, 0.f, 0.f};
                ptx::mma_bf16(u, q[0], k[0][2 * t], k[0][2 * t + 1]);
#pragma unroll
                for (int e = 0; e < 4; ++e) big[t][e] += u[e];
            }
        }
        float x[2][4];
#pragma unroll
        for (int t = 0; t < 2; ++t)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                x[t][e] = big[t][e] + small[t][e];
                if (key0 + t * 8 + (lane & 3) * 2 + (e & 1) > bound[e >> 1]) x[t][e] = -INFINITY;
            }
        uint32_t p[3][4];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float mx = fmaxf(fmaxf(x[0][2 * h], x[0][2 * h + 1]), fmaxf(x[1][2 * h], x[1][2 * h + 1]));
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
            const float m_new = fmaxf(m[h], mx), ref = (m_new == -INFINITY) ? 0.f : m_new;
            const float alpha = f32_rescale(a, m[h] - ref);
            m[h] = m_new;
            float sum = 0.f;
#pragma unroll
            for (int t = 0; t < 2; ++t) {
                const uint64_t w = f32_weights(a, ptx::pack2(x[t][2 * h] - ref, x[t][2 * h + 1] - ref));
                float w0, w1;
                ptx::unpack2(w, w0, w1);
                sum += w0 + w1;
                split3(w, p[0][2 * t + h], p[1][2 * t + h], p[2][2 * t + h]);
            }
            l[h] = fmaf(l[h], alpha, sum);
#pragma unroll
            for (int t = 0; t < kT; ++t) {
                o[t][2 * h] *= alpha;
                o[t][2 * h + 1] *= alpha;
            }
        }
#pragma unroll
        for (int c = 0; c < D / 16; ++c) {
            uint32_t v[3][4];
#pragma unroll
            for (int y = 0; y < 3; ++y) ptx::ldmatrix_x4_trans(v[y], base + Plan::kVOff + y * Plan::kPart + swz_at(v_row, 2 * c + v_chunk, Plan::kBlk));
#pragma unroll
            for (int t = 0; t < 2; ++t) {
                float u[4] = {0.f, 0.f, 0.f, 0.f};
                ptx::mma_bf16(u, p[2], v[0][2 * t], v[0][2 * t + 1]);
                ptx::mma_bf16(u, p[0], v[2][2 * t], v[2][2 * t + 1]);
                ptx::mma_bf16(u, p[1], v[1][2 * t], v[1][2 * t + 1]);
                ptx::mma_bf16(u, p[1], v[0][2 * t], v[0][2 * t + 1]);
                ptx::mma_bf16(u, p[0], v[1][2 * t], v[1][2 * t + 1]);
                ptx::mma_bf16(u, p[0], v[0][2 * t], v[0][2 * t + 1]);
#pragma unroll
                for (int e = 0; e < 4; ++e) o[2 * c + t][e] += u[e];
            }
        }
    }

    // ---- the four warps of a row into shared memory, where the tiles were ----
    __syncthreads();
    if (f32_huge(a, top)) *s_huge = 1;
    {
        float* s_o = reinterpret_cast<float*>(smem) + warp * 16 * Plan::kStride;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int r = h * 8 + (lane >> 2);
#pragma unroll
            for (int t = 0; t < kT; ++t)
                *reinterpret_cast<float2*>(s_o + r * Plan::kStride + t * 8 + (lane & 3) * 2) = make_float2(o[t][2 * h], o[t][2 * h + 1]);
            float sum = l[h];
            sum += __shfl_xor_sync(0xffffffffu, sum, 1);
            sum += __shfl_xor_sync(0xffffffffu, sum, 2);
            if ((lane & 3) == 0) {
                s_stat[warp * 16 + r] = m[h];
                s_stat[128 + warp * 16 + r] = sum;
            }
        }
    }
    __syncthreads();
    // Eight threads a row, all rows at once: vectors c, c + 8, .. of 4 channels.  (A warp a row, four rows in turn: 0.9 us more.)
    float* s_rows = reinterpret_cast<float*>(smem + Plan::kQOff);
    float* s_lse = reinterpret_cast<float*>(smem + Plan::kLseOff);
    {
        constexpr int kV = D / 32;
        const int r = tid >> 3, c = tid & 7, w0 = r >> 4, rr = r & 15;
        float w[4], M = -INFINITY;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            w[i] = s_stat[(w0 + 2 * i) * 16 + rr];
            M = fmaxf(M, w[i]);
        }
        const float ref = (M == -INFINITY) ? 0.f : M;
        float sum = 0.f;
        float4 y[kV];
#pragma unroll
        for (int v = 0; v < kV; ++v) y[v] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            w[i] = f32_rescale(a, w[i] - ref);
            sum = fmaf(w[i], s_stat[128 + (w0 + 2 * i) * 16 + rr], sum);
            const float4* at = reinterpret_cast<const float4*>(reinterpret_cast<const float*>(smem) + ((w0 + 2 * i) * 16 + rr) * Plan::kStride);
#pragma unroll
            for (int v = 0; v < kV; ++v) {
                const float4 x = at[c + 8 * v];
                y[v].x = fmaf(w[i], x.x, y[v].x);
                y[v].y = fmaf(w[i], x.y, y[v].y);
                y[v].z = fmaf(w[i], x.z, y[v].z);
                y[v].w = fmaf(w[i], x.w, y[v].w);
            }
        }
        // (done again in floats: see attn_f32.cuh)
        bool odd = *s_huge != 0, low = false;
#pragma unroll
        for (int v = 0; v < kV; ++v) {
            odd |= !(fabsf(y[v].x) + fabsf(y[v].y) + fabsf(y[v].z) + fabsf(y[v].w) <= 3.0e38f);
            low |= f32_small(y[v].x) || f32_small(y[v].y) || f32_small(y[v].z) || f32_small(y[v].w);
        }
        uint32_t bad = __ballot_sync(0xffffffffu, odd && r < rows);
        const uint32_t lows = __ballot_sync(0xffffffffu, low && r < rows);
        if (lows & ~bad) {
            bool inexact = false;
            for (int i = lane; i < keys * (D / 4); i += 32) inexact |= f32_inexact(reinterpret_cast<const float4*>(vb)[i]);
            if (__any_sync(0xffffffffu, inexact)) bad |= lows;
        }
        const long prow0 = ((long)split * a.Hkv + g) * R + row0;
        if (r < rows) {
            const float inv = (sum > 0.f) ? 1.f / sum : 0.f;
            float4* op = reinterpret_cast<float4*>(FUSED ? s_rows + r * Plan::kStride : a.o_part + (prow0 + r) * D);
#pragma unroll
            for (int v = 0; v < kV; ++v) op[c + 8 * v] = make_float4(y[v].x * inv, y[v].y * inv, y[v].z * inv, y[v].w * inv);
            if (c == 0) *(FUSED ? s_lse + r : a.lse_part + prow0 + r) = f32_lse(a, M, sum);
        }
        __syncwarp();
        while (bad) {                                        // the warp's rows that are not: a row by the whole warp
            const int first = (__ffs(bad) - 1) & ~7, br = (tid & ~31) / 8 + first / 8;
            bad &= ~(0xffu << first);
            // (FUSED: the block of split 0 has written q_rot ahead of the cluster's meeting)
            simt_row<float, D>((const float*)a.q_rot + ((long)g * R + row0 + br) * D, kb, vb, FUSED ? s_rows + br * Plan::kStride : a.o_part + (prow0 + br) * D,
                               FUSED ? s_lse + br : a.lse_part + prow0 + br, a.scale,
                               min(keys, a.cache_len + (int)fast_div((uint32_t)(row0 + br), div_g) + 1 - t_lo));
        }
    }

    if constexpr (FUSED) {
        // every block merges an equal share of the rows, sixteen threads a row: the combine kernel's arithmetic, partials
        // from the cluster's shared memory
        constexpr int kV = D / 64;
        const int S = a.num_splits, sub = tid & 15;
        __syncwarp();
        ptx::cluster_arrive();
        ptx::cluster_wait();
        for (int r0 = split; r0 < rows; r0 += S * (NT / 16)) {
            const int r = r0 + S * (tid >> 4);
            const bool mine = r < rows;
            const uint32_t lse_at = base + Plan::kLseOff + r * 4, row_at = base + Plan::kQOff + r * Plan::kStride * 4 + sub * 16;
            const float my_lse = mine && sub < S ? ptx::ld_cluster_f32(ptx::map_to_cta(lse_at, sub)) : -INFINITY;
            float4 x[kSmallCluster / 2][kV], y[kV];
#pragma unroll
            for (int v = 0; v < kV; ++v) y[v] = make_float4(0.f, 0.f, 0.f, 0.f);
            auto fetch = [&](int i0) {
#pragma unroll
                for (int i = 0; i < kSmallCluster / 2; ++i)
#pragma unroll
                    for (int v = 0; v < kV; ++v) {
                        x[i][v] = make_float4(0.f, 0.f, 0.f, 0.f);
                        if (mine && i0 + i < S) x[i][v] = ptx::ld_cluster_f32x4(ptx::map_to_cta(row_at + v * 256, i0 + i));
                    }
            };
            fetch(0);
            float M = my_lse;
#pragma unroll
            for (int off = 8; off > 0; off >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, off));
            const float w = (my_lse == -INFINITY) ? 0.f : expf(my_lse - M);
            float wsum = w;
#pragma unroll
            for (int off = 8; off > 0; off >>= 1) wsum += __shfl_xor_sync(0xffffffffu, wsum, off);
            auto add = [&](int i0) {
#pragma unroll
                for (int i = 0; i < kSmallCluster / 2; ++i) {
                    const float wi = __shfl_sync(0xffffffffu, w, i0 + i, 16);
                    if (i0 + i >= 4 && wi == 0.f) continue;
#pragma unroll
                    for (int v = 0; v < kV; ++v) {
                        y[v].x = fmaf(wi, x[i][v].x, y[v].x);
                        y[v].y = fmaf(wi, x[i][v].y, y[v].y);
                        y[v].z = fmaf(wi, x[i][v].z, y[v].z);
                        y[v].w = fmaf(wi, x[i][v].w, y[v].w);
                    }
                }
            };
            add(0);
            if (S > kSmallCluster / 2) {
                fetch(kSmallCluster / 2);
                add(kSmallCluster / 2);
            }
            if (mine) {
                const float inv = (wsum > 0.f) ? 1.f / wsum : 0.f;
                const int row = row0 + r, tok = (int)fast_div((uint32_t)row, div_g);
                const long at = (long)tok * a.Hkv * a.G + g * a.G + (row - tok * a.G);
                float4* dst = reinterpret_cast<float4*>(f.out + at * D) + sub;
#pragma unroll
                for (int v = 0; v < kV; ++v) dst[v * 16] = make_float4(y[v].x * inv, y[v].y * inv, y[v].z * inv, y[v].w * inv);
                if (f.lse_out && sub == 0) f.lse_out[at] = (wsum > 0.f) ? M + logf(wsum) : -INFINITY;
            }
        }
        __syncwarp();
        ptx::cluster_arrive_relaxed();                       // nobody leaves while others read its rows
        ptx::cluster_wait();
    }
}

}  // namespace evln
