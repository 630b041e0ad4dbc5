// fp32 step attention on the 5th-generation tensor cores.
//
// A float is exactly the sum of three bf16 numbers (8 + 8 + 8 bits and the signs of the rests; down to 2^-109), so a product of
// floats is nine products of bf16 numbers, which the tensor core forms exactly and adds in fp32.  Six of them are
// taken (the other three are below 2^-26 of the product), the small ones first, so that the accumulator's own
// rounding (towards zero, at its size of the moment) sees the large ones only.  An accumulator never runs on
// across key tiles: every tile's products with V start from zero, and so do its scores, in two sums over half of the channels each; the
// results are added in registers, rounded to nearest.  (A score of 128 normal channels against fp64: in one sum 1.3e-7 off, of which
// 1.0e-7 is what the tensor core cuts off, always towards zero; in two sums 8.6e-8 and 6e-8; a chain of float FMAs 1.5e-7, either way.)
//
// Bound: the tensor pipe (6 x 4 D bf16 flop per visible pair), with all SMs at work the latency of K and V out of L2.  A block of 16 + 1 warps owns 128 packed query rows of
// one kv head and walks its key tiles, 64 keys at a time:
//   16 warps, four per TMEM lane quarter: a thread has a row, 16 of the tile's 64 score columns and a
//            quarter of the channels.  Per tile they split the next K tile into its three parts (from
//            registers into swizzled shared memory), take the scores, exchange the row maximum (four threads a
//            row), split the V tile, add the previous tile's product to the accumulator in registers, and leave the
//            probabilities' three parts in tensor memory (at head_dim 128 the third in shared memory).
//   1 warp   issues: S_j = Q K_j^T (A = Q's parts in tensor memory) and O_j = P_j V_j (A = P_j's parts), in the order
//            S_0, S_1, O_0, S_2, O_1, ..: the scores of a tile run while the softmax of the one before does.
// Tensor memory columns: Q's parts 0 .. 3 D/2, O_j (D), S_j (two sums of 64: even and odd 16 channels), P_j's first two parts (64); all 512 at
// head_dim 128, where P_j's third part is in shared memory.
//
// SHARE: as in attn_simt.cuh, one block per SM with an equal share of all (row block, key tile) pairs.
//
// Measured: a tile 2.2 us at head_dim 128 (the products alone 1.9; about 3 with a block on every SM), 1.5 at 64; 196 tokens of the 7B shape over 1024 keys 95.3 us a step
// in float FMAs, 33.2 so (32.0 with the scores in one sum); 256 tokens over 2048 206 and 62; 252 tokens of 16 heads over 2031 123 and 37.9.
#pragma once

#include "attn_pair.cuh"
#include "attn_simt.cuh"

namespace evln {

constexpr int kF32Compute = 512, kF32Threads = kF32Compute + 32;
constexpr int kF32Keys = kSimtKeys;
static_assert(kF32Keys == 64, "a key tile is one 64-key block of 128-byte rows");

template <int D> struct F32Plan {
    static constexpr int kBlk = kF32Keys * 128;              // 64 keys x 64 channels of one part, 128-byte swizzle
    static constexpr int kPart = kBlk * (D / 64);            // one part of a K or V tile
    static constexpr int kTile = 3 * kPart;
    static constexpr int kKOff = 0, kVOff = 2 * kTile;       // two tiles each
    static constexpr int kPLoOff = kVOff + 2 * kTile;        // the probabilities' third part, 128 rows x 64 keys, 128-byte swizzle
    static constexpr int kBarOff = kPLoOff + (D == 128 ? kTileM * 128 : 0);   // barriers, TMEM address, flags
    static constexpr int kMaxOff = kBarOff + 128;            // float [2][4][128]: row maxima, tiles in turn
    static constexpr int kSumOff = kMaxOff + 2 * 4 * 128 * 4;    // float [4][128]: row sums
    static constexpr int kBytes = kSumOff + 4 * 128 * 4 + 1024;
    static constexpr uint32_t kColO = 3 * D / 2, kColS = kColO + D, kColP = kColS + 2 * kF32Keys;
    static constexpr int kOutStride = D + 16;                // bytes per row of a warp's D / 4 channels when they are written out
    static constexpr bool kPLoTmem = kColP + 3 * kF32Keys / 2 <= 512;          // P_j's third part beside the others (one in shared memory: 1.5 % of a step more)
    static_assert(kPLoTmem == (D == 64), "room for the third part");
    static_assert(kColP + kF32Keys <= 512, "tensor memory");
    static_assert(kBytes <= 227 * 1024, "shared memory per CTA");
    static_assert(16 * 32 * kOutStride <= 2 * kTile, "the rows are written out through the K tiles");
};

// x = hi + mid + lo, two numbers at a time (each rest is exact)
__device__ __forceinline__ void split3(uint64_t x, uint32_t& hi, uint32_t& mid, uint32_t& lo)
{
    const uint64_t minus = ptx::pack2(-1.f, -1.f);
    float x0, x1;
    ptx::unpack2(x, x0, x1);
    hi = ptx::pack_bf16x2(x0, x1);
    x = ptx::fma2(ptx::pack2(__uint_as_float(hi << 16), __uint_as_float(hi & 0xffff0000u)), minus, x);
    ptx::unpack2(x, x0, x1);
    mid = ptx::pack_bf16x2(x0, x1);
    x = ptx::fma2(ptx::pack2(__uint_as_float(mid << 16), __uint_as_float(mid & 0xffff0000u)), minus, x);
    ptx::unpack2(x, x0, x1);
    lo = ptx::pack_bf16x2(x0, x1);
}

// The parts are exact down to 2^-109 and no further off than 2^-134 below.  What that leaves out of a score is nothing (2^-30) unless the
// number's partner is huge, so row blocks that meet a query or key of 2^90 (divided by a softmax scale above 1) are done in floats.
__device__ __forceinline__ bool f32_huge(const SimtAttnArgs& a, uint32_t top)        // top: max_abs_bf16x2 of first parts
{
    return (top & 0x7fffu) >= a.huge || ((top >> 16) & 0x7fffu) >= a.huge;
}

// A row's weights are kept 2^64 times as large: the third part of one down to 2^-149 is then no smaller than bf16 holds.
constexpr float kWeightUnit = 18446744073709551616.f, kPerWeightUnit = 1.f / kWeightUnit;
// A value's parts are 2^-134 off at most, and with weights of 2^64 each a row's sum over 2^24 keys 2^-46: bits of sums below 2^-18 may be
// lost, if the row's values are of the kind whose third part is not exact.
constexpr float kSmallSum = 3.814697265625e-6f;
__device__ __forceinline__ bool f32_small(float sum) { return sum != 0.f && fabsf(sum) < kSmallSum; }
__device__ __forceinline__ bool f32_inexact(const float4& v)                         // any of them not 0 and below 2^-109
{
    auto tiny = [](float x) { return __float_as_uint(x) * 2u - 1u < 2u * 0x09000000u - 1u; };
    return tiny(v.x) || tiny(v.y) || tiny(v.z) || tiny(v.w);
}
constexpr float kLeastWeight = -191.f;                       // exponent from which on a weight is 0

// Weights of two score differences d <= 0: 2^(64 + d * scale2).  The exponent's integer n is split off before the scale's rest joins, so that
// ex2 sees a fraction in [-0.5, 0.5] with the accuracy of the difference and not that of n.  The largest score's weight is exact.  Undefined
// differences stay undefined.  (Nothing here or in the scale is fitted to inputs.  Against fp64, geometric means over 62 shapes of 64 to 2048
// keys: outputs 2.2e-7 off, 3.2e-7 with float FMAs and expf; log-sum-exps 2.8e-8 both.)
__device__ __forceinline__ uint64_t f32_weights(const SimtAttnArgs& a, uint64_t d2)
{
    const uint64_t hi = ptx::pack2(a.scale2_hi, a.scale2_hi), magic = ptx::pack2(12582912.f, 12582912.f);
    float d0, d1, t0, t1, f0, f1;
    ptx::unpack2(d2, d0, d1);
    d2 = ptx::pack2(ptx::max_nan(d0, a.diff_min), ptx::max_nan(d1, a.diff_min));
    const uint64_t t = ptx::fma2(d2, hi, magic);             // n in its low bits
    const uint64_t minus_n = ptx::fma2(t, ptx::pack2(-1.f, -1.f), magic);
    ptx::unpack2(ptx::fma2(d2, ptx::pack2(a.scale2_lo, a.scale2_lo), ptx::fma2(d2, hi, minus_n)), f0, f1);
    ptx::unpack2(t, t0, t1);
    constexpr uint32_t kBias = (127u + 64u) << 23;           // 2^(64 + n); the field is 0, and so is the weight, from n = kLeastWeight on
    return ptx::mul2(ptx::pack2(ptx::ex2(f0), ptx::ex2(f1)),
                     ptx::pack2(__uint_as_float((__float_as_uint(t0) << 23) + kBias), __uint_as_float((__float_as_uint(t1) << 23) + kBias)));
}
// ... what a running sum is multiplied by when its maximum moves up by -d, in fewer steps: the error of a larger exponent goes with a
// smaller factor.  Factors below the least normal number are kept (ex2 alone would make them 0).
__device__ __forceinline__ float f32_rescale(const SimtAttnArgs& a, float d)
{
    d = fmaxf(d, a.diff_min);
    const float x = fmaf(d, a.scale2_hi, d * a.scale2_lo);
    return x < -64.f ? ptx::ex2(x + 64.f) * kPerWeightUnit : ptx::ex2(x);
}

// Log-sum-exp of a row: unscaled maximum and sum of weights.  The sum of the two parts is rounded once.
__device__ __forceinline__ float f32_lse(const SimtAttnArgs& a, float m, float weights)
{
    const float sum = weights * kPerWeightUnit;
    if (!(sum > 0.f)) return -INFINITY;
    const float top = m * a.scale, rest = fmaf(m, a.scale_lo, fmaf(m, a.scale, -top)), lg = logf(sum);
    const float s = top + lg, b = s - top;
    return s + (((top - (s - b)) + (lg - b)) + rest);
}

template <int D, typename TilesT>
__global__ void __launch_bounds__(kF32Threads, 1)
attn_f32_kernel(const SimtAttnArgs a, const __grid_constant__ TilesT tiles)
{
    constexpr bool SHARE = std::is_same<TilesT, SimtTiles>::value;
    using Plan = F32Plan<D>;
    constexpr int BM = kTileM, BN = kF32Keys;
    constexpr int kVecs = BN * D / 4 / kF32Compute;          // float4 of a K or V tile per thread
    constexpr int kCh = D / 4;                               // channels of O per thread
    extern __shared__ uint8_t f32_smem_raw[];
    const uint32_t smem_base = (ptx::smem_u32(f32_smem_raw) + 1023u) & ~1023u;
    uint8_t* smem = f32_smem_raw + (smem_base - ptx::smem_u32(f32_smem_raw));

    const uint32_t bar_s_ready = smem_base + Plan::kBarOff;  // K_j in shared memory, S_{j-1} read (a warp each)
    const uint32_t bar_p_ready = bar_s_ready + 8;            // P_j in tensor memory, V_j in shared memory, O_{j-1} read
    const uint32_t bar_s_done = bar_p_ready + 8;             // S_j there
    const uint32_t bar_o_done = bar_s_done + 8;              // O_j there
    uint32_t* s_tmem = reinterpret_cast<uint32_t*>(smem + Plan::kBarOff + 32);
    volatile int* s_abort = reinterpret_cast<volatile int*>(smem + Plan::kBarOff + 36);
    int* s_bad = reinterpret_cast<int*>(smem + Plan::kBarOff + 40);      // [2], row blocks in turn: 1 done again, 2 small sums
    int* s_inexact = s_bad + 2;                                          // [2]
    float* s_max = reinterpret_cast<float*>(smem + Plan::kMaxOff);
    float* s_sum = reinterpret_cast<float*>(smem + Plan::kSumOff);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int R = a.num_new * a.G;
    const int total = a.cache_len + a.num_new;
    int rb, g, split, j_lo, j_hi;                            // the row block and its key tiles
    int left = 0;                                            // tiles of the block's share behind them
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
        split = blockIdx.x - (first - j_lo) / a.share;       // shares that the row block met before
    } else {
        rb = blockIdx.x;
        g = blockIdx.y;
        split = blockIdx.z;
        const int all_tiles = (total + BN - 1) / BN;
        j_lo = (int)((long)split * all_tiles / a.num_splits);
        j_hi = (int)((long)(split + 1) * all_tiles / a.num_splits);
    }
    // the next row block of the share, if there is one
    auto next_block = [&]() -> bool {
        if constexpr (SHARE) {
            if (left <= 0) return false;
            if (tiles.off[rb + 1] == tiles.off[kSimtShareBlocks]) {
                rb = 0;
                ++g;
            } else {
                ++rb;
            }
            split = j_lo = 0;
            j_hi = min(tiles.off[rb + 1] - tiles.off[rb], left);
            left -= j_hi;
            return true;
        }
        return false;
    };
    // keys past the row block's last token are visible to none of its rows
    auto keys_of = [&]() -> int {
        const int last_row = min(rb * BM + BM, R) - 1;
        return min(min(total, j_hi * BN), a.cache_len + last_row / a.G + 1) - j_lo * BN;
    };

    if (tid == 0) {
        ptx::mbar_init(bar_s_ready, kF32Compute / 32);
        ptx::mbar_init(bar_p_ready, kF32Compute / 32);
        ptx::mbar_init(bar_s_done, 1);
        ptx::mbar_init(bar_o_done, 1);
        ptx::fence_barrier_init();
        *s_abort = 0;
        s_bad[0] = s_bad[1] = s_inexact[0] = s_inexact[1] = 0;
    }
    if (warp == kF32Compute / 32) {
        ptx::tmem_alloc(ptx::smem_u32(s_tmem), 512);
        ptx::tmem_relinquish();
    }
    ptx::fence_before_sync();
    __syncthreads();
    ptx::fence_after_sync();
    const uint32_t tmem = *(volatile uint32_t*)s_tmem;
    ptx::grid_dependency_wait();                             // programmatic dependent launch: inputs ready
    ptx::grid_launch_dependents();

    // A wait that runs out raises the abort flag and leaves a code in the status word: nobody waits any more then,
    // and everybody goes through the motions to the end.
    int base = 0;                                            // tiles of the row blocks before this one
    if (warp == kF32Compute / 32) {
        // ================= issuer =================
        constexpr int kPa[6] = {2, 0, 1, 1, 0, 0}, kPb[6] = {0, 2, 1, 0, 1, 0};
        const uint32_t idesc_s = make_idesc(false, BM, BN), idesc_o = make_idesc(true, BM, D);
        const uint64_t kdesc0 = make_sdesc(smem_base + Plan::kKOff, 16, 1024);
        const uint64_t vdesc0 = make_sdesc(smem_base + Plan::kVOff, Plan::kBlk, 1024);
        const uint64_t pdesc = make_sdesc(smem_base + Plan::kPLoOff, 16, 1024);
        do {
            const int keys = keys_of(), ntiles = keys > 0 ? (keys + BN - 1) / BN : 0;
            for (int j = 0; j <= ntiles && ntiles > 0; ++j) {
                if (j < ntiles) {
                    const int gj = base + j;
                    warp_wait(bar_s_ready, gj & 1, kDevTimeoutMmaKV, a.status, s_abort, lane);
                    ptx::fence_after_sync();
                    if (ptx::elect_one()) {
                        const uint64_t kd = kdesc0 + (uint64_t)(((gj & 1) * Plan::kTile) >> 4);
#pragma unroll
                        for (int x = 0; x < 6; ++x)
#pragma unroll
                            for (int ks = 0; ks < D / 16; ++ks)
                                ptx::mma_ts(tmem + Plan::kColS + (ks & 1) * BN, tmem + kPa[x] * (D / 2) + ks * 8,
                                            kd + (uint64_t)((kPb[x] * Plan::kPart + (ks >> 2) * Plan::kBlk + (ks & 3) * 32) >> 4), idesc_s, x > 0 || ks > 1);
                        ptx::mma_commit(bar_s_done);
                    }
                    __syncwarp();
                }
                if (j > 0) {
                    const int gj = base + j - 1;
                    warp_wait(bar_p_ready, gj & 1, kDevTimeoutMmaP, a.status, s_abort, lane);
                    ptx::fence_after_sync();
                    if (ptx::elect_one()) {
                        const uint64_t vd = vdesc0 + (uint64_t)(((gj & 1) * Plan::kTile) >> 4);
#pragma unroll
                        for (int x = 0; x < 6; ++x)
#pragma unroll
                            for (int ks = 0; ks < BN / 16; ++ks) {
                                const uint64_t v = vd + (uint64_t)((kPb[x] * Plan::kPart + ks * 2048) >> 4);
                                if (!Plan::kPLoTmem && kPa[x] == 2) ptx::mma_ss(tmem + Plan::kColO, pdesc + (uint64_t)(ks * 2), v, idesc_o, x > 0 || ks > 0);
                                else ptx::mma_ts(tmem + Plan::kColO, tmem + Plan::kColP + kPa[x] * (BN / 2) + ks * 8, v, idesc_o, x > 0 || ks > 0);
                            }
                        ptx::mma_commit(bar_o_done);
                    }
                    __syncwarp();
                }
            }
            base += ntiles;
        } while (next_block());
    } else {
        // ================= operands, softmax, accumulation =================
        const int quarter = warp & 3, part = warp >> 2;      // TMEM lane quarter; score columns and channels
        const int r_tile = quarter * 32 + lane;              // row of the block
        const uint32_t t_lane = tmem + ((uint32_t)(quarter << 5) << 16);
        auto all_compute = []() { asm volatile("bar.sync 5, 512;" ::: "memory"); };
        auto arrive = [&](uint32_t bar) {
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(bar);
        };
        // a tile of K or V: 4 channels of a key per vector, a key's D channels side by side in a warp
        constexpr int kRowStep = kF32Compute / (D / 4);      // keys between a thread's vectors
        static_assert(kRowStep % 8 == 0, "a thread's keys have the same place in the swizzle");
        const int t_row = tid / (D / 4), t_vec = tid % (D / 4);
        const uint32_t t_place = (t_vec >> 4) * Plan::kBlk + t_row * 128 + ((((t_vec & 15) >> 1) ^ (t_row & 7)) << 4) + (t_vec & 1) * 8;
        auto load_tile = [&](ulonglong2 (&x)[kVecs], const float* from, int rows) {
#pragma unroll
            for (int i = 0; i < kVecs; ++i) {
                x[i] = make_ulonglong2(0ull, 0ull);
                if (t_row + i * kRowStep < rows) x[i] = *reinterpret_cast<const ulonglong2*>(from + tid * 4 + i * (kF32Compute * 4));
            }
        };
        int turn = 0;
        auto store_tile = [&](const ulonglong2 (&x)[kVecs], uint8_t* to, bool is_k) {
            uint32_t top = 0;
#pragma unroll
            for (int i = 0; i < kVecs; ++i) {
                uint2 p[3];
                split3(x[i].x, p[0].x, p[1].x, p[2].x);
                split3(x[i].y, p[0].y, p[1].y, p[2].y);
                if (is_k) top = ptx::max_abs_bf16x2(ptx::max_abs_bf16x2(top, p[0].x), p[0].y);
#pragma unroll
                for (int y = 0; y < 3; ++y) *reinterpret_cast<uint2*>(to + t_place + i * (kRowStep * 128) + y * Plan::kPart) = p[y];
            }
            if (is_k && f32_huge(a, top)) atomicOr(&s_bad[turn & 1], 1);
        };
        do {
            const int row0 = rb * BM, t_lo = j_lo * BN, keys = keys_of(), ntiles = keys > 0 ? (keys + BN - 1) / BN : 0;
            const int row = row0 + r_tile;
            const bool row_valid = row < R;
            const float* kb = (const float*)a.k_cache + ((long)g * a.cache_cap + t_lo) * D;
            const float* vb = (const float*)a.v_cache + ((long)g * a.cache_cap + t_lo) * D;
            const float* qrow = (const float*)a.q_rot + ((long)g * R + row) * D + part * kCh;
            const int seen = a.cache_len + row / a.G - t_lo - part * 16;    // columns 0 .. seen of this thread's tile 0

            ulonglong2 x[kVecs];                             // the next tile of K or V to split, on its way
            uint64_t acc[kCh / 2];                           // channel pairs
#pragma unroll
            for (int c = 0; c < kCh / 2; ++c) acc[c] = 0ull;
            float m = -INFINITY, l = 0.f;
            if (ntiles > 0) {
                load_tile(x, kb, keys);
                // the row's channels of this thread: three parts into tensor memory (the scores of the row block
                // before are done: all its warps waited for them)
                ulonglong2 q[kCh / 4];
#pragma unroll
                for (int c = 0; c < kCh / 4; ++c) {
                    q[c] = make_ulonglong2(0ull, 0ull);
                    if (row_valid) q[c] = reinterpret_cast<const ulonglong2*>(qrow)[c];
                }
                uint32_t top = 0;
                __syncwarp();
#pragma unroll
                for (int h = 0; h < kCh / 16; ++h) {
                    uint32_t p[3][8];
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        split3(q[4 * h + c].x, p[0][2 * c], p[1][2 * c], p[2][2 * c]);
                        split3(q[4 * h + c].y, p[0][2 * c + 1], p[1][2 * c + 1], p[2][2 * c + 1]);
                        top = ptx::max_abs_bf16x2(ptx::max_abs_bf16x2(top, p[0][2 * c]), p[0][2 * c + 1]);
                    }
#pragma unroll
                    for (int y = 0; y < 3; ++y) ptx::tmem_st8(t_lane + y * (D / 2) + part * (kCh / 2) + h * 8, p[y]);
                }
                if (f32_huge(a, top)) atomicOr(&s_bad[turn & 1], 1);
                store_tile(x, smem + Plan::kKOff + (base & 1) * Plan::kTile, true);
                ptx::tmem_st_wait();
                ptx::fence_before_sync();
                ptx::fence_proxy_async();
                arrive(bar_s_ready);
                if (ntiles > 1) load_tile(x, kb + (long)BN * D, keys - BN);
            }
            for (int j = 0; j < ntiles; ++j) {
                const int gj = base + j;
                // (tile j - 1 of the scores is done, and with it that K buffer)
                if (j + 1 < ntiles) store_tile(x, smem + Plan::kKOff + ((gj + 1) & 1) * Plan::kTile, true);
                load_tile(x, vb + (long)j * BN * D, keys - j * BN);
                warp_wait(bar_s_done, gj & 1, kDevTimeoutSoftmaxS, a.status, s_abort, lane);
                ptx::fence_after_sync();
                uint32_t s[16];
                ptx::tmem_ld16(t_lane + Plan::kColS + part * 16, s);
                {
                    uint32_t odd[16];
                    ptx::tmem_ld16(t_lane + Plan::kColS + BN + part * 16, odd);
                    ptx::tmem_ld_wait();
#pragma unroll
                    for (int e = 0; e < 16; e += 2) {
                        float lo, hi;
                        ptx::unpack2(ptx::add2(ptx::pack2(__uint_as_float(s[e]), __uint_as_float(s[e + 1])), ptx::pack2(__uint_as_float(odd[e]), __uint_as_float(odd[e + 1]))), lo, hi);
                        s[e] = __float_as_uint(lo);
                        s[e + 1] = __float_as_uint(hi);
                    }
                }
                ptx::fence_before_sync();
                if (j + 1 < ntiles) {
                    ptx::fence_proxy_async();
                    arrive(bar_s_ready);
                }

                const int lim = seen - j * BN;
                if (!__all_sync(0xffffffffu, lim >= 15)) {
#pragma unroll
                    for (int e = 0; e < 16; ++e)
                        if (e > lim) s[e] = 0xff800000u;
                }
                float mx0 = -INFINITY, mx1 = -INFINITY;
#pragma unroll
                for (int e = 0; e < 16; e += 4) {
                    mx0 = ptx::max3(mx0, __uint_as_float(s[e]), __uint_as_float(s[e + 1]));
                    mx1 = ptx::max3(mx1, __uint_as_float(s[e + 2]), __uint_as_float(s[e + 3]));
                }
                float* xm = s_max + (gj & 1) * 512 + r_tile;
                xm[part * 128] = fmaxf(mx0, mx1);
                asm volatile("bar.sync %0, 128;" ::"r"(1 + quarter) : "memory");
                // (the maximum stays unscaled: a difference of scores is as exact as the scores, and 0 for the largest)
                const float m_new = fmaxf(ptx::max3(m, xm[0], xm[128]), fmaxf(xm[256], xm[384]));
                const float ref = (m_new == -INFINITY) ? 0.f : m_new;      // a row that has seen no key yet: every p is 0
                const float alpha = f32_rescale(a, m - ref);                // m = -inf: 0
                m = m_new;
                const uint64_t minus_ref = ptx::pack2(-ref, -ref);
                uint64_t sum2 = 0ull, pp[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    pp[e] = f32_weights(a, ptx::add2(ptx::pack2(__uint_as_float(s[2 * e]), __uint_as_float(s[2 * e + 1])), minus_ref));
                    sum2 = ptx::add2(sum2, pp[e]);
                }
                {
                    float s0, s1;
                    ptx::unpack2(sum2, s0, s1);
                    l = l * alpha + (s0 + s1);
                }
                store_tile(x, smem + Plan::kVOff + (gj & 1) * Plan::kTile, false);        // (the product of tile j - 2 is done)
                if (j + 2 < ntiles) load_tile(x, kb + (long)(j + 2) * BN * D, keys - (j + 2) * BN);
                if (j > 0) {
                    warp_wait(bar_o_done, (gj - 1) & 1, kDevTimeoutSoftmaxO, a.status, s_abort, lane);
                    ptx::fence_after_sync();
#pragma unroll
                    for (int h = 0; h < kCh; h += 16) {
                        uint32_t o[16];
                        ptx::tmem_ld16(t_lane + Plan::kColO + part * kCh + h, o);
                        ptx::tmem_ld_wait();
#pragma unroll
                        for (int c = 0; c < 16; c += 2)
                            acc[(h + c) / 2] = ptx::mul2(ptx::add2(acc[(h + c) / 2], ptx::pack2(__uint_as_float(o[c]), __uint_as_float(o[c + 1]))), ptx::pack2(alpha, alpha));
                    }
                }
                {
                    uint32_t p[3][8];
#pragma unroll
                    for (int e = 0; e < 8; ++e) split3(pp[e], p[0][e], p[1][e], p[2][e]);
#pragma unroll
                    for (int y = 0; y < (Plan::kPLoTmem ? 3 : 2); ++y) ptx::tmem_st8(t_lane + Plan::kColP + y * (BN / 2) + part * 8, p[y]);
#pragma unroll
                    for (int h = 0; h < (Plan::kPLoTmem ? 0 : 2); ++h)
                        *reinterpret_cast<uint4*>(smem + Plan::kPLoOff + r_tile * 128 + (((2 * part + h) ^ (r_tile & 7)) << 4)) =
                            make_uint4(p[2][4 * h], p[2][4 * h + 1], p[2][4 * h + 2], p[2][4 * h + 3]);
                }
                ptx::tmem_st_wait();
                ptx::fence_before_sync();
                ptx::fence_proxy_async();
                arrive(bar_p_ready);
            }
            bool bad = false, small = false;
            if (ntiles > 0) {
                warp_wait(bar_o_done, (base + ntiles - 1) & 1, kDevTimeoutSoftmaxO, a.status, s_abort, lane);
                ptx::fence_after_sync();
#pragma unroll
                for (int h = 0; h < kCh; h += 16) {
                    uint32_t o[16];
                    ptx::tmem_ld16(t_lane + Plan::kColO + part * kCh + h, o);
                    ptx::tmem_ld_wait();
#pragma unroll
                    for (int c = 0; c < 16; c += 2)
                        acc[(h + c) / 2] = ptx::add2(acc[(h + c) / 2], ptx::pack2(__uint_as_float(o[c]), __uint_as_float(o[c + 1])));
                }
                ptx::fence_before_sync();
                // Infinities and undefined numbers do not split, and a masked key's probability of 0 times an infinite value is
                // undefined: a row block whose results are not all finite is done again row by row, in floats, each row over the keys
                // it sees; so are small sums of values whose parts are not exact.
#pragma unroll
                for (int c = 0; c < kCh / 2; ++c) {
                    float y0, y1;
                    ptx::unpack2(acc[c], y0, y1);
                    bad |= !(fabsf(y0) + fabsf(y1) <= 3.0e38f);
                    small |= f32_small(y0) || f32_small(y1);
                }
                bad = bad && row_valid;
                small = small && row_valid;
            }
            s_sum[part * 128 + r_tile] = l;
            if (bad || small) atomicOr(&s_bad[turn & 1], (bad ? 1 : 0) + (small ? 2 : 0));
            all_compute();
            if (tid == 0) s_bad[(turn & 1) ^ 1] = s_inexact[(turn & 1) ^ 1] = 0;
            int again = *(volatile int*)&s_bad[turn & 1];
            if (again == 2) {                                // (a look at the values costs a fraction of doing the block again)
                bool inexact = false;
                for (int i = tid; i < keys * (D / 4); i += kF32Compute) inexact |= f32_inexact(reinterpret_cast<const float4*>(vb)[i]);
                if (inexact) s_inexact[turn & 1] = 1;
                all_compute();
                again = *(volatile int*)&s_inexact[turn & 1];
            }
            if (again == 0) {
                const float sum = (s_sum[r_tile] + s_sum[128 + r_tile]) + (s_sum[256 + r_tile] + s_sum[384 + r_tile]);
                const float inv = (sum > 0.f) ? 1.f / sum : 0.f;
                const long prow0 = ((long)split * a.Hkv + g) * R + row0 + quarter * 32;
                const int rows_here = R - row0 - quarter * 32;
                // 32 rows of D / 4 channels a warp, through shared memory so that stores are whole lines
                uint8_t* stage = smem + Plan::kKOff + warp * 32 * Plan::kOutStride;
#pragma unroll
                for (int c = 0; c < kCh; c += 4)
                    *reinterpret_cast<ulonglong2*>(stage + lane * Plan::kOutStride + c * 4) =
                        make_ulonglong2(ptx::mul2(acc[c / 2], ptx::pack2(inv, inv)), ptx::mul2(acc[c / 2 + 1], ptx::pack2(inv, inv)));
                __syncwarp();
                constexpr int kLanes = kCh / 4;              // lanes a row
#pragma unroll
                for (int i = 0; i < 32; i += 32 / kLanes) {
                    const int r = i + lane / kLanes;
                    if (r < rows_here)
                        *reinterpret_cast<float4*>(a.o_part + (prow0 + r) * D + part * kCh + (lane % kLanes) * 4) =
                            *reinterpret_cast<const float4*>(stage + r * Plan::kOutStride + (lane % kLanes) * 16);
                }
                if (part == 0 && row_valid) a.lse_part[prow0 + lane] = f32_lse(a, m, sum);
            } else {
                const int last_row = min(row0 + BM, R) - 1;
                for (int r = row0 + warp; r <= last_row; r += kF32Compute / 32) {
                    const long prow = ((long)split * a.Hkv + g) * R + r;
                    simt_row<float, D>((const float*)a.q_rot + ((long)g * R + r) * D, kb, vb, a.o_part + prow * D, a.lse_part + prow, a.scale,
                                       min(keys, a.cache_len + r / a.G + 1 - t_lo));
                }
            }
            all_compute();                                   // the sums and the staged rows are read
            base += ntiles;
            ++turn;
        } while (next_block());
    }

    ptx::fence_before_sync();
    __syncthreads();
    if (warp == kF32Compute / 32) {
        if (*s_abort) {                                      // products that nobody waited for have time to end
            const long long t0 = clock64();
            while (clock64() - t0 < 400000) { }
        }
        ptx::fence_after_sync();
        ptx::tmem_dealloc(tmem, 512);
    }
}

}  // namespace evln
