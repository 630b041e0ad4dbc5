// Re-indexing of an un-rotated cache (Sec. 3.2: the KV cache is stored before the rotation, the
// frame sampler picks the frames to keep, the kept tokens get contiguous position ids and RoPE is
// applied on the fly).
//
// store_append_kernel: the new frame's raw (un-rotated) K and V go to the store, head-major.
// gather_rope_kernel: the kept segments of the store are laid out back to back in a working cache;
// the token that lands in working slot p is rotated at position p (keys) or copied (values); angles in double precision as in the append kernel (or from the
// caller's position table).  HBM-bound: every
// kept element is read once and written once with 128-bit accesses.
#pragma once

#include "common.cuh"
#include "rope_append.cuh"

namespace evln {

constexpr int kMaxSegments = 256;

// Kept segments, passed by value: segment s = store slots [src[s], src[s] + dst_off[s+1] - dst_off[s])
// -> working slots [dst_off[s], dst_off[s+1]).
struct SegList {
    int src[kMaxSegments];
    int dst_off[kMaxSegments + 1];
};

struct GatherArgs {
    const void* k_src;      // store_append: k_new [n, Hkv, D] (token stride given); gather: store [Hkv, store_cap, D]
    const void* v_src;
    void* k_dst;            // store_append: store; gather: working cache [Hkv, work_cap, D]
    void* v_dst;
    long k_stride, v_stride;    // store_append only: token strides of k_new / v_new in elements
    int Hkv, D;
    int src_cap, dst_cap;
    int first_slot;         // store_append: first store slot written
    int num_tokens;         // destination tokens
    int num_segments;       // gather only
    double log2_theta;      // gather only
    const double2* table;   // gather only, optional: (cos, sin) per (position - table_first, j)
    int table_first;
    // gather only, by the host: log2 of the 16-byte vectors per half head vector, chunks per token
    int vph_shift, k_chunks, v_chunks;
    FastDiv div_chunks;     // division by k_chunks + v_chunks
};

template <typename T>
__global__ void __launch_bounds__(128)
store_append_kernel(const GatherArgs a)
{
    constexpr int V = VecTraits<T>::kVec;
    const int tok = blockIdx.x;
    const int per_row = a.D / V;
    const int items = 2 * a.Hkv * per_row;
    if (a.num_tokens <= kRopeFewTokens) {                    // as in the append kernel (746 and 740 us for the same step)
        const int lines = a.Hkv * a.D * (int)sizeof(T) / 128;
        for (int i = threadIdx.x; i < 2 * lines; i += blockDim.x)
            ptx::prefetch_l2(reinterpret_cast<const char*>(i < lines ? (const T*)a.k_src + tok * a.k_stride : (const T*)a.v_src + tok * a.v_stride) +
                             (i < lines ? i : i - lines) * 128);
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    for (int it = threadIdx.x; it < items; it += blockDim.x) {
        const bool is_v = it >= a.Hkv * per_row;
        const int e = is_v ? it - a.Hkv * per_row : it;
        const int g = e / per_row, d0 = (e % per_row) * V;
        const T* src = (const T*)(is_v ? a.v_src : a.k_src) + (long)tok * (is_v ? a.v_stride : a.k_stride) + (long)g * a.D + d0;
        T* dst = (T*)(is_v ? a.v_dst : a.k_dst) + ((long)g * a.dst_cap + a.first_slot + tok) * a.D + d0;
        *reinterpret_cast<uint4*>(dst) = *reinterpret_cast<const uint4*>(src);
    }
}

// A warp per chunk of a destination token: 32 vector pairs of its keys, or 64 vectors of its values.  Warps
// do not wait for each other, so a call of a few thousand tokens is one wave of short chains (a block
// per token, all of it behind the angles: 6.5 us for 3392 tokens of 4 kv heads; this: 5.3).  For tokens whose keys are
// one chunk, and for few tokens: every further chunk of keys needs the token's angles again.
// WAVE: all blocks run at once.  Then they are there while the previous kernel ends, and each warp requests its source rows into L2
// meanwhile; bounded to 40 registers (a few words spilled to L1), so that six blocks fit an SM instead of the five that 48 registers
// leave (28 re-indexed layers of 3392 kept tokens 774 us, 736 with the requests, 724 with six blocks; eight, at 32 registers: 780).
// More tokens run in several rounds, whose blocks are not there ahead of time: requests and spills only cost (us a layer, 20000 tokens
// of 4 kv heads without a table 20.5, 23.9 in the form for one wave; 5000 of 1 head 6.1 and 6.9).  Two rounds are a little faster so where
// warps are full and the angles come from a table (1700 tokens of 32 kv heads of 64 channels 7.2 and 6.7, 5000 of 4 in fp32 5.5 and 5.2).
constexpr int kGatherWarps = 8, kGatherWaveBlocks = 6;
// Nor is that form used where the SMs have several blocks of little to request each (844 tokens of one kv head 2.16 us and 2.53; 250
// 2.07 and 2.06, 3392 5.7 and 4.4), or a block's warps share a token's many chunks of keys (60 tokens of 32 kv heads 2.59 and 2.68).
inline bool gather_one_wave(int k_items, int k_chunks, long blocks, bool table, int sms)
{
    if (blocks > (long)kGatherWaveBlocks * sms * (table && k_items >= 32 ? 2 : 1)) return false;
    return k_chunks > 4 ? blocks > sms : blocks <= sms || k_items * blocks > 32L * sms;
}

template <typename T, bool WAVE>
__global__ void __launch_bounds__(32 * kGatherWarps, WAVE ? kGatherWaveBlocks : 0)
gather_rope_kernel(const GatherArgs a, const __grid_constant__ SegList segs)
{
    constexpr int V = VecTraits<T>::kVec;
    __shared__ typename Rotation<T>::Angle s_angles[kGatherWarps][Rotation<T>::kAngles];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t task = blockIdx.x * (uint32_t)kGatherWarps + (uint32_t)warp;
    const int pos = (int)fast_div(task, a.div_chunks);     // working slot = new position id
    const int chunk = (int)task - pos * (a.k_chunks + a.v_chunks);
    const int D = a.D, half = D / 2;
    int lo = 0, hi = a.num_segments;                       // largest s with dst_off[s] <= pos
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (segs.dst_off[mid] <= pos) lo = mid; else hi = mid;
    }
    const long src_slot = segs.src[lo] + (pos - segs.dst_off[lo]);
    if (WAVE && pos < a.num_tokens) {
        const bool is_k = chunk < a.k_chunks;
        const int row_lines = D * (int)sizeof(T) / 128, chunks = is_k ? a.k_chunks : a.v_chunks, lines = (a.Hkv * row_lines + chunks - 1) / chunks;
        const char* from = reinterpret_cast<const char*>((const T*)(is_k ? a.k_src : a.v_src) + src_slot * D);
        for (int i = lane; i < lines; i += 32) {
            const int line = (is_k ? chunk : chunk - a.k_chunks) * lines + i, g = line / row_lines;
            if (g < a.Hkv) ptx::prefetch_l2(from + (long)g * a.src_cap * D * sizeof(T) + line % row_lines * 128);
        }
    }
    // (so far launch parameters only)
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (pos >= a.num_tokens) return;

    if (chunk < a.k_chunks) {
        const int it = chunk * 32 + lane, k = it & ((1 << a.vph_shift) - 1), g = it >> a.vph_shift;
        const bool mine = g < a.Hkv;
        const T* src = (const T*)a.k_src + ((long)g * a.src_cap + src_slot) * D + k * V;
        uint4 lo_raw = make_uint4(0u, 0u, 0u, 0u), hi_raw = lo_raw;
        if (mine) {
            lo_raw = *reinterpret_cast<const uint4*>(src);
            hi_raw = *reinterpret_cast<const uint4*>(src + half);
        }
        for (int j = lane; j < half; j += 32)
            Rotation<T>::put(s_angles[warp], j, a.table ? a.table[(long)(pos - a.table_first) * half + j] : rope_cos_sin(pos, j, D, a.log2_theta));
        __syncwarp();
        if (mine) {
            uint4 out_lo, out_hi;
            Rotation<T>::turn(s_angles[warp], k, lo_raw, hi_raw, out_lo, out_hi);
            T* dst = (T*)a.k_dst + ((long)g * a.dst_cap + pos) * D + k * V;
            *reinterpret_cast<uint4*>(dst) = out_lo;
            *reinterpret_cast<uint4*>(dst + half) = out_hi;
        }
    } else {
        uint4 x[2];
        const int it = (chunk - a.k_chunks) * 64 + lane;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int d = (it + 32 * i) & ((2 << a.vph_shift) - 1), g = (it + 32 * i) >> (a.vph_shift + 1);
            if (g < a.Hkv) x[i] = *reinterpret_cast<const uint4*>((const T*)a.v_src + ((long)g * a.src_cap + src_slot) * D + d * V);
        }
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int d = (it + 32 * i) & ((2 << a.vph_shift) - 1), g = (it + 32 * i) >> (a.vph_shift + 1);
            if (g < a.Hkv) *reinterpret_cast<uint4*>((T*)a.v_dst + ((long)g * a.dst_cap + pos) * D + d * V) = x[i];
        }
    }
}

// A block per destination token, which forms (or reads) the token's angles once for all its heads: more than one chunk of
// keys, and enough tokens (of few, a warp per chunk spreads the work further).  3392 tokens of 8 kv heads: without a
// table bf16 6.5 us, a warp per chunk 8.5, fp32 7.6 and 11.7; with one 5.8 and 6.0, 6.9 and 8.5.  32 heads of 250 fp32
// tokens with a table 4.8 and 3.3, of 60 without one 4.9 and 3.3.  bf16 of head_dim 64 with a table (short rows, one
// read of the angles per 64 channels) stays with the warps: 16 heads, 20000 tokens 39.8 and 33.4.
constexpr int kGatherBlockThreads = 128;
inline bool gather_by_block(int k_chunks, long tokens, bool table, bool bf16, int D)
{
    return k_chunks > 1 && tokens > (table ? 512 : 128) && !(table && bf16 && D == 64);
}

template <typename T>
__global__ void __launch_bounds__(kGatherBlockThreads, 12)
gather_rope_block_kernel(const GatherArgs a, const __grid_constant__ SegList segs)
{
    constexpr int V = VecTraits<T>::kVec;
    __shared__ typename Rotation<T>::Angle s_angle[Rotation<T>::kAngles];
    const int pos = (int)blockIdx.x;                       // working slot = new position id
    const int D = a.D, half = D / 2;
    int lo = 0, hi = a.num_segments;                       // largest s with dst_off[s] <= pos
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (segs.dst_off[mid] <= pos) lo = mid; else hi = mid;
    }
    const long src_slot = segs.src[lo] + (pos - segs.dst_off[lo]);
    // (so far launch parameters only)
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if ((int)threadIdx.x < half) {
        const int j = threadIdx.x;
        Rotation<T>::put(s_angle, j, a.table ? a.table[(long)(pos - a.table_first) * half + j] : rope_cos_sin(pos, j, D, a.log2_theta));
    }
    __syncthreads();

    const int k_items = a.Hkv << a.vph_shift, v_items = a.Hkv << (a.vph_shift + 1);
    for (int it = threadIdx.x; it < k_items + v_items; it += kGatherBlockThreads) {
        if (it < k_items) {
            const int k = it & ((1 << a.vph_shift) - 1), g = it >> a.vph_shift;
            const T* src = (const T*)a.k_src + ((long)g * a.src_cap + src_slot) * D + k * V;
            const uint4 lo_raw = *reinterpret_cast<const uint4*>(src), hi_raw = *reinterpret_cast<const uint4*>(src + half);
            uint4 out_lo, out_hi;
            Rotation<T>::turn(s_angle, k, lo_raw, hi_raw, out_lo, out_hi);
            T* dst = (T*)a.k_dst + ((long)g * a.dst_cap + pos) * D + k * V;
            *reinterpret_cast<uint4*>(dst) = out_lo;
            *reinterpret_cast<uint4*>(dst + half) = out_hi;
        } else {
            const int e = it - k_items, d = e & ((2 << a.vph_shift) - 1), g = e >> (a.vph_shift + 1);
            *reinterpret_cast<uint4*>((T*)a.v_dst + ((long)g * a.dst_cap + pos) * D + d * V) =
                *reinterpret_cast<const uint4*>((const T*)a.v_src + ((long)g * a.src_cap + src_slot) * D + d * V);
        }
    }
}

}  // namespace evln
