// Fused RoPE-rotate-and-append kernel (Sec. 3.2: contiguous position ids, rotation,
// concatenation of the new frame with the reused cache).
//
// One CTA per new token.  D/2 threads get the token's cos/sin of phi_j = pos * theta^(-2j/D) in double
// precision (pos reaches tens of thousands; a float angle would be off by ~1e-3 rad) into shared memory
// for all heads: from the caller's position table when there is one (the table depends on the positions
// only, so a model makes it once per navigation step for all its layers: rope_table_kernel below), else
// formed on the spot.  Every thread moves 16-byte vectors (a work item is a pair of vectors (j.., j + D/2..)
// of a query or key head, or one vector of a value head): rotated query halves to the kv-head-grouped
// q_rot scratch, rotated key halves and the unchanged values to the token's cache slot; the loads are
// issued before the cos/sin are waited for.
// Bound: a step's few hundred tokens are one chain of latencies (2.3 us for 196 tokens of the 7B shape,
// 1.8 for one; 3.4 and 2.6 before the rotation was packed), thousands are bound by the instructions of
// the rotation and then by HBM (each element read once and written once: 2048 tokens 9.8 us, 3136 paged
// ones 17.6, 16 and 25 before; 6 and 9 us at the copy rate).
// (Letting every thread read the table entries of its own vector instead of sharing them through shared
// memory was measured slower: 32 heads re-read the same 64 entries.)
#pragma once

#include "common.cuh"
#include "ptx_sm100.cuh"

namespace evln {

struct RopeArgs {
    const void* q_new;
    const void* k_new;
    const void* v_new;
    void* q_rot;
    void* k_cache;      // contiguous: [Hkv, cap, D]; paged: pool [pages, Hkv, page, D]
    void* v_cache;
    const int* page_table;   // paged only: [batch, max_pages]
    long q_stride, k_stride, v_stride;   // token strides in elements
    int Hq, Hkv, D;
    int cache_len;      // contiguous only
    int num_new;        // contiguous: n; paged: total new tokens
    int cache_cap;      // contiguous only
    int batch, page_size, max_pages;     // paged only
    double log2_theta;
    const double2* table;   // optional: (cos, sin) per (position - table_first, j), [count][D/2]
    int table_first;
    // derived by the host (finish_rope_args): the threads decode their work with shifts and one
    // multiplication instead of integer divisions
    int G;                  // Hq / Hkv
    FastDiv div_g;
    int vph_shift;          // log2 of the 16-byte vectors per half head vector (D/2 / V)
    int page_shift;         // log2(page_size)
};

// cos/sin of pos * theta^(-2j/D): the one definition the append, gather and table kernels share
__device__ __forceinline__ double rope_omega(int j, int D, double log2_theta)
{
    return exp2(-(2.0 * (double)j / (double)D) * log2_theta);
}
__device__ __forceinline__ double2 rope_cos_sin_at(long pos, double omega)
{
    double s, c;
    // sin/cos(pos * omega) through sincospi: its range reduction is exact and cheap, where a
    // plain sincos of an argument of thousands of radians takes the slow reduction path
    sincospi((double)pos * omega * 0.31830988618379067154, &s, &c);
    return make_double2(c, s);
}
__device__ __forceinline__ double2 rope_cos_sin(long pos, int j, int D, double log2_theta)
{
    return rope_cos_sin_at(pos, rope_omega(j, D, log2_theta));
}

// The rotation itself.  Products and sums are formed with at least 40 bits, then rounded once to float and
// once to the storage dtype (a float product would lose bits exactly where x0*c and x1*s cancel).
//  - float: in double.
//  - bf16: in pairs of floats, two channels per packed instruction.  A double operation and the
//    conversions around it issue at a small fraction of the float rate (32 double operations and 32
//    conversions per vector pair kept an SM at ~7 per cycle), and what bounds the append and gather
//    kernels for thousands of tokens is the instructions they issue.  The angle is split into 16 bits and
//    a float rest (40 bits), so a bf16 value times the first part is an exact float; the two exact products
//    are added with the rounding error recovered (Knuth's two-sum), which the products with the rest join.
// put(): angle j into a shared-memory array of kAngles; turn(): vector k (of a half head) of both halves.
template <typename T> struct Rotation;
template <> struct Rotation<float> {
    typedef double2 Angle;                       // (cos, sin); angle j at j + j / 8 (bank spread)
    static constexpr int kAngles = 72;
    static __device__ __forceinline__ void put(Angle* s, int j, const double2& cs) { s[j + (j >> 3)] = cs; }
    static __device__ __forceinline__ void turn(const Angle* s, int k, const uint4& lo, const uint4& hi, uint4& out_lo, uint4& out_hi)
    {
        const float* x0 = reinterpret_cast<const float*>(&lo);
        const float* x1 = reinterpret_cast<const float*>(&hi);
        float* y0 = reinterpret_cast<float*>(&out_lo);
        float* y1 = reinterpret_cast<float*>(&out_hi);
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            const int j = 4 * k + v;
            const Angle a = s[j + (j >> 3)];
            y0[v] = (float)((double)x0[v] * a.x - (double)x1[v] * a.y);
            y1[v] = (float)((double)x1[v] * a.x + (double)x0[v] * a.y);
        }
    }
};
template <> struct Rotation<__nv_bfloat16> {
    // a channel pair is two of these: (cos 16 bits of both, rest of both), (sin ..., ...); the pairs of a
    // 16-byte vector take 9 places, so that the vectors of a half head start in different banks
    typedef float4 Angle;
    static constexpr int kAngles = 72;
    static __device__ __forceinline__ int place(int pair) { return 2 * pair + (pair >> 2); }
    static __device__ __forceinline__ void put(Angle* s, int j, const double2& cs)
    {
        const float ch = __uint_as_float(__float_as_uint((float)cs.x) & 0xffffff00u);
        const float sh = __uint_as_float(__float_as_uint((float)cs.y) & 0xffffff00u);
        float* at = reinterpret_cast<float*>(s + place(j >> 1)) + (j & 1);
        at[0] = ch;
        at[2] = (float)(cs.x - (double)ch);
        at[4] = sh;
        at[6] = (float)(cs.y - (double)sh);
    }
    // x * (ch + cl) + z * (sh + sl)
    static __device__ __forceinline__ uint64_t combine(uint64_t x, uint64_t z, uint64_t ch, uint64_t cl, uint64_t sh, uint64_t sl)
    {
        const uint64_t minus = ptx::pack2(-1.f, -1.f);
        const uint64_t p = ptx::mul2(x, ch), q = ptx::mul2(z, sh);
        const uint64_t d = ptx::add2(p, q);
        const uint64_t nb = ptx::fma2(d, minus, p);                     // p - d: minus the part of q that d holds
        const uint64_t err = ptx::add2(ptx::fma2(ptx::add2(d, nb), minus, p), ptx::add2(q, nb));
        float r0, r1;
        ptx::unpack2(ptx::fma2(z, sl, ptx::fma2(x, cl, err)), r0, r1);
        // (an infinite or undefined d stays what it is: its rest is undefined, and min() drops that)
        return ptx::add2(d, ptx::pack2(fminf(r0, 3.0e38f), fminf(r1, 3.0e38f)));
    }
    // a channel pair: words of the lower and the upper half
    static __device__ __forceinline__ void turn_pair(const Angle& c, const Angle& s, uint32_t lo, uint32_t hi, uint32_t& out_lo,
                                                     uint32_t& out_hi)
    {
        const uint32_t nhi = hi ^ 0x80008000u;
        const uint64_t x0 = ptx::pack2(__uint_as_float(lo << 16), __uint_as_float(lo & 0xffff0000u));
        const uint64_t x1 = ptx::pack2(__uint_as_float(hi << 16), __uint_as_float(hi & 0xffff0000u));
        const uint64_t n1 = ptx::pack2(__uint_as_float(nhi << 16), __uint_as_float(nhi & 0xffff0000u));
        const uint64_t ch = ptx::pack2(c.x, c.y), cl = ptx::pack2(c.z, c.w), sh = ptx::pack2(s.x, s.y), sl = ptx::pack2(s.z, s.w);
        float a, b;
        ptx::unpack2(combine(x0, n1, ch, cl, sh, sl), a, b);
        out_lo = ptx::pack_bf16x2(a, b);
        ptx::unpack2(combine(x1, x0, ch, cl, sh, sl), a, b);
        out_hi = ptx::pack_bf16x2(a, b);
    }
    static __device__ __forceinline__ void turn(const Angle* s, int k, const uint4& lo, const uint4& hi, uint4& out_lo, uint4& out_hi)
    {
        const Angle* a = s + place(4 * k);
        const uint32_t x0[4] = {lo.x, lo.y, lo.z, lo.w}, x1[4] = {hi.x, hi.y, hi.z, hi.w};
        uint32_t y0[4], y1[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) turn_pair(a[2 * i], a[2 * i + 1], x0[i], x1[i], y0[i], y1[i]);
        out_lo = make_uint4(y0[0], y0[1], y0[2], y0[3]);
        out_hi = make_uint4(y1[0], y1[1], y1[2], y1[3]);
    }
};

// Position table: entry (p, j) = (cos, sin) of (first_pos + p) * theta^(-2j/D).
__global__ void __launch_bounds__(128)
rope_table_kernel(double2* table, int first_pos, int count, int D, double log2_theta)
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int half = D / 2;
    const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (long)count * half) return;
    const int p = (int)(i / half), j = (int)(i % half);
    table[i] = rope_cos_sin((long)first_pos + p, j, D, log2_theta);
}

// LensT is BatchLens for the paged kernel and NoLens (a stub) for the contiguous one.

// A block per token with one thread per work item (in whole warps, at most kRopeThreadsMax): every load of
// the token is in flight at once, and the other blocks of the SM hide its chain.  (Blocks that run through
// several tokens and prefetch the next one's vectors were measured slower, 10.3 against 9.8 us for 2048
// tokens and 19 against 17.6 for 3136 paged ones: what counts is warps, i.e. registers.)
constexpr int kRopeThreadsMax = 448;
constexpr int kRopeFewTokens = 256;      // (64 query heads: 8 tokens 27.2 us a step, 25.7 with two blocks each; 256 tokens 38.7 and 37.3)

// Where one new token comes from and goes to.
struct TokenPlace {
    int src_tok;             // its row of q_new / k_new / v_new
    int m;                   // its number in its run: query rows m * G ..
    int episode;             // paged: its episode; packed: 1 for an action token
    long kv_row;             // its key / value row of kv head 0
};
// The buffers a token's run goes to.
template <typename T>
struct TokenRun {
    T* q;                    // [Hkv, q_rows, D]
    T* k;                    // rows of kv head g start kv_rows * g behind those of head 0
    T* v;
    long q_rows, kv_rows;
};

// Rotates and stores token blockIdx.x with the whole block (gridDim.y > 1: a share of its work items).  place(token, t) fills in the token's place and
// returns its position, run(t) says which buffers it goes to.
template <typename T, typename Place, typename Run>
__device__ __forceinline__ void rope_token(const RopeArgs& a, Place&& place, Run&& run)
{
    constexpr int V = VecTraits<T>::kVec;
    typedef typename Rotation<T>::Angle Angle;
    __shared__ Angle s_angle[Rotation<T>::kAngles];
    const int D = a.D, half = D / 2, G = a.G;
    const int vph = a.vph_shift, vpr = a.vph_shift + 1;       // vectors per half head vector / per head vector (log2)
    const int q_items = a.Hq << vph;
    const int k_items = a.Hkv << vph;
    const int v_items = a.Hkv << vpr;
    const int items = q_items + k_items + v_items;

    // a work item `it` of a token: a pair of 16-byte vectors (j0.., j0+half..) of a query or key head, or one
    // 16-byte vector of a value head
    auto load_item = [&](const TokenPlace& t, int it, uint4& r0, uint4& r1) {
        if (it < q_items + k_items) {
            const bool is_q = it < q_items;
            const int e = is_q ? it : it - q_items;
            const int h = e >> vph;
            const int j0 = (e & ((1 << vph) - 1)) * V;
            const T* src = (is_q ? (const T*)a.q_new + t.src_tok * a.q_stride : (const T*)a.k_new + t.src_tok * a.k_stride) + (long)h * D;
            r0 = *reinterpret_cast<const uint4*>(src + j0);
            r1 = *reinterpret_cast<const uint4*>(src + j0 + half);
        } else {
            const int e = it - q_items - k_items;
            const int g = e >> vpr;
            const int d0 = (e & ((1 << vpr) - 1)) * V;
            r0 = *reinterpret_cast<const uint4*>((const T*)a.v_new + t.src_tok * a.v_stride + (long)g * D + d0);
        }
    };
    auto finish_item = [&](const TokenPlace& t, const Angle* s_angle, int it, const uint4& lo_raw, const uint4& hi_raw) {
        const TokenRun<T> to = run(t);
        if (it < q_items + k_items) {
            const bool is_q = it < q_items;
            const int e = is_q ? it : it - q_items;
            const int h = e >> vph;
            const int j0 = (e & ((1 << vph) - 1)) * V;
            T* dst;
            if (is_q) {
                const int g = (int)fast_div((uint32_t)h, a.div_g);
                dst = to.q + ((long)g * to.q_rows + (long)t.m * G + (h - g * G)) * D;
            } else {
                dst = to.k + ((long)h * to.kv_rows + t.kv_row) * D;
            }
            uint4 out_lo_raw, out_hi_raw;
            Rotation<T>::turn(s_angle, e & ((1 << vph) - 1), lo_raw, hi_raw, out_lo_raw, out_hi_raw);
            *reinterpret_cast<uint4*>(dst + j0) = out_lo_raw;
            *reinterpret_cast<uint4*>(dst + j0 + half) = out_hi_raw;
        } else {
            const int e = it - q_items - k_items;
            const int g = e >> vpr;
            const int d0 = (e & ((1 << vpr) - 1)) * V;
            *reinterpret_cast<uint4*>(to.v + ((long)g * to.kv_rows + t.kv_row) * D + d0) = lo_raw;
        }
    };

    const int j = threadIdx.x;
    // without a table: the thread's frequency, once (j / D as in rope_cos_sin)
    const double omega = !a.table && j < half ? rope_omega(j, D, a.log2_theta) : 0.0;
    auto angle_of = [&](long pos) -> double2 {
        return a.table ? a.table[(pos - a.table_first) * half + j] : rope_cos_sin_at(pos, omega);
    };

    const int tok = blockIdx.x;
    TokenPlace t;
    const long pos = place(tok, t);
    uint4 r0 = make_uint4(0u, 0u, 0u, 0u), r1 = r0;
    const int first = j + (int)(blockIdx.y * blockDim.x);
    if (first < items) load_item(t, first, r0, r1);   // in flight while the angles arrive
    if (j < half) Rotation<T>::put(s_angle, j, angle_of(pos));
    __syncthreads();
    if (first < items) finish_item(t, s_angle, first, r0, r1);
    for (int it = first + (int)(gridDim.y * blockDim.x); it < items; it += (int)(gridDim.y * blockDim.x)) {
        load_item(t, it, r0, r1);
        finish_item(t, s_angle, it, r0, r1);
    }
}

// FEW: at most kRopeFewTokens tokens.  Their blocks are all there while the previous kernel ends, so each requests its token's
// vectors into L2 meanwhile.  (28 layers of 256 tokens on an empty cache 277 us a pass, 271 so; 8 tokens over 20656 505 and 497.
// Many tokens, whose blocks are in line, 22.4 us for 21.8 of a step of 1024.)
template <typename T, bool PAGED, typename LensT, bool FEW>
__global__ void __launch_bounds__(kRopeThreadsMax, PAGED ? 3 : 1)
rope_append_kernel(const RopeArgs a, const __grid_constant__ LensT lens)
{
    constexpr int V = VecTraits<T>::kVec;
    const int D = a.D;
    int b = 0;                                    // the token's episode
    if (PAGED && (int)blockIdx.x >= a.num_new) {
        // An episode's last page is only partly filled: clear the value slots behind its last token so that a
        // tile load of the whole page never brings in stale bits.  (A block per episode: behind the stores of
        // the last token's block it was the longest chain of the launch, 4.65 us for 16 episodes of one token.)
        b = blockIdx.x - a.num_new;
        const int len = lens.cache_len[b] + lens.new_off[b + 1] - lens.new_off[b], used = len & (a.page_size - 1);
        asm volatile("griddepcontrol.wait;" ::: "memory");
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
        if (lens.new_off[b + 1] == lens.new_off[b] || used == 0) return;
        const long row = (long)a.page_table[(long)b * a.max_pages + (len >> a.page_shift)] * a.Hkv * a.page_size + used;
        const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
        for (int g = blockIdx.y; g < a.Hkv; g += gridDim.y) {
            uint4* dst = reinterpret_cast<uint4*>((T*)a.v_cache + (row + (long)g * a.page_size) * D);
            for (int it = threadIdx.x; it < (a.page_size - used) * (D / V); it += blockDim.x) dst[it] = zero;
        }
        return;
    }
    if (PAGED) {
        int hi = a.batch;                         // largest b with new_off[b] <= tok
        while (hi - b > 1) {
            const int mid = (b + hi) >> 1;
            if (lens.new_off[mid] <= (int)blockIdx.x) b = mid; else hi = mid;
        }
    }
    if constexpr (FEW) {
        const int tok = blockIdx.x, lines = D * (int)sizeof(T) / 128, q = a.Hq * lines, kv = a.Hkv * lines;
        for (int i = (int)(blockIdx.y * blockDim.x + threadIdx.x); i < q + 2 * kv; i += (int)(gridDim.y * blockDim.x)) {
            const T* row = i < q ? (const T*)a.q_new + tok * a.q_stride : i < q + kv ? (const T*)a.k_new + tok * a.k_stride : (const T*)a.v_new + tok * a.v_stride;
            ptx::prefetch_l2(reinterpret_cast<const char*>(row) + (i < q ? i : i < q + kv ? i - q : i - q - kv) * 128);
        }
    }
    // (so far launch parameters only; what follows reads memory that earlier kernels may have written)
    asm volatile("griddepcontrol.wait;" ::: "memory");          // programmatic dependent launch: inputs ready
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    auto place = [&](int tok, TokenPlace& t) -> long {          // tok: index into the packed new tokens
        t.src_tok = t.m = tok;
        if (!PAGED) return t.kv_row = (long)a.cache_len + tok;
        const int pos = lens.cache_len[b] + tok - lens.new_off[b];
        t.episode = b;
        t.kv_row = (long)a.page_table[(long)b * a.max_pages + (pos >> a.page_shift)] * a.Hkv * a.page_size + (pos & (a.page_size - 1));
        return pos;
    };
    auto run = [&](const TokenPlace&) -> TokenRun<T> {
        return {(T*)a.q_rot, (T*)a.k_cache, (T*)a.v_cache, (long)a.num_new * a.G, PAGED ? (long)a.page_size : (long)a.cache_cap};
    };
    rope_token<T>(a, place, run);
}

// The tokens of a packed sequence I, v_1, a_1, ..., v_N, a_N in one launch (Sec. 3.3): the instruction and
// visual tokens at contiguous positions into the cache, then the action tokens, chunk t at the positions
// that continue v_t, into buffers of their own.
struct RopePackedArgs {
    RopeArgs r;              // visual run: q_rot, k_cache, v_cache, cache_cap; num_new = all tokens
    int num_visual, num_action;
    int I, F, A;
    FastDiv div_f, div_a;
    void* q_rot_act;         // [Hkv, num_action * G, D]
    void* k_act;             // [Hkv, num_action, D]
    void* v_act;
};

__global__ void __launch_bounds__(kRopeThreadsMax, 3)
rope_packed_kernel(const RopePackedArgs p)
{
    typedef __nv_bfloat16 T;
    const RopeArgs& a = p.r;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    auto place = [&](int tok, TokenPlace& t) -> long {
        const bool action = tok >= p.num_visual;
        const int m = action ? tok - p.num_visual : tok;             // within its run
        long pos = m;
        t.src_tok = m;
        if (action) {
            const int c = (int)fast_div((uint32_t)m, p.div_a), i = m - c * p.A;
            pos = (long)p.I + (long)(c + 1) * p.F + i;
            t.src_tok = p.I + c * (p.F + p.A) + p.F + i;
        } else if (m >= p.I && p.F > 0) {
            t.src_tok += (int)fast_div((uint32_t)(m - p.I), p.div_f) * p.A;
        }
        t.m = m;
        t.kv_row = m;
        t.episode = action;
        return pos;
    };
    auto run = [&](const TokenPlace& t) -> TokenRun<T> {
        if (t.episode) return {(T*)p.q_rot_act, (T*)p.k_act, (T*)p.v_act, (long)p.num_action * a.G, p.num_action};
        return {(T*)a.q_rot, (T*)a.k_cache, (T*)a.v_cache, (long)p.num_visual * a.G, a.cache_cap};
    };
    rope_token<T>(a, place, run);
}

}  // namespace evln
