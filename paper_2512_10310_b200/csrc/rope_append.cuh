// Fused RoPE-rotate-and-append kernel (Sec. 3.2: contiguous position ids, rotation,
// concatenation of the new frame with the reused cache).
//
// One CTA per new token.  Phase 1: D/2 threads get the token's cos/sin of phi_j = pos * theta^(-2j/D)
// in double precision (pos reaches tens of thousands; a float angle would be off by ~1e-3 rad)
// into shared memory for all heads: from the caller's position table when there is one (the
// table depends on the positions only, so a model makes it once per navigation step for all its
// layers: rope_table_kernel below), else formed on the spot.  Phase 2: every thread moves 16-byte
// vectors (a work item is a pair of vectors (j.., j + D/2..) of a query or key head, or one vector
// of a value head): rotated query halves to the kv-head-grouped q_rot scratch, rotated key halves
// and the unchanged values to the token's cache slot; the loads of a thread's first item are issued
// before the cos/sin are waited for.  HBM-bound by bytes (each element is read once and written
// once with 128-bit accesses); at the sizes of a step it is one chain of latencies, which is why
// nothing in it divides, and why a call of few tokens gets one thread per work item (all loads of
// a token in flight at once).  (Letting every thread read the table entries of its own vector
// instead of sharing them through shared memory was measured slower: 32 heads re-read the same 64
// entries.)
#pragma once

#include "common.cuh"

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
__device__ __forceinline__ double2 rope_cos_sin(long pos, int j, int D, double log2_theta)
{
    const double omega = exp2(-(2.0 * (double)j / (double)D) * log2_theta);
    double s, c;
    // sin/cos(pos * omega) through sincospi: its range reduction is exact and cheap, where a
    // plain sincos of an argument of thousands of radians takes the slow reduction path
    sincospi((double)pos * omega * 0.31830988618379067154, &s, &c);
    return make_double2(c, s);
}

// The rotation itself.  Products and sums are formed with at least 47 bits, then rounded once to float and
// once to the storage dtype (a float product would lose bits exactly where x0*c and x1*s cancel).
//  - float: in double.
//  - bf16: in pairs of floats.  A double operation and the conversions around it issue at a small
//    fraction of the float rate (measured: 32 double operations and 32 conversions per vector pair kept
//    an SM at ~7 per cycle; the rotation was most of the append and gather kernels' time), and a bf16
//    value times a cosine split into two floats is exact up to 2^-48: p + e is the exact product with
//    the high part (fma), the low part joins the residual, the two products are subtracted with the
//    rounding error recovered (Knuth's two-sum).
template <typename T> struct Rotation;
template <> struct Rotation<float> {
    typedef double2 Angle;                       // (cos, sin)
    static __device__ __forceinline__ Angle angle(const double2& cs) { return cs; }
    static __device__ __forceinline__ void turn(float x0, float x1, const Angle& a, float& y0, float& y1)
    {
        y0 = (float)((double)x0 * a.x - (double)x1 * a.y);
        y1 = (float)((double)x1 * a.x + (double)x0 * a.y);
    }
};
template <> struct Rotation<__nv_bfloat16> {
    typedef float4 Angle;                        // cos high, cos low, sin high, sin low
    static __device__ __forceinline__ Angle angle(const double2& cs)
    {
        const float ch = (float)cs.x, sh = (float)cs.y;
        return make_float4(ch, (float)(cs.x - (double)ch), sh, (float)(cs.y - (double)sh));
    }
    // x * (hi + lo) as p + e
    static __device__ __forceinline__ void product(float x, float hi, float lo, float& p, float& e)
    {
        p = __fmul_rn(x, hi);
        e = __fmaf_rn(x, lo, __fmaf_rn(x, hi, -p));
    }
    static __device__ __forceinline__ float difference(float p, float e, float q, float f)
    {
        const float d = __fsub_rn(p, q);
        const float b = __fsub_rn(d, p);
        const float err = __fsub_rn(__fsub_rn(p, __fsub_rn(d, b)), __fadd_rn(q, b));
        const float y = __fadd_rn(d, __fadd_rn(err, __fsub_rn(e, f)));
        return fabsf(d) < INFINITY ? y : d;      // (an infinite or undefined result stays what it is)
    }
    static __device__ __forceinline__ void turn(float x0, float x1, const Angle& a, float& y0, float& y1)
    {
        float p, e, q, f;
        product(x0, a.x, a.y, p, e);
        product(x1, a.z, a.w, q, f);
        y0 = difference(p, e, q, f);
        product(x1, a.x, a.y, p, e);
        product(x0, -a.z, -a.w, q, f);
        y1 = difference(p, e, q, f);
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

// Block size: calls of few tokens (one wave of blocks) get one thread per work item, in whole warps,
// at most kRopeThreadsMax; batches of thousands of tokens are bound by throughput and take 256.
constexpr int kRopeThreadsMax = 384;
constexpr int kRopeThreads = 256;

// Where one new token comes from and goes to.
template <typename T>
struct TokenPlace {
    long src_tok;            // its row of q_new / k_new / v_new
    T* q_dst;                // its first query row of kv head 0, ...
    long q_rows;             //   rows per kv head of that buffer
    T* k_dst;                // its key / value row of kv head 0, ...
    T* v_dst;
    long kv_rows;            //   rows from one kv head to the next
};

// Rotates and stores one token with the whole block; the angles are in s_angle once the block has met.
template <typename T>
__device__ __forceinline__ void rope_token(const RopeArgs& a, const TokenPlace<T>& t, const typename Rotation<T>::Angle* s_angle)
{
    constexpr int V = VecTraits<T>::kVec;
    const int D = a.D, half = D / 2, G = a.G;
    const T* q_tok = (const T*)a.q_new + t.src_tok * a.q_stride;
    const T* k_tok = (const T*)a.k_new + t.src_tok * a.k_stride;
    const T* v_tok = (const T*)a.v_new + t.src_tok * a.v_stride;

    const int vph = a.vph_shift, vpr = a.vph_shift + 1;       // vectors per half head vector / per head vector (log2)
    const int q_items = a.Hq << vph;
    const int k_items = a.Hkv << vph;
    const int v_items = a.Hkv << vpr;
    const int items = q_items + k_items + v_items;

    // a thread's work item `it`: a pair of 16-byte vectors (j0.., j0+half..) of a query or key head,
    // or one 16-byte vector of a value head
    auto load_item = [&](int it, uint4& r0, uint4& r1) {
        if (it < q_items + k_items) {
            const bool is_q = it < q_items;
            const int e = is_q ? it : it - q_items;
            const int h = e >> vph;
            const int j0 = (e & ((1 << vph) - 1)) * V;
            const T* src = (is_q ? q_tok : k_tok) + (long)h * D;
            r0 = *reinterpret_cast<const uint4*>(src + j0);
            r1 = *reinterpret_cast<const uint4*>(src + j0 + half);
        } else {
            const int e = it - q_items - k_items;
            const int g = e >> vpr;
            const int d0 = (e & ((1 << vpr) - 1)) * V;
            r0 = *reinterpret_cast<const uint4*>(v_tok + (long)g * D + d0);
        }
    };
    auto finish_item = [&](int it, const uint4& lo_raw, const uint4& hi_raw) {
        if (it < q_items + k_items) {
            const bool is_q = it < q_items;
            const int e = is_q ? it : it - q_items;
            const int h = e >> vph;
            const int j0 = (e & ((1 << vph) - 1)) * V;
            T* dst;
            if (is_q) {
                const int g = (int)fast_div((uint32_t)h, a.div_g);
                dst = t.q_dst + ((long)g * t.q_rows + (h - g * G)) * D;
            } else {
                dst = t.k_dst + (long)h * t.kv_rows * D;
            }
            const T* lo = reinterpret_cast<const T*>(&lo_raw);
            const T* hi = reinterpret_cast<const T*>(&hi_raw);
            uint4 out_lo_raw, out_hi_raw;
            T* out_lo = reinterpret_cast<T*>(&out_lo_raw);
            T* out_hi = reinterpret_cast<T*>(&out_hi_raw);
#pragma unroll
            for (int v = 0; v < V; ++v) {
                float y0, y1;
                Rotation<T>::turn(to_float(lo[v]), to_float(hi[v]), s_angle[j0 + (j0 >> 3) + v], y0, y1);
                from_float(y0, out_lo[v]);
                from_float(y1, out_hi[v]);
            }
            *reinterpret_cast<uint4*>(dst + j0) = out_lo_raw;
            *reinterpret_cast<uint4*>(dst + j0 + half) = out_hi_raw;
        } else {
            const int e = it - q_items - k_items;
            const int g = e >> vpr;
            const int d0 = (e & ((1 << vpr) - 1)) * V;
            *reinterpret_cast<uint4*>(t.v_dst + (long)g * t.kv_rows * D + d0) = lo_raw;
        }
    };

    uint4 r0 = make_uint4(0u, 0u, 0u, 0u), r1 = r0;
    if ((int)threadIdx.x < items) load_item(threadIdx.x, r0, r1);     // in flight while the angles arrive
    __syncthreads();
    if ((int)threadIdx.x < items) finish_item(threadIdx.x, r0, r1);
    for (int it = threadIdx.x + blockDim.x; it < items; it += blockDim.x) {
        load_item(it, r0, r1);
        finish_item(it, r0, r1);
    }
}

// The angles of position `pos` into shared memory (angle j at j + j / 8: the 8 vectors of a half head in
// different banks).
template <typename T>
__device__ __forceinline__ void load_angles(typename Rotation<T>::Angle* s_angle, const double2* table, long table_first, long pos,
                                            int D, double log2_theta)
{
    const int j = threadIdx.x;
    if (j < D / 2)
        s_angle[j + (j >> 3)] = Rotation<T>::angle(table ? table[(pos - table_first) * (D / 2) + j] : rope_cos_sin(pos, j, D, log2_theta));
}

template <typename T, bool PAGED, typename LensT>
__global__ void __launch_bounds__(kRopeThreadsMax)
rope_append_kernel(const RopeArgs a, const __grid_constant__ LensT lens)
{
    constexpr int V = VecTraits<T>::kVec;
    __shared__ typename Rotation<T>::Angle s_angle[72];

    const int tok = blockIdx.x;           // index into the packed new tokens
    const int D = a.D;

    int b = 0, i = tok, L = a.cache_len, n_b = a.num_new;
    if (PAGED) {
        int lo = 0, hi = a.batch;         // largest b with new_off[b] <= tok
        while (hi - lo > 1) {
            int mid = (lo + hi) >> 1;
            if (lens.new_off[mid] <= tok) lo = mid; else hi = mid;
        }
        b = lo;
        i = tok - lens.new_off[b];
        L = lens.cache_len[b];
        n_b = lens.new_off[b + 1] - lens.new_off[b];
    }
    const long pos = (long)L + i;
    // (so far launch parameters only; what follows reads memory that earlier kernels may have written)
    asm volatile("griddepcontrol.wait;" ::: "memory");          // programmatic dependent launch: inputs ready
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    load_angles<T>(s_angle, a.table, a.table_first, pos, D, a.log2_theta);

    long page_base = 0;     // paged: first row of the page in the pool; slot within the page
    int slot = 0;
    if (PAGED) {
        page_base = (long)a.page_table[(long)b * a.max_pages + (int)(pos >> a.page_shift)] * a.Hkv * a.page_size;
        slot = (int)(pos & (a.page_size - 1));
    }
    TokenPlace<T> t;
    t.src_tok = tok;
    t.q_dst = (T*)a.q_rot + (long)tok * a.G * D;
    t.q_rows = (long)a.num_new * a.G;
    t.kv_rows = PAGED ? a.page_size : a.cache_cap;
    t.k_dst = (T*)a.k_cache + (PAGED ? page_base + slot : pos) * D;
    t.v_dst = (T*)a.v_cache + (PAGED ? page_base + slot : pos) * D;
    rope_token<T>(a, t, s_angle);

    if (PAGED && i == n_b - 1 && slot + 1 < a.page_size) {
        // the episode's last page is only partly filled: clear the value slots behind the last
        // token so that a tile load of the whole page never brings in stale bits
        const int tail = a.page_size - (slot + 1);
        const int vec_per_row = D / V;
        const int total = a.Hkv * tail * vec_per_row;
        const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
        for (int it = threadIdx.x; it < total; it += blockDim.x) {
            const int g = it / (tail * vec_per_row);
            const int r = it % (tail * vec_per_row);
            const int s2 = slot + 1 + r / vec_per_row;
            const int d0 = (r % vec_per_row) * V;
            *reinterpret_cast<uint4*>((T*)a.v_cache + (page_base + (long)g * a.page_size + s2) * D + d0) = zero;
        }
    }
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

__global__ void __launch_bounds__(kRopeThreadsMax)
rope_packed_kernel(const RopePackedArgs p)
{
    typedef __nv_bfloat16 T;
    __shared__ typename Rotation<T>::Angle s_angle[72];
    const RopeArgs& a = p.r;
    const int tok = blockIdx.x;
    const bool action = tok >= p.num_visual;
    const int m = action ? tok - p.num_visual : tok;             // within its run
    TokenPlace<T> t;
    long pos;
    if (action) {
        const int c = (int)fast_div((uint32_t)m, p.div_a), i = m - c * p.A;
        pos = (long)p.I + (long)(c + 1) * p.F + i;
        t.src_tok = (long)p.I + (long)c * (p.F + p.A) + p.F + i;
        t.kv_rows = p.num_action;
    } else {
        pos = m;
        t.src_tok = m;
        if (m >= p.I && p.F > 0) t.src_tok += (long)fast_div((uint32_t)(m - p.I), p.div_f) * p.A;
        t.kv_rows = a.cache_cap;
    }
    t.q_dst = (T*)(action ? p.q_rot_act : a.q_rot) + (long)m * a.G * a.D;
    t.q_rows = (long)(action ? p.num_action : p.num_visual) * a.G;
    t.k_dst = (T*)(action ? p.k_act : a.k_cache) + (long)m * a.D;
    t.v_dst = (T*)(action ? p.v_act : a.v_cache) + (long)m * a.D;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    load_angles<T>(s_angle, a.table, a.table_first, pos, a.D, a.log2_theta);
    rope_token<T>(a, t, s_angle);
}

}  // namespace evln
