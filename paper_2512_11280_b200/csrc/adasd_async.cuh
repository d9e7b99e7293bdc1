// Asynchronous building blocks for sm_100a shared by the streaming kernels: cluster-scope
// mbarrier and st.async wrappers, tensor memory as a scratchpad, 16-byte units of a row.
#pragma once

#include "adasd_cluster.cuh"
#include "adasd_pdl.cuh"

namespace adasd {

// ---- mbarriers and DSMEM -----------------------------------------------------------------
__device__ __forceinline__ void mbar_arrive_cta(uint64_t* bar) {
    asm volatile("mbarrier.arrive.release.cta.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// shared::cluster address of `p` (an address in this CTA's shared memory) as seen in CTA `cta`
__device__ __forceinline__ uint32_t mapa_u32(const void* p, uint32_t cta) {
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_u32(p)), "r"(cta));
    return r;
}
// 16 bytes into another CTA's shared memory; their arrival is counted (complete_tx) on a
// barrier of THAT CTA, so the receiver needs no fence and the sender no second message
__device__ __forceinline__ void st_async_v4(uint32_t remote_addr, float4 v, uint32_t remote_bar) {
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];"
                 ::"r"(remote_addr), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w), "r"(remote_bar)
                 : "memory");
}

// ---- tensor memory as a scratchpad ---------------------------------------------------------
// Allocation and release are warp-wide; the address lands in shared memory.
__device__ __forceinline__ void tmem_alloc(uint32_t* smem_dst, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(smem_dst)), "r"(ncols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
// Loads are asynchronous: the registers hold the values only after tmem_wait_ld, which
// takes them as operands so that nothing that uses them can be scheduled ahead of the wait.
__device__ __forceinline__ void tmem_wait_ld(float (&a)[8], float (&b)[8]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+f"(a[0]), "+f"(a[1]), "+f"(a[2]), "+f"(a[3]), "+f"(a[4]), "+f"(a[5]), "+f"(a[6]), "+f"(a[7]),
                   "+f"(b[0]), "+f"(b[1]), "+f"(b[2]), "+f"(b[3]), "+f"(b[4]), "+f"(b[5]), "+f"(b[6]), "+f"(b[7])
                 :
                 : "memory");
}
// {x, x} as an operand of packed arithmetic, kept in its register pair: a pair the compiler can see through
// is made again at its uses, up to two moves for each packed instruction.
__device__ __forceinline__ float2 pair2(float x) {
    float2 r = make_float2(x, x);
    asm volatile("" : "+f"(r.x), "+f"(r.y));
    return r;
}

__device__ __forceinline__ float rcp_approx(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ double warp_sum_f64(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    return v;
}

// ---- 16-byte units of a logit row ----------------------------------------------------------
// A row is cut into units of 16 bytes that are ALIGNED IN MEMORY, whatever the row's own address:
// a row that starts m elements past a 16-byte boundary has unit u = its elements u N - m ..
// u N - m + N - 1, and the elements before its start and past its end read as -inf.  Per type: N
// elements a unit, packed maximum with NaN kept, the cut of an adjusted distribution (to -inf), unpacking to fp32 with -inf (and NaN) clamped to a finite floor
// (unpack_raw: not clamped, for sums in which no product with a -inf occurs).
template <typename T>
struct Unit;

template <>
struct Unit<__nv_bfloat16> {
    static constexpr int N = 8;
    using Max = uint32_t;                     // packed pair
    static __device__ __forceinline__ Max max0() { return 0xFF80FF80u; }
    static __device__ __forceinline__ void max_add(Max& m, const uint4& w) {
        m = bmax2(bmax2(m, w.x), bmax2(w.y, bmax2(w.z, w.w)));
    }
    // largest element of a unit (NaN kept), and as one number (NaN dropped)
    static __device__ __forceinline__ Max unit_max(const uint4& w) { return bmax2(bmax2(w.x, w.y), bmax2(w.z, w.w)); }
    static __device__ __forceinline__ void max_join(Max& m, Max h) { m = bmax2(m, h); }
    static __device__ __forceinline__ float top(Max h) {
        const float2 v = unpack2(h);
        return fmaxf(v.x, v.y);
    }
    static __device__ __forceinline__ float max_val(Max m, uint32_t& bad) {
        const float2 v = unpack2(m);
        if (v.x != v.x || v.y != v.y) bad = 1u;
        return fmaxf(v.x, v.y);
    }
    using Cut = uint32_t;
    static __device__ __forceinline__ Cut make_cut(float c) { return cut_pair(c); }
    static __device__ __forceinline__ uint32_t cut2(uint32_t a, uint32_t c) {
        uint32_t m;
        asm("set.lt.u32.bf16x2 %0, %1, %2;" : "=r"(m) : "r"(a), "r"(c));   // 0xFFFF per half that is below; a NaN is not
        return (a & ~m) | (0xFF80FF80u & m);
    }
    static __device__ __forceinline__ void cut(uint4& w, Cut c) {
        w = make_uint4(cut2(w.x, c), cut2(w.y, c), cut2(w.z, c), cut2(w.w, c));
    }
    static __device__ __forceinline__ uint4 none4() { return make_uint4(0xFF80FF80u, 0xFF80FF80u, 0xFF80FF80u, 0xFF80FF80u); }
    // elements outside [lo, hi) of the unit become -inf
    static __device__ __forceinline__ void mask(uint4& w, int lo, int hi) {
        uint32_t* p = &w.x;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (2 * j < lo || 2 * j >= hi) p[j] = (p[j] & 0xFFFF0000u) | 0xFF80u;
            if (2 * j + 1 < lo || 2 * j + 1 >= hi) p[j] = (p[j] & 0xFFFFu) | 0xFF800000u;
        }
    }
    static __device__ __forceinline__ void unpack(const uint4& w, float2 (&z)[4]) {
        z[0] = unpack2(bclamp2(w.x));
        z[1] = unpack2(bclamp2(w.y));
        z[2] = unpack2(bclamp2(w.z));
        z[3] = unpack2(bclamp2(w.w));
    }
    static __device__ __forceinline__ void unpack_raw(const uint4& w, float2 (&z)[4]) {
        z[0] = unpack2(w.x);
        z[1] = unpack2(w.y);
        z[2] = unpack2(w.z);
        z[3] = unpack2(w.w);
    }
    // the unit that starts s elements into the 32 bytes a|b
    static __device__ __forceinline__ uint4 realign(const uint4& a, const uint4& b, int s) {
        uint32_t x0 = a.x, x1 = a.y, x2 = a.z, x3 = a.w, x4 = b.x, x5 = b.y, x6 = b.z;
        if (s & 4) { x0 = x2; x1 = x3; x2 = x4; x3 = x5; x4 = x6; x5 = b.w; x6 = 0u; }
        if (s & 2) { x0 = x1; x1 = x2; x2 = x3; x3 = x4; x4 = x5; }
        const uint32_t sh = (s & 1) * 16;
        return make_uint4(__funnelshift_r(x0, x1, sh), __funnelshift_r(x1, x2, sh), __funnelshift_r(x2, x3, sh),
                          __funnelshift_r(x3, x4, sh));
    }
};

template <>
struct Unit<float> {
    static constexpr int N = 4;
    using Max = float;
    static __device__ __forceinline__ Max max0() { return -INFINITY; }
    static __device__ __forceinline__ float fmax_nan(float a, float b) {
        float d;
        asm("max.NaN.f32 %0, %1, %2;" : "=f"(d) : "f"(a), "f"(b));
        return d;
    }
    static __device__ __forceinline__ void max_add(Max& m, const uint4& w) {
        m = fmax_nan(fmax_nan(m, __uint_as_float(w.x)),
                     fmax_nan(__uint_as_float(w.y), fmax_nan(__uint_as_float(w.z), __uint_as_float(w.w))));
    }
    static __device__ __forceinline__ Max unit_max(const uint4& w) {
        return fmax_nan(fmax_nan(__uint_as_float(w.x), __uint_as_float(w.y)), fmax_nan(__uint_as_float(w.z), __uint_as_float(w.w)));
    }
    static __device__ __forceinline__ void max_join(Max& m, Max h) { m = fmax_nan(m, h); }
    static __device__ __forceinline__ float top(Max h) { return h; }
    static __device__ __forceinline__ float max_val(Max m, uint32_t& bad) {
        if (m != m) bad = 1u;
        return m;
    }
    using Cut = float;
    static __device__ __forceinline__ Cut make_cut(float c) { return c; }
    static __device__ __forceinline__ uint32_t cut1(uint32_t w, float c) {
        return __uint_as_float(w) < c ? 0xFF800000u : w;
    }
    static __device__ __forceinline__ void cut(uint4& w, Cut c) {
        w = make_uint4(cut1(w.x, c), cut1(w.y, c), cut1(w.z, c), cut1(w.w, c));
    }
    static __device__ __forceinline__ uint4 none4() { return make_uint4(0xFF800000u, 0xFF800000u, 0xFF800000u, 0xFF800000u); }
    static __device__ __forceinline__ void mask(uint4& w, int lo, int hi) {
        uint32_t* p = &w.x;
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (j < lo || j >= hi) p[j] = 0xFF800000u;
    }
    static __device__ __forceinline__ void unpack(const uint4& w, float2 (&z)[2]) {
        z[0] = make_float2(fmaxf(__uint_as_float(w.x), kFloor), fmaxf(__uint_as_float(w.y), kFloor));
        z[1] = make_float2(fmaxf(__uint_as_float(w.z), kFloor), fmaxf(__uint_as_float(w.w), kFloor));
    }
    static __device__ __forceinline__ void unpack_raw(const uint4& w, float2 (&z)[2]) {
        z[0] = make_float2(__uint_as_float(w.x), __uint_as_float(w.y));
        z[1] = make_float2(__uint_as_float(w.z), __uint_as_float(w.w));
    }
    static __device__ __forceinline__ uint4 realign(const uint4& a, const uint4& b, int s) {
        uint32_t x0 = a.x, x1 = a.y, x2 = a.z, x3 = a.w, x4 = b.x, x5 = b.y;
        if (s & 2) { x0 = x2; x1 = x3; x2 = x4; x3 = x5; x4 = b.z; }
        if (s & 1) { x0 = x1; x1 = x2; x2 = x3; x3 = x4; }
        return make_uint4(x0, x1, x2, x3);
    }
};

}  // namespace adasd
