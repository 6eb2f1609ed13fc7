// ns_mem.cuh -- loads and stores with L2 cache policies, shared by the execute kernels.
#pragma once
#include <type_traits>

#include "ns_internal.cuh"

namespace ns {

// ---------------------------------------------------------------------------------------------
// memory helpers with L2 cache policies
// ---------------------------------------------------------------------------------------------
struct Policies {
    uint64_t first, last;
};

__device__ __forceinline__ Policies make_policies()
{
    Policies p;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p.first));
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p.last));
    return p;
}

template <bool HINT>
__device__ __forceinline__ int32_t ld_stream_i32(const int32_t* p, uint64_t pol)
{
    int32_t v;
    if (HINT)
        asm volatile("ld.global.nc.L1::no_allocate.L2::cache_hint.b32 %0, [%1], %2;"
                     : "=r"(v) : "l"(p), "l"(pol));
    else
        v = __ldg(p);
    return v;
}

template <bool HINT>
__device__ __forceinline__ float ld_stream_f32(const float* p, uint64_t pol)
{
    float v;
    if (HINT)
        asm volatile("ld.global.nc.L1::no_allocate.L2::cache_hint.f32 %0, [%1], %2;"
                     : "=f"(v) : "l"(p), "l"(pol));
    else
        v = __ldg(p);
    return v;
}

// Four consecutive B elements as loaded: 16 B of FP32 or 8 B of BF16.  Rings of gathers keep
// this raw form and widen a vector only where it is used: a conversion next to its load would
// wait for the load there and leave one gather in flight instead of the ring's depth.
template <bool BF16>
using BRaw = std::conditional_t<BF16, uint2, float4>;

template <bool BF16, bool HINT>
__device__ __forceinline__ BRaw<BF16> ld_braw(const void* p, uint64_t pol)
{
    BRaw<BF16> r;
    if constexpr (!BF16) {
        if (HINT)
            asm volatile("ld.global.nc.L2::cache_hint.v4.f32 {%0,%1,%2,%3}, [%4], %5;"
                         : "=f"(r.x), "=f"(r.y), "=f"(r.z), "=f"(r.w) : "l"(p), "l"(pol));
        else
            r = __ldg(reinterpret_cast<const float4*>(p));
    } else {
        if (HINT)
            asm volatile("ld.global.nc.L2::cache_hint.v2.b32 {%0,%1}, [%2], %3;"
                         : "=r"(r.x), "=r"(r.y) : "l"(p), "l"(pol));
        else
            r = __ldg(reinterpret_cast<const uint2*>(p));
    }
    return r;
}

template <bool BF16>
__device__ __forceinline__ BRaw<BF16> braw_zero()
{
    if constexpr (BF16) return make_uint2(0u, 0u);
    else return make_float4(0.f, 0.f, 0.f, 0.f);
}

__device__ __forceinline__ float4 widen(const float4& v) { return v; }
__device__ __forceinline__ float4 widen(const uint2& v)  // BF16 is the high half of an FP32
{
    return make_float4(__uint_as_float(v.x << 16), __uint_as_float(v.x & 0xffff0000u),
                       __uint_as_float(v.y << 16), __uint_as_float(v.y & 0xffff0000u));
}

template <bool HINT>
__device__ __forceinline__ void st_c4(float* p, float4 v, uint64_t pol)
{
    if (HINT)
        asm volatile("st.global.L2::cache_hint.v4.f32 [%0], {%1,%2,%3,%4}, %5;"
                     :: "l"(p), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w), "l"(pol) : "memory");
    else
        *reinterpret_cast<float4*>(p) = v;
}

__device__ __forceinline__ float4 f4_fma(float a, float4 b, float4 c)
{
    c.x = fmaf(a, b.x, c.x);
    c.y = fmaf(a, b.y, c.y);
    c.z = fmaf(a, b.z, c.z);
    c.w = fmaf(a, b.w, c.w);
    return c;
}
__device__ __forceinline__ float4 f4_add(float4 a, float4 b)
{
    return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w);
}

// ---- BF16 pieces of FP32 values ----
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi)  // round to nearest even
{
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}

// The three BF16 pieces of two values, each pair packed (first value low): x = x0 + x1 + x2 with x0
// truncated (it never overflows) and x1, x2 rounded to nearest.
__device__ __forceinline__ void split3(float x, float y, uint32_t& p0, uint32_t& p1, uint32_t& p2)
{
    const uint32_t xi = __float_as_uint(x), yi = __float_as_uint(y);
    p0 = __byte_perm(xi, yi, 0x7632);
    x -= __uint_as_float(xi & 0xffff0000u);
    y -= __uint_as_float(yi & 0xffff0000u);
    p1 = pack_bf16(x, y);
    x -= __uint_as_float(p1 << 16);
    y -= __uint_as_float(p1 & 0xffff0000u);
    p2 = pack_bf16(x, y);
}

// The end of a persistent launch, called by the whole CTA: the last CTA out resets the tickets for the
// next launch (stream order makes it visible) and reports a nonzero status word to the host.  A
// copy and an event after every launch did that before, two calls and a copy engine's turn: 13.5 ->
// 9.2 us for an execute of 65 536 nonzeros at K = 32, 110.5 -> 105.1 us for the attention mask's.
__device__ __forceinline__ void end_launch(int32_t* ctrl, const ExecDesc& d0, bool single)
{
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        const int done = atomicAdd(ctrl + 1, 1);
        if (done == (int)gridDim.x - 1) {
            atomicExch(ctrl + 0, 0);
            atomicExch(ctrl + 3, 0);
            atomicExch(reinterpret_cast<unsigned long long*>(ctrl + 4), 0ull);
            atomicExch(ctrl + 1, 0);
            if (single && d0.status_out) {
                const int32_t st = atomicOr(d0.status, 0);
                if (st) *reinterpret_cast<volatile int32_t*>(d0.status_out) = st;
            }
        }
    }
}

}  // namespace ns
