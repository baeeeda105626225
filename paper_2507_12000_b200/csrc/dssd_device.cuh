// Device-side helpers shared by the verification kernels (sm_100a).
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "dssd.h"

namespace dssd {

constexpr int kThreads = 256;           // threads per CTA in every kernel
constexpr int kWarps = kThreads / 32;
#define DSSD_NEG_INF (__int_as_float(0xff800000))

// ---- memory ------------------------------------------------------------------------------

// 16-byte streaming load of data that no one writes during the kernel; does not allocate in L1.
__device__ __forceinline__ uint4 ld_stream16(const void *p)
{
    uint4 v;
    asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p));
    return v;
}

// two floats rounded to IEEE binary16 (nearest even), low half = first
__device__ __forceinline__ uint32_t pack_half2(float lo, float hi)
{
    const __half2 h = __floats2half2_rn(lo, hi);
    return *reinterpret_cast<const uint32_t *>(&h);
}

__device__ __forceinline__ unsigned short to_half_bits(float x) { return __half_as_ushort(__float2half_rn(x)); }

// ---- programmatic dependent launch (see launch.h) -----------------------------------------------

// everything the kernels before this one wrote is visible after it
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// the next kernel's CTAs may be scheduled once every CTA of this one has said so (or has ended)
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// ---- thread-block clusters ---------------------------------------------------------------------

__device__ __forceinline__ unsigned cluster_rank()
{
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// every thread of every CTA of the cluster arrives once per phase; what was stored before an arrival, in
// any CTA's shared memory, is visible after the wait.  Both want the warp's threads together, which after divergent code is
// not to be had without saying so.
__device__ __forceinline__ void cluster_arrive()
{
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait()
{
    __syncwarp();
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// stores to the variable at the same place in the shared memory of the cluster's CTA `rank`
__device__ __forceinline__ uint32_t cluster_addr(const void *p, unsigned rank)
{
    uint32_t a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
    return a;
}
__device__ __forceinline__ void cluster_store(double *p, unsigned rank, double v)
{
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(cluster_addr(p, rank)), "d"(v) : "memory");
}

__device__ __forceinline__ void cluster_store(unsigned long long *p, unsigned rank, unsigned long long v)
{
    asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(cluster_addr(p, rank)), "l"(v) : "memory");
}

// Scalar loads that stay behind pdl_wait() (a plain __ldg may be moved across it), served by L2.
__device__ __forceinline__ uint32_t ld_after_u32(const void *p)
{
    uint32_t v;
    asm volatile("ld.global.cg.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ int ld_after(const int32_t *p) { return (int)ld_after_u32(p); }
__device__ __forceinline__ float ld_after(const float *p) { return __uint_as_float(ld_after_u32(p)); }
__device__ __forceinline__ unsigned long long ld_after(const unsigned long long *p)
{
    unsigned long long v;
    asm volatile("ld.global.cg.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ double ld_after(const double *p)
{
    return __longlong_as_double((long long)ld_after(reinterpret_cast<const unsigned long long *>(p)));
}

// ---- arithmetic --------------------------------------------------------------------------

// 2^x on the special-function unit (max relative error about 2^-22; -inf -> 0, NaN -> NaN).
__device__ __forceinline__ float ex2(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// elementwise maximum of two packed bfloat16 pairs (a NaN element yields the other operand)
__device__ __forceinline__ uint32_t max_bf16x2(uint32_t a, uint32_t b)
{
    uint32_t d;
    asm("max.bf16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
    return d;
}

// ---- packed pairs of float32 (sm_100: one instruction works on both halves) ---------------------

typedef unsigned long long f32x2;

__device__ __forceinline__ f32x2 pack2(float lo, float hi)
{
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}

__device__ __forceinline__ void unpack2(f32x2 v, float &lo, float &hi)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}

__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c)
{
    f32x2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b)
{
    f32x2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b)
{
    f32x2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

__device__ __forceinline__ float bf16_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }

template <int DT>
struct Elem;
template <>
struct Elem<DSSD_F32> {
    static constexpr int kBytes = 4;
    __device__ static __forceinline__ float load(const void *row, int64_t i)
    {
        float f;
        asm volatile("ld.global.nc.f32 %0, [%1];" : "=f"(f) : "l"(reinterpret_cast<const float *>(row) + i));
        return f;
    }
};
template <>
struct Elem<DSSD_BF16> {
    static constexpr int kBytes = 2;
    __device__ static __forceinline__ float load(const void *row, int64_t i)
    {
        unsigned short h;
        asm volatile("ld.global.nc.u16 %0, [%1];" : "=h"(h) : "l"(reinterpret_cast<const unsigned short *>(row) + i));
        return __uint_as_float((uint32_t)h << 16);
    }
};

__device__ __forceinline__ double warp_sum(double x)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}

__device__ __forceinline__ float warp_max(float x)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x = fmaxf(x, __shfl_xor_sync(0xffffffffu, x, o));
    return x;
}

__device__ __forceinline__ float warp_sum(float x)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}

}  // namespace dssd
