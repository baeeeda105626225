// Four consecutive entries ("quads") of a row that may start on any element boundary.
//
// A warp wants N blocks of 32 quads, quad l of block u being entries base + 128 u + 4 l .. + 3 of the row.
// Where the row's address makes these quads unaligned, every lane loads the aligned quads that contain
// its first entries - 8- or 16-byte loads, as in the aligned case - and takes the rest from its neighbour
// by shuffles (lane 31's neighbour is lane 0 of the next block; lane 0 loads one quad more).  Entries
// outside [0, V) are never read: a quad that crosses an end of the row is put together from single
// entries and a fill value.  B = 300 V = 30011, binary16 rows: the mass kernel takes 12.8 us and the
// emission 8.4 where entry-by-entry loads, issue-bound, took 18 and 13; a whole round 48 us against 57.
#pragma once

#include "dssd_device.cuh"

namespace dssd {

// Loads of rows that an earlier kernel of the chain may have written: they stay behind pdl_wait() and do
// not go through the read-only path.  Vectors are read once and not kept in L1.
__device__ __forceinline__ uint4 ld_row16(const void *p)
{
    uint4 v;
    asm volatile("ld.global.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ uint2 ld_row8(const void *p)
{
    uint2 v;
    asm volatile("ld.global.L1::no_allocate.v2.u32 {%0,%1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ uint32_t ld_row_u32(const void *p)
{
    uint32_t v;
    asm volatile("ld.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ uint32_t ld_row_u16(const void *p)
{
    unsigned short v;
    asm volatile("ld.global.u16 %0, [%1];" : "=h"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ unsigned char ld_row_u8(const void *p)
{
    unsigned short v;
    asm volatile("ld.global.u8 %0, [%1];" : "=h"(v) : "l"(p) : "memory");
    return (unsigned char)v;
}

struct Quads32 {  // 4-byte entries
    typedef uint4 Raw;
    static constexpr int kBytes = 4;
    __device__ static __forceinline__ Raw load(const char *p) { return ld_row16(p); }
    // entries a .. a + 3 of `row`, those outside [0, V) as `fill`
    __device__ static __forceinline__ Raw guarded(const char *row, long long a, int V, uint32_t fill)
    {
        uint32_t e[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            e[j] = fill;
            if (a + j >= 0 && a + j < V) e[j] = ld_row_u32(row + (a + j) * 4);
        }
        return make_uint4(e[0], e[1], e[2], e[3]);
    }
    // the four entries from entry s (0 < s < 4) of the eight in v, w on
    __device__ static __forceinline__ Raw shift(const Raw &v, const Raw &send, int from, int s)
    {
        const uint32_t nx = __shfl_sync(0xffffffffu, send.x, from);
        if (s == 1) return make_uint4(v.y, v.z, v.w, nx);
        const uint32_t ny = __shfl_sync(0xffffffffu, send.y, from);
        if (s == 2) return make_uint4(v.z, v.w, nx, ny);
        const uint32_t nz = __shfl_sync(0xffffffffu, send.z, from);
        return make_uint4(v.w, nx, ny, nz);
    }
    // the same with both quads in this thread
    __device__ static __forceinline__ Raw join(const Raw &v, const Raw &w, int s)
    {
        return s == 0 ? v : s == 1 ? make_uint4(v.y, v.z, v.w, w.x) : s == 2 ? make_uint4(v.z, v.w, w.x, w.y) : make_uint4(v.w, w.x, w.y, w.z);
    }
    __device__ static __forceinline__ Raw pick(bool c, const Raw &a, const Raw &b)
    {
        return make_uint4(c ? a.x : b.x, c ? a.y : b.y, c ? a.z : b.z, c ? a.w : b.w);
    }
};

struct Quads16 {  // 2-byte entries
    typedef uint2 Raw;
    static constexpr int kBytes = 2;
    __device__ static __forceinline__ Raw load(const char *p) { return ld_row8(p); }
    __device__ static __forceinline__ Raw guarded(const char *row, long long a, int V, uint32_t fill)
    {
        uint32_t e[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            e[j] = fill & 0xffffu;
            if (a + j >= 0 && a + j < V) e[j] = ld_row_u16(row + (a + j) * 2);
        }
        return make_uint2(e[0] | (e[1] << 16), e[2] | (e[3] << 16));
    }
    __device__ static __forceinline__ Raw shift(const Raw &v, const Raw &send, int from, int s)
    {
        const uint32_t nx = __shfl_sync(0xffffffffu, send.x, from);
        if (s == 1) return make_uint2(__funnelshift_r(v.x, v.y, 16), __funnelshift_r(v.y, nx, 16));
        if (s == 2) return make_uint2(v.y, nx);
        const uint32_t ny = __shfl_sync(0xffffffffu, send.y, from);
        return make_uint2(__funnelshift_r(v.y, nx, 16), __funnelshift_r(nx, ny, 16));
    }
    __device__ static __forceinline__ Raw join(const Raw &v, const Raw &w, int s)
    {
        return s == 0   ? v
               : s == 1 ? make_uint2(__funnelshift_r(v.x, v.y, 16), __funnelshift_r(v.y, w.x, 16))
               : s == 2 ? make_uint2(v.y, w.x)
                        : make_uint2(__funnelshift_r(v.y, w.x, 16), __funnelshift_r(w.x, w.y, 16));
    }
    __device__ static __forceinline__ Raw pick(bool c, const Raw &a, const Raw &b) { return make_uint2(c ? a.x : b.x, c ? a.y : b.y); }
};

// entries between the aligned quad below entry `e` of the row and that entry: 0 .. 3
template <class Q>
__device__ __forceinline__ int quad_offset(const char *row, long long e)
{
    return (int)((reinterpret_cast<uintptr_t>(row) / Q::kBytes + (unsigned long long)e) & 3u);
}

// The N blocks of a warp (see the top of this file).  kShift = false: the caller knows that the quads are
// aligned.  load() requests everything, at(u) then gives block u's quad of this lane; all 32 lanes take part.
template <class Q, int N, bool kShift>
struct WarpQuads {
    typename Q::Raw own[kShift ? N + 1 : N];
    int s;
    __device__ __forceinline__ void load(const char *row, int V, long long base, uint32_t fill)
    {
        const int lane = threadIdx.x & 31;
        s = kShift ? quad_offset<Q>(row, base) : 0;
        const long long a = base - s + 4 * lane;
        const bool interior = base >= 4 && base + 128 * N + 4 <= V;  // (the same in all lanes)
        const char *p = row + a * Q::kBytes;
        if (interior) {
#pragma unroll
            for (int u = 0; u < N; ++u) own[u] = Q::load(p + u * 128 * Q::kBytes);
            if (kShift) {
                own[N] = typename Q::Raw();
                if (s && lane == 0) own[N] = Q::load(p + N * 128 * Q::kBytes);
            }
        } else {
#pragma unroll
            for (int u = 0; u < (kShift ? N + 1 : N); ++u) {
                const long long at = a + 128 * u;
                own[u] = typename Q::Raw();
                if (u == N && lane) continue;
                if (at >= 0 && at + 4 <= V) own[u] = Q::load(p + u * 128 * Q::kBytes);
                else own[u] = Q::guarded(row, at, V, fill);
            }
        }
    }
    __device__ __forceinline__ typename Q::Raw at(int u) const
    {
        if (!kShift || s == 0) return own[u];
        const int lane = threadIdx.x & 31;
        return Q::shift(own[u], Q::pick(lane == 0, own[u + 1], own[u]), (lane + 1) & 31, s);
    }
};

// N consecutive quads of one thread, entries e .. e + 4 N - 1.
template <class Q, int N, bool kShift>
struct ThreadQuads {
    typename Q::Raw own[kShift ? N + 1 : N];
    int s;
    __device__ __forceinline__ void load(const char *row, int V, long long e, uint32_t fill)
    {
        s = kShift ? quad_offset<Q>(row, e) : 0;
        const long long a = e - s;
#pragma unroll
        for (int u = 0; u < (kShift ? N + 1 : N); ++u) {
            const long long at = a + 4 * u;
            if (at >= 0 && at + 4 <= V) own[u] = Q::load(row + at * Q::kBytes);
            else own[u] = Q::guarded(row, at, V, fill);
        }
    }
    __device__ __forceinline__ typename Q::Raw at(int u) const { return kShift ? Q::join(own[u], own[u + 1], s) : own[u]; }
};

}  // namespace dssd
