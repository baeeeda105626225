// Emission of a row of probabilities, a tile per CTA: shared by the dense and the vocabulary-sharded edge.
#pragma once

#include "dssd_device.cuh"
#include "quads.cuh"

namespace dssd {

constexpr int kEmitTile = 8192;  // entries that one CTA emits

// do the logits and the output rows all start on boundaries of four entries?
inline bool emit_aligned(const void *logits, int64_t row_stride, int esz, const void *out, int64_t out_stride, int osz)
{
    return out_stride % 4 == 0 && reinterpret_cast<uintptr_t>(out) % (4 * osz) == 0 && row_stride % 4 == 0 &&
           reinterpret_cast<uintptr_t>(logits) % (4 * esz) == 0;
}
// tiles of a row (an unaligned row's first tile starts up to three entries before it)
inline int emit_tiles(int V, bool aligned) { return (int)(((long long)V + (aligned ? 0 : 3) + kEmitTile - 1) / kEmitTile); }

// default stores: the rows written last are still in L2 when the draw reads them
__device__ __forceinline__ void store_quad(float *o, float a, float b, float c, float d)
{
    *reinterpret_cast<float4 *>(o) = make_float4(a, b, c, d);
}
__device__ __forceinline__ void store_quad(uint16_t *o, float a, float b, float c, float d)
{
    *reinterpret_cast<uint2 *>(o) = make_uint2(pack_half2(a, b), pack_half2(c, d));
}
__device__ __forceinline__ void store_one(float *o, float a) { *o = a; }
__device__ __forceinline__ void store_one(uint16_t *o, float a) { *o = to_half_bits(a); }

// out[0..3] = 2^(z * c1 - ref2) * invS for four logits, as two packed pairs
template <class OUT>
__device__ __forceinline__ void emit_quad(OUT *out, float z0, float z1, float z2, float z3, f32x2 cc, f32x2 nn, f32x2 ss)
{
    float a, b, c, d;
    unpack2(fma2(pack2(z0, z1), cc, nn), a, b);
    unpack2(fma2(pack2(z2, z3), cc, nn), c, d);
    unpack2(mul2(pack2(ex2(a), ex2(b)), ss), a, b);
    unpack2(mul2(pack2(ex2(c), ex2(d)), ss), c, d);
    store_quad(out, a, b, c, d);
}

__device__ __forceinline__ void emit_raw(float *out, const uint2 &w, f32x2 cc, f32x2 nn, f32x2 ss)
{
    emit_quad(out, bf16_lo(w.x), bf16_hi(w.x), bf16_lo(w.y), bf16_hi(w.y), cc, nn, ss);
}
__device__ __forceinline__ void emit_raw(uint16_t *out, const uint2 &w, f32x2 cc, f32x2 nn, f32x2 ss)
{
    emit_quad(out, bf16_lo(w.x), bf16_hi(w.x), bf16_lo(w.y), bf16_hi(w.y), cc, nn, ss);
}
template <class OUT>
__device__ __forceinline__ void emit_raw(OUT *out, const uint4 &w, f32x2 cc, f32x2 nn, f32x2 ss)
{
    emit_quad(out, __uint_as_float(w.x), __uint_as_float(w.y), __uint_as_float(w.z), __uint_as_float(w.w), cc, nn, ss);
}

template <class OUT>
struct OutQuads {
    typedef Quads32 Q;
};
template <>
struct OutQuads<uint16_t> {
    typedef Quads16 Q;
};
template <int DT>
struct LogitQuads {
    typedef Quads32 Q;
};
template <>
struct LogitQuads<DSSD_BF16> {
    typedef Quads16 Q;
};

// entries of the quad that crosses the start of an unaligned output row and lie before it
template <class OUT>
__device__ __forceinline__ int emit_lead(const OUT *outp)
{
    return quad_offset<typename OutQuads<OUT>::Q>(reinterpret_cast<const char *>(outp), 0);
}

// outp[e] = 2^(l_e * c1 - ref2) * invS for the 128 kN entries from `base` on that lie in a row of V entries, by a warp.
// `base` is where the output's quads are aligned; the logits' quads may lie on any element
// boundary (quads.cuh).  All of a thread's loads are requested before the first is used.
template <int DT, bool kShift, int kN, class OUT>
__device__ __forceinline__ void emit_piece(const char *rowp, OUT *outp, int V, long long base, float c1, float ref2, float invS)
{
    using Q = typename LogitQuads<DT>::Q;
    const int lane = threadIdx.x & 31;
    const float nref = -ref2;
    const f32x2 cc = pack2(c1, c1), nn = pack2(nref, nref), ss = pack2(invS, invS);
    WarpQuads<Q, kN, kShift> w;
    w.load(rowp, V, base, 0u);
#pragma unroll
    for (int u = 0; u < kN; ++u) {
        const typename Q::Raw v = w.at(u);
        const long long e = base + 128 * u + 4 * lane;
        if (e >= 0 && e + 4 <= V) {
            emit_raw(outp + e, v, cc, nn, ss);
        } else if (e + 4 > 0 && e < V) {  // a quad that crosses an end of the row
            for (int j = 0; j < 4; ++j)
                if (e + j >= 0 && e + j < V) store_one(outp + e + j, ex2(fmaf(Elem<DT>::load(rowp, e + j), c1, nref)) * invS);
        }
    }
}

// One tile of a row by a CTA of kThreads threads.
template <int DT, bool kShift, class OUT>
__device__ __forceinline__ void emit_tile(const char *rowp, OUT *outp, int V, int tile, float c1, float ref2, float invS)
{
    constexpr int kN = kEmitTile / 4 / kThreads;
    const long long e0 = (long long)tile * kEmitTile - (kShift ? emit_lead(outp) : 0);
    emit_piece<DT, kShift, kN>(rowp, outp, V, e0 + (int)(threadIdx.x >> 5) * (128 * kN), c1, ref2, invS);
}

}  // namespace dssd
