// The parts of a draw that its kernels share: the rows as float32, binary16 or logits, the sums of a
// segment's residuals, the pick of the segment that holds the target, the walk inside it.
#pragma once

#include <math.h>

#include "dssd_device.cuh"
#include "edge_verify.h"
#include "quads.cuh"

namespace dssd {

constexpr int kKeep = 8;  // chunk sums that a lane keeps: enough for 256 chunks without a second look

__device__ __forceinline__ double res(float p, float q) { return fmax(0.0, (double)p - (double)q); }

__device__ __forceinline__ float4 as_f4(const uint4 &v)
{
    return make_float4(__uint_as_float(v.x), __uint_as_float(v.y), __uint_as_float(v.z), __uint_as_float(v.w));
}

// The row p comes as float32, as IEEE binary16 bit patterns (the 16-bit payload), or - for the
// fused verification of Algorithm 1, where no row is ever written - as the target logits of row n
// together with the row's reference exponent and 1 / sum, from which p_v = 2^(l_v c1 - ref2) / S is
// formed on the fly exactly as the edge kernel forms it when it emits a row.  The kernel is
// written once over these views.  A "quad" is four consecutive entries.
__device__ __forceinline__ float4 half_quad(uint2 v)
{
    const float2 a = __half22float2(*reinterpret_cast<const __half2 *>(&v.x));
    const float2 b = __half22float2(*reinterpret_cast<const __half2 *>(&v.y));
    return make_float4(a.x, a.y, b.x, b.y);
}
struct RowF32 {  // p_row as float32
    typedef Quads32 Q;
    static constexpr uint32_t kFill = 0u;
    static constexpr bool kFixed = true;  // the row does not depend on the accepted length
    const char *row;
    template <class Params>
    __device__ static __forceinline__ RowF32 make(const Params &P, int64_t b, int)
    {
        RowF32 r;
        r.row = static_cast<const char *>(P.p_row) + (size_t)b * P.V * 4;
        return r;
    }
    __device__ __forceinline__ float4 quad(const Q::Raw &v) const { return as_f4(v); }
};

struct RowF16 {  // p_row as binary16 bit patterns
    typedef Quads16 Q;
    static constexpr uint32_t kFill = 0u;
    static constexpr bool kFixed = true;  // the row does not depend on the accepted length
    const char *row;
    template <class Params>
    __device__ static __forceinline__ RowF16 make(const Params &P, int64_t b, int)
    {
        RowF16 r;
        r.row = static_cast<const char *>(P.p_row) + (size_t)b * P.V * 2;
        return r;
    }
    __device__ __forceinline__ float4 quad(const Q::Raw &v) const { return half_quad(v); }
};

// four consecutive logits: how they are loaded and widened
template <int DT>
struct LogitQuad;
template <>
struct LogitQuad<DSSD_F32> {
    typedef Quads32 Q;
    static constexpr uint32_t kNegInf = 0xff800000u;
    __device__ static __forceinline__ float4 widen(const uint4 &v) { return as_f4(v); }
};
template <>
struct LogitQuad<DSSD_BF16> {
    typedef Quads16 Q;
    static constexpr uint32_t kNegInf = 0xff80u;
    __device__ static __forceinline__ float4 widen(const uint2 &v)
    {
        return make_float4(bf16_lo(v.x), bf16_hi(v.x), bf16_lo(v.y), bf16_hi(v.y));
    }
};

template <int DT>
struct RowLogits {  // row n of the target logits, turned into probabilities on the fly
    typedef typename LogitQuad<DT>::Q Q;
    static constexpr uint32_t kFill = LogitQuad<DT>::kNegInf;
    static constexpr bool kFixed = false;
    const char *row;
    float c1, nref, invS;
    template <class Params>
    __device__ static __forceinline__ RowLogits make(const Params &P, int64_t b, int n)
    {
        RowLogits r;
        r.row = reinterpret_cast<const char *>(P.logits) +
                ((size_t)b * (size_t)(P.gamma + 1) + (size_t)n) * (size_t)P.row_stride * Elem<DT>::kBytes;
        const ReadySlot *s = reinterpret_cast<const ReadySlot *>(P.ready) + b;
        r.c1 = P.c1;
        r.nref = -ld_after(&s->ref2);
        r.invS = ld_after(&s->invS);
        return r;
    }
    __device__ __forceinline__ float prob(float l) const { return ex2(fmaf(l, c1, nref)) * invS; }
    __device__ __forceinline__ float4 quad(const typename Q::Raw &v) const
    {
        const float4 l = LogitQuad<DT>::widen(v);
        return make_float4(prob(l.x), prob(l.y), prob(l.z), prob(l.w));
    }
};

// This thread's part of a chunk sum: the four quads of its warp's half of a chunk, entries base + 128 u +
// 4 lane .. + 3.  All loads are requested before the first is used.  q is not read without kHasQ (then
// r = p); with kPlain the sum of p goes to `plain`.
template <bool kHasQ, bool kPlain, bool kShift, typename RV>
__device__ __forceinline__ double share_mass(const RV &row, const WarpQuads<typename RV::Q, 4, kShift> &a, const float *q, int V, long long base,
                                             double &plain)
{
    WarpQuads<Quads32, 4, kShift> b;
    if (kHasQ) b.load(reinterpret_cast<const char *>(q), V, base, 0u);
    double acc = 0.0;
    plain = 0.0;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const float4 x = row.quad(a.at(u));
        if (kHasQ) {
            const float4 y = as_f4(b.at(u));
            acc += (res(x.x, y.x) + res(x.y, y.y)) + (res(x.z, y.z) + res(x.w, y.w));
        }
        if (!kHasQ || kPlain) {
            const double s = ((double)x.x + (double)x.y) + ((double)x.z + (double)x.w);
            if (kPlain) plain += s;
            if (!kHasQ) acc += s;
        }
    }
    return acc;
}
template <bool kHasQ, bool kPlain, bool kShift, typename RV>
__device__ __forceinline__ double share_mass(const RV &row, const float *q, int V, long long base, double &plain)
{
    WarpQuads<typename RV::Q, 4, kShift> a;
    a.load(row.row, V, base, RV::kFill);
    return share_mass<kHasQ, kPlain, kShift>(row, a, q, V, base, plain);
}

// r for the segment of 512 entries from `base` on: r[4 u + j] is entry base + 128 u + 4 lane + j.  `a` holds the row's quads.
template <bool kShift, typename RV>
__device__ __forceinline__ void segment_residuals(const RV &row, const WarpQuads<typename RV::Q, 4, kShift> &a, const float *q, int V,
                                                  long long base, double (&r)[16])
{
    if (q) {
        WarpQuads<Quads32, 4, kShift> d;
        d.load(reinterpret_cast<const char *>(q), V, base, 0u);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float4 x = row.quad(a.at(k)), y = as_f4(d.at(k));
            r[4 * k] = res(x.x, y.x), r[4 * k + 1] = res(x.y, y.y), r[4 * k + 2] = res(x.z, y.z), r[4 * k + 3] = res(x.w, y.w);
        }
    } else {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float4 x = row.quad(a.at(k));
            r[4 * k] = x.x, r[4 * k + 1] = x.y, r[4 * k + 2] = x.z, r[4 * k + 3] = x.w;
        }
    }
}

constexpr unsigned long long kNoSum = ~0ull;  // stored in place of a withheld chunk sum (a sum is never this NaN)

__device__ __forceinline__ bool missing(double m) { return (unsigned long long)__double_as_longlong(m) == kNoSum; }

// Where in a row the draw falls.
struct Pick {
    bool ok;        // the row's mass Z is positive and finite
    bool late;      // a chunk sum is missing
    bool beyond;    // no chunk prefix exceeds the target: take the last positive entry
    int chunk;
    double base;    // mass before that chunk
    double target;  // the running mass that the token's must exceed
};

__device__ __forceinline__ double warp_scan(double x)  // inclusive, in lane order
{
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const double up = __shfl_up_sync(0xffffffffu, x, o);
        if ((int)(threadIdx.x & 31) >= o) x += up;
    }
    return x;
}

__device__ __forceinline__ double shfl_f64(double x, int src) { return __shfl_sync(0xffffffffu, x, src); }

// The chunk sums that lane l of a warp looks at: a contiguous share of the n_sub, the first kKeep of
// them in registers.  sum(c) loads chunk sum c.
struct LaneSums {
    int c0, c1;
    double m[kKeep];
};
template <class Sum>
__device__ __forceinline__ void load_sums(LaneSums &L, int n_sub, Sum sum)
{
    const int per = (n_sub + 31) / 32;
    L.c0 = min(n_sub, (int)(threadIdx.x & 31) * per);
    L.c1 = min(n_sub, L.c0 + per);
#pragma unroll
    for (int k = 0; k < kKeep; ++k) L.m[k] = L.c0 + k < L.c1 ? sum(L.c0 + k) : 0.0;
}

// By one warp, or by several that all do the same: a prefix over the lanes' shares gives Z, and the
// first chunk whose inclusive prefix exceeds target(Z) - the last one with mass when there is none - is
// the pick.  `beyond` set by the caller means that no prefix is known to exceed the target.  The
// float64 additions that depend on one another are what this costs: the prefix within a lane's share is
// formed once and compared in parallel.
template <class Sum, class Target>
__device__ __forceinline__ Pick pick_chunk(const LaneSums &L, Sum sum, bool beyond, Target target)
{
    const int lane = threadIdx.x & 31;
    double pre[kKeep];
    double s = 0.0;
    bool late = false;
    unsigned positive = 0;
#pragma unroll
    for (int k = 0; k < kKeep; ++k) {
        s += L.m[k];
        pre[k] = s;
        late |= missing(L.m[k]);
        positive |= L.m[k] > 0.0 ? 1u << k : 0u;
    }
    for (int c = L.c0 + kKeep; c < L.c1; ++c) {
        const double x = sum(c);
        s += x;
        late |= missing(x);
    }
    const double incl = warp_scan(s);
    const double up = __shfl_up_sync(0xffffffffu, incl, 1);
    const double excl = lane ? up : 0.0;
    Pick pk;
    const double Z = shfl_f64(incl, 31);
    pk.late = __any_sync(0xffffffffu, late);
    pk.ok = (Z > 0.0) && (Z < INFINITY);
    pk.target = target(Z);
    const unsigned cross = beyond ? 0u : __ballot_sync(0xffffffffu, s > 0.0 && incl > pk.target);
    const unsigned mass = __ballot_sync(0xffffffffu, s > 0.0);
    pk.beyond = cross == 0;
    const int owner = cross ? __ffs(cross) - 1 : mass ? 31 - __clz(mass) : 0;
    // the lane's own chunks: the first that crosses, else the last with mass
    int k = 0;
    unsigned over = 0;
#pragma unroll
    for (int j = 0; j < kKeep; ++j) over |= cross && excl + pre[j] > pk.target ? 1u << j : 0u;
    over &= positive;
    bool hit = over != 0;
    if (hit) k = __ffs(over) - 1;
    else if (positive) k = 31 - __clz(positive);
    double base = excl;
#pragma unroll
    for (int j = 1; j < kKeep; ++j)
        if (j == k) base = excl + pre[j - 1];
    if (lane == owner && !hit) {  // (beyond kKeep chunks per lane only)
        double C = excl + pre[kKeep - 1];
        for (int c = L.c0 + kKeep; c < L.c1 && !hit; ++c) {
            const double x = sum(c);
            if (x > 0.0) {
                k = c - L.c0;
                base = C;
                hit = cross != 0 && C + x > pk.target;
            }
            C += x;
        }
    }
    pk.chunk = __shfl_sync(0xffffffffu, L.c0 + k, owner);
    pk.base = shfl_f64(base, owner);
    return pk;
}

// The same for more than 32 kKeep chunks (vocabularies beyond 262144): the lane whose share holds the target is found first, and
// then its share is what all lanes look at, as often as it takes.  load_sums has loaded the first chunks of every share.
template <class Sum, class Target>
__device__ __forceinline__ Pick pick_long(LaneSums L, Sum sum, bool beyond, Target target)
{
    const int lane = threadIdx.x & 31;
    Pick pk;
    double base = 0.0;  // mass before the chunks that are looked at
    for (bool first = true;; first = false) {
        double s = 0.0;
        bool late = false;
#pragma unroll
        for (int k = 0; k < kKeep; ++k) {
            s += L.m[k];
            late |= missing(L.m[k]);
        }
        for (int c = L.c0 + kKeep; c < L.c1; c += kKeep) {
            double x[kKeep];
#pragma unroll
            for (int k = 0; k < kKeep; ++k) x[k] = c + k < L.c1 ? sum(c + k) : 0.0;
#pragma unroll
            for (int k = 0; k < kKeep; ++k) {
                s += x[k];
                late |= missing(x[k]);
            }
        }
        const double incl = warp_scan(s);
        const double up = __shfl_up_sync(0xffffffffu, incl, 1);
        const double excl = lane ? base + up : base;
        if (first) {
            const double Z = shfl_f64(incl, 31);
            pk.late = __any_sync(0xffffffffu, late);
            pk.ok = (Z > 0.0) && (Z < INFINITY);
            pk.target = target(Z);
        }
        const unsigned cross = beyond ? 0u : __ballot_sync(0xffffffffu, s > 0.0 && base + incl > pk.target);
        const unsigned mass = __ballot_sync(0xffffffffu, s > 0.0);
        beyond |= cross == 0;  // (in a later look: by rounding; the share's last mass then)
        if (first) pk.beyond = beyond;
        const int owner = cross ? __ffs(cross) - 1 : mass ? 31 - __clz(mass) : 0;
        const int at = __shfl_sync(0xffffffffu, L.c0, owner), n = __shfl_sync(0xffffffffu, L.c1, owner) - at;
        base = shfl_f64(excl, owner);
        if (n <= 1) {
            pk.chunk = at;
            pk.base = base;
            return pk;
        }
        load_sums(L, n, [&](int c) { return sum(at + c); });
        L.c0 += at;
        L.c1 += at;
    }
}

// The draw inside a segment of 512 entries, by a warp: of segment g's entries in r (segment_residuals) the first whose
// running mass exceeds the target, else (rounding, or pk.beyond) the last with mass; -1: none has.
__device__ __forceinline__ int walk_segment(const Pick &pk, const double (&r)[16], int g)
{
    const int lane = threadIdx.x & 31;
    double in[4], C = pk.base;
#pragma unroll
    for (int k = 0; k < 4; ++k) in[k] = warp_scan((r[4 * k] + r[4 * k + 1]) + (r[4 * k + 2] + r[4 * k + 3]));
    int tok = -1;
    bool hit = false;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const double up = __shfl_up_sync(0xffffffffu, in[k], 1);
        const double c0 = C + (lane ? up : 0.0), c1 = c0 + r[4 * k], c2 = c1 + r[4 * k + 1], c3 = c2 + r[4 * k + 2], c4 = c3 + r[4 * k + 3];
        const unsigned pos = (r[4 * k] > 0.0 ? 1u : 0u) | (r[4 * k + 1] > 0.0 ? 2u : 0u) | (r[4 * k + 2] > 0.0 ? 4u : 0u) |
                             (r[4 * k + 3] > 0.0 ? 8u : 0u);
        const unsigned over = pk.beyond ? 0u : pos & ((c1 > pk.target ? 1u : 0u) | (c2 > pk.target ? 2u : 0u) |
                                                      (c3 > pk.target ? 4u : 0u) | (c4 > pk.target ? 8u : 0u));
        const unsigned cross = __ballot_sync(0xffffffffu, over != 0), mass = __ballot_sync(0xffffffffu, pos != 0);
        const int at = cross ? __ffs(cross) - 1 : mass ? 31 - __clz(mass) : 0;
        const int j = __shfl_sync(0xffffffffu, over ? __ffs(over) - 1 : 31 - __clz(pos | 1u), at);
        if (!hit && mass) {
            tok = 512 * g + 128 * k + 4 * at + j;
            hit = cross != 0;
        }
        C += shfl_f64(in[k], 31);
    }
    return tok;
}

// The draw of a sequence by a cluster of csize CTAs (or one CTA) whose warps hold a segment of 512 entries each, warp number
// g the entries from 512 g on; `a` is the row's part of it.  The segments' sums go to every CTA's shared memory, after one
// cluster barrier each CTA's first warp picks the segment that holds the target, and the warp that holds it finds the token.
// u is warp 0's, `sums` has room for 2 n_warps; the cluster's CTAs are known to run.
template <bool kShift, typename RV>
__device__ __forceinline__ void draw_held(const RV &row, const WarpQuads<typename RV::Q, 4, kShift> &a, const float *q, int V, int g,
                                          int n_warps, unsigned csize, unsigned rank, float u, double *sums, Pick &s_pick, int32_t *token,
                                          uint32_t *flags)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned fl = q ? 0u : DSSD_RS_FLAG_BONUS;
    double r[16];
    Pick pk;
    for (int attempt = 0;; ++attempt) {
        double *mine = sums + attempt * n_warps;
        segment_residuals<kShift>(row, a, q, V, 512ll * g, r);
        double t = 0.0;
#pragma unroll
        for (int k = 0; k < 4; ++k) t += (r[4 * k] + r[4 * k + 1]) + (r[4 * k + 2] + r[4 * k + 3]);
        t = warp_sum(t);
        if (csize > 1) {
            if (lane < (int)csize) cluster_store(mine + g, (unsigned)lane, t);
            cluster_arrive();
            cluster_wait();
        } else {
            if (lane == 0) mine[g] = t;
            __syncthreads();
        }
        // one warp per CTA: its float64 operations would hold up the others' if every warp did them
        if (warp == 0) {
            LaneSums L;
            auto sum = [&](int c) { return mine[c]; };
            load_sums(L, n_warps, sum);
            const Pick got = pick_chunk(L, sum, false, [&](double Z) { return (double)u * Z; });
            if (lane == 0) s_pick = got;
        }
        __syncthreads();
        pk = s_pick;
        if (pk.ok || !q) break;
        q = nullptr;  // residual has no mass (p == q): draw from p instead
        fl |= DSSD_RS_FLAG_FALLBACK;
        __syncthreads();  // the pick has been read
    }
    if (!pk.ok) {
        if (rank == 0 && threadIdx.x == 0) {
            *token = -1;
            if (flags) *flags = fl | DSSD_RS_FLAG_INVALID;
        }
        return;
    }
    if (g != pk.chunk) return;
    const int tok = walk_segment(pk, r, g);
    if (lane == 0) {
        *token = tok;
        if (flags) *flags = fl | (tok < 0 ? DSSD_RS_FLAG_INVALID : 0u);
    }
}

// The same where the warps take segments in turns: warp g of the n_warps the segments g, g + n_warps, ..  The sums go to the first
// CTA's shared memory, and after a cluster barrier its first warp picks the segment that holds the target, fetches it
// again and walks it.  `a` is the row's part of the warp's first segment.
constexpr int kDrawSegs = 1024;  // most segments of such a row (8 KB)
struct DrawShared {
    double sum[kDrawSegs];
    Pick pick;
    int again;
};
template <bool kShift, typename RV>
__device__ __forceinline__ void draw_streamed(const RV &row, WarpQuads<typename RV::Q, 4, kShift> &a, const float *q, int V, int g, int n_warps,
                                              unsigned csize, unsigned rank, float u, DrawShared &sh, int32_t *token, uint32_t *flags)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, segs = (V + 511) / 512;
    unsigned fl = q ? 0u : DSSD_RS_FLAG_BONUS;
    for (int i = g; i < segs; i += n_warps) {
        double none, t;
        if (i != g) a.load(row.row, V, 512ll * i, RV::kFill);
        if (q) t = share_mass<true, false, kShift>(row, a, q, V, 512ll * i, none);
        else t = share_mass<false, false, kShift>(row, a, q, V, 512ll * i, none);
        t = warp_sum(t);
        if (lane == 0) {
            if (csize > 1) cluster_store(&sh.sum[i], 0u, t);
            else sh.sum[i] = t;
        }
    }
    if (csize > 1) {
        cluster_arrive();
        cluster_wait();
    } else {
        __syncthreads();
    }
    if (rank) return;
    Pick pk;
    auto pick = [&]() {
        LaneSums L;
        auto sum = [&](int c) { return sh.sum[c]; };
        load_sums(L, segs, sum);
        pk = pick_chunk(L, sum, false, [&](double Z) { return (double)u * Z; });
    };
    if (warp == 0) {
        pick();
        if (lane == 0) sh.again = !pk.ok && q;
    }
    __syncthreads();
    if (sh.again) {  // the residual has no mass (p == q): draw from p instead; rare, so by this CTA alone
        q = nullptr;
        fl |= DSSD_RS_FLAG_FALLBACK;
        for (int i = warp; i < segs; i += (int)(blockDim.x >> 5)) {
            double none;
            const double t = warp_sum(share_mass<false, false, kShift>(row, q, V, 512ll * i, none));
            if (lane == 0) sh.sum[i] = t;
        }
        __syncthreads();
        if (warp == 0) pick();
    }
    if (warp) return;
    int tok = -1;
    if (pk.ok) {
        double r[16];
        a.load(row.row, V, 512ll * pk.chunk, RV::kFill);
        segment_residuals<kShift>(row, a, q, V, 512ll * pk.chunk, r);
        tok = walk_segment(pk, r, pk.chunk);
    }
    if (lane == 0) {
        *token = tok;
        if (flags) *flags = fl | (tok < 0 ? DSSD_RS_FLAG_INVALID : 0u);
    }
}

}  // namespace dssd
