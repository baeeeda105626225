// Edge half of the verification round, as two or three kernels whose CTAs the hardware schedules.
//
//   edge_lse_kernel   one CTA per run of one target row (16 to 64 KB of logits): an online maximum and
//                     sum of 2^(l * c1 - ref) per thread in float32, reduced to the run's (ref, sum)
//                     and stored.  ref is an integer, so partials combine by exact power-of-two
//                     scaling.  The CTA whose run holds the row's drafted token also leaves that
//                     token's logit (and its draft probability, when the draft rows are given).
//   edge_fold_kernel  one CTA per sequence: log-sum-exps, acceptance tests, first rejection (edge_fold.cuh).
//                     Small launches have no such kernel: every emission CTA folds its sequence itself.
//   edge_emit_kernel  one CTA per tile of row n of a sequence: reads its tile of row n again and writes
//                     p_row = 2^(l * c1 - ref) / S.
//
//
// Where a sequence's rows are few or short for the number of sequences, one kernel does it all instead:
//
//   edge_cluster_kernel  a CTA or a cluster of CTAs per sequence; the partial sums go through shared memory.
//
// The end of a kernel (and the cluster's barrier) is the only synchronisation: no counter, no flag, no wait on another CTA,
// nothing in the workspace that has to be cleared.  A kernel's CTAs are scheduled while the one
// before it drains (launch.h).
#include "edge_verify.h"

#include <math.h>

#include "draw.cuh"
#include "dssd_device.cuh"
#include "edge_fold.cuh"
#include "emit.cuh"
#include "launch.h"

namespace dssd {

namespace {

constexpr int kSegVecs = 32 * kLseLoads;  // 16-byte vectors of a warp's segment of a row in the cluster kernel (4 KB)
constexpr int kPieceQuads = 4;            // quads per lane that a warp emits at a time there (eight: 0.4 us slower at B = 8 V = 32000)

template <int DT>
__device__ __forceinline__ const char *row_ptr(const EdgeParams &P, long long row)
{
    return static_cast<const char *>(P.logits) + (size_t)row * (size_t)P.row_stride * Elem<DT>::kBytes;
}

// ---- per-thread online log-sum-exp state ---------------------------------------------------

struct Online {
    float m;    // running maximum of the raw logits (-inf: nothing seen)
    float ref;  // rint(m * c1), or 0 while m == -inf: terms are 2^(l * c1 - ref) <= 2^0.5
    f32x2 s0, s1, s2, s3;  // eight running sums, as four packed pairs
};

__device__ __forceinline__ void online_raise(Online &o, float bm, float c1)
{
    if (bm > o.m) {
        const float nref = rintf(bm * c1);
        if (nref == DSSD_NEG_INF) return;  // all of them lie below float32's range (a mask of the type's lowest value): like -inf
        const float f = (o.m == DSSD_NEG_INF) ? 0.f : ex2(o.ref - nref);  // an exact power of two
        const f32x2 ff = pack2(f, f);
        o.s0 = mul2(o.s0, ff);
        o.s1 = mul2(o.s1, ff);
        o.s2 = mul2(o.s2, ff);
        o.s3 = mul2(o.s3, ff);
        o.m = bm;
        o.ref = nref;
    }
}

// acc += 2^(a * c1 - ref), 2^(b * c1 - ref)
__device__ __forceinline__ void add_pair(f32x2 &acc, float a, float b, f32x2 cc, f32x2 nn)
{
    float x, y;
    unpack2(fma2(pack2(a, b), cc, nn), x, y);
    acc = add2(acc, pack2(ex2(x), ex2(y)));
}

// x within [-127, 128]; a NaN stays one
__device__ __forceinline__ float clamp_nan(float x)
{
    float r;
    asm("{\n\t.reg .f32 t;\n\tmax.NaN.f32 t, %1, 0fC2FE0000;\n\tmin.NaN.f32 %0, t, 0f43000000;\n\t}" : "=f"(r) : "f"(x));
    return r;
}

// The same without the special-function unit, which bf16 rows keep four fifths busy: 2^x = 2^n 2^f with n = rint(x)
// and a polynomial for 2^f, |f| <= 1/2, of degree 6, fitted for the least relative error by Remez exchange (1.9e-9; 8e-8 with float32
// roundings, the unit's own error is 2^-22).  Adding kRound leaves n + 127 in the last bits, which shifted up are the
// float 2^n: 0 for n = -127 and infinity for n = 128, where the unit's results end too.  A NaN stays one.
__device__ __forceinline__ void add_pair_by_fma(f32x2 &acc, float a, float b, f32x2 cc, f32x2 nn)
{
    constexpr float kRound = 12582912.f + 127.f;
    float x, y, tx, ty;
    unpack2(fma2(pack2(a, b), cc, nn), x, y);
    const f32x2 z = pack2(clamp_nan(x), clamp_nan(y));
    const f32x2 t = add2(z, pack2(kRound, kRound));
    const f32x2 f = fma2(add2(t, pack2(-kRound, -kRound)), pack2(-1.f, -1.f), z);
    unpack2(t, tx, ty);
    f32x2 p = pack2(1.534581242594868e-4f, 1.534581242594868e-4f);
    p = fma2(p, f, pack2(1.3399930903688073e-3f, 1.3399930903688073e-3f));
    p = fma2(p, f, pack2(9.618489071726799e-3f, 9.618489071726799e-3f));
    p = fma2(p, f, pack2(5.550328642129898e-2f, 5.550328642129898e-2f));
    p = fma2(p, f, pack2(2.4022646248340607e-1f, 2.4022646248340607e-1f));
    p = fma2(p, f, pack2(6.931471824645996e-1f, 6.931471824645996e-1f));
    p = fma2(p, f, pack2(1.f, 1.f));
    acc = fma2(p, pack2(__uint_as_float(__float_as_uint(tx) << 23), __uint_as_float(__float_as_uint(ty) << 23)), acc);
}

template <int DT>
__device__ __forceinline__ float vec_max(const uint4 &v)
{
    if (DT == DSSD_BF16) {
        const uint32_t m = max_bf16x2(max_bf16x2(v.x, v.y), max_bf16x2(v.z, v.w));
        return fmaxf(bf16_lo(m), bf16_hi(m));
    }
    return fmaxf(fmaxf(__uint_as_float(v.x), __uint_as_float(v.y)), fmaxf(__uint_as_float(v.z), __uint_as_float(v.w)));
}

// kFma: a quarter of a bf16 vector's terms on the FMA pipe
template <int DT, bool kFma>
__device__ __forceinline__ void add_vec(Online &o, const uint4 &v, f32x2 cc, f32x2 nn)
{
    if (DT == DSSD_BF16) {
        add_pair(o.s0, bf16_lo(v.x), bf16_hi(v.x), cc, nn);
        add_pair(o.s1, bf16_lo(v.y), bf16_hi(v.y), cc, nn);
        add_pair(o.s2, bf16_lo(v.z), bf16_hi(v.z), cc, nn);
        if (kFma) add_pair_by_fma(o.s3, bf16_lo(v.w), bf16_hi(v.w), cc, nn);
        else add_pair(o.s3, bf16_lo(v.w), bf16_hi(v.w), cc, nn);
    } else {
        add_pair(o.s0, __uint_as_float(v.x), __uint_as_float(v.y), cc, nn);
        add_pair(o.s1, __uint_as_float(v.z), __uint_as_float(v.w), cc, nn);
    }
}

template <int DT>
__device__ __forceinline__ uint4 neg_inf_vec()
{
    return DT == DSSD_BF16 ? make_uint4(0xff80ff80u, 0xff80ff80u, 0xff80ff80u, 0xff80ff80u)
                           : make_uint4(0xff800000u, 0xff800000u, 0xff800000u, 0xff800000u);
}

template <int DT>
__device__ __forceinline__ void add_tile(Online &o, const uint4 (&v)[kLseLoads], float c1)
{
    float bm = vec_max<DT>(v[0]);
#pragma unroll
    for (int u = 1; u < kLseLoads; ++u) bm = fmaxf(bm, vec_max<DT>(v[u]));
    online_raise(o, bm, c1);
    const f32x2 cc = pack2(c1, c1), nn = pack2(-o.ref, -o.ref);
    // every second vector: B = 256 gamma = 4 V = 151936 63.3 us against 64.5 without and 63.9 with every vector
#pragma unroll
    for (int u = 0; u < kLseLoads; u += 2) {
        add_vec<DT, true>(o, v[u], cc, nn);
        add_vec<DT, false>(o, v[u + 1], cc, nn);
    }
}

// one entry more
__device__ __forceinline__ void add_extra(Online &o, float extra, float c1)
{
    if (extra > DSSD_NEG_INF || extra != extra) {
        online_raise(o, extra, c1);
        o.s0 = add2(o.s0, pack2(ex2(fmaf(extra, c1, -o.ref)), 0.f));
    }
}

// the warp's (ref, sum): exact power-of-two scaling; a NaN sum stays one
__device__ __forceinline__ void online_total(const Online &o, float &R, float &s)
{
    float a, b;
    unpack2(add2(add2(o.s0, o.s1), add2(o.s2, o.s3)), a, b);
    s = a + b;
    const float r = o.m == DSSD_NEG_INF ? DSSD_NEG_INF : o.ref;
    R = warp_max(r);
    s = warp_sum(r == DSSD_NEG_INF ? (s != s ? s : 0.f) : s * ex2(r - R));
}

__device__ __forceinline__ unsigned long long partial_word(float R, float s)
{
    if (s != s) s = __int_as_float(0x7fc00000);
    return (unsigned long long)__float_as_uint(R == DSSD_NEG_INF ? 0.f : R) | ((unsigned long long)__float_as_uint(s) << 32);
}

// Bound by HBM: 128 threads with eight 16-byte loads in flight each, eight CTAs per SM (64 registers) read
// B = 256 gamma = 4 V = 151936 bf16 (389 MB) in 63 us and B = 1024 gamma = 16 V = 50272 float32 (3.5 GB) in
// 500 us, 7.0 TB/s; a pure read of the same shape takes 60 and 497 us, so the exponentials are nearly
// hidden.  256 threads: 68 us, four loads and sixteen CTAs: 95 us, six or nine CTAs per SM: 69 us.  The
// persistent kernel it replaces (tickets, ring, fold warp, scout) had the fold and the emission inside
// and took 100 us where this one, the fold and the emission take 103, but 15.6 us where they take 6.5
// (B = 1 V = 50272), 43 where they take 40 (B = 64 gamma = 8 V = 128256) and 54 where they take 37 (B = 300
// V = 30011, unaligned rows).
// One CTA per (row, run).  A row's vectors start at its first 16-byte boundary; the up to seven
// entries before it belong to the first run, those after the last whole vector to the last run.
template <int DT>
__global__ void __launch_bounds__(kLseThreads, 8) edge_lse_kernel(const __grid_constant__ EdgeParams P)
{
    using E = Elem<DT>;
    __shared__ float2 s_warp[kLseThreads / 32];
    const int tid = threadIdx.x;
    const unsigned row = blockIdx.x / (unsigned)P.runs;
    const int run = (int)(blockIdx.x - row * (unsigned)P.runs);
    const char *rowp = row_ptr<DT>(P, row);
    const float c1 = P.c1;
    const long long rowbytes = (long long)P.V * E::kBytes;
    int head = (int)((16u - (unsigned)(reinterpret_cast<uintptr_t>(rowp) & 15u)) & 15u);
    if (head > rowbytes) head = (int)rowbytes;
    const int nvec = (int)((rowbytes - head) >> 4);
    const int v0 = min(nvec, run * P.run_vecs), v1 = run + 1 == P.runs ? nvec : min(nvec, v0 + P.run_vecs);
    const uint4 *src = reinterpret_cast<const uint4 *>(rowp + head);
    const unsigned seq = row / (unsigned)(P.gamma + 1);
    const int pos = (int)(row - seq * (unsigned)(P.gamma + 1));
    pdl_wait();
    pdl_trigger();
    // the drafted token's id travels with the first vectors
    const bool scout = tid == 0 && pos < P.gamma;
    long long x = -1;
    if (scout) x = (long long)ld_after(P.draft_tokens + (size_t)seq * P.gamma + pos) - (long long)P.v_begin;
    // the entries outside the vectors: at most one per thread
    float extra = DSSD_NEG_INF;
    if (run == 0 && tid < head / E::kBytes) extra = E::load(rowp, tid);
    if (run + 1 == P.runs && tid >= 32) {
        const int e = (int)((head + ((long long)nvec << 4)) / E::kBytes) + tid - 32;
        if (e < P.V) extra = E::load(rowp, e);
    }
    Online o;
    o.m = DSSD_NEG_INF;
    o.ref = 0.f;
    o.s0 = o.s1 = o.s2 = o.s3 = 0ull;
    int i = v0 + tid;
    for (; i + (kLseLoads - 1) * kLseThreads < v1; i += kLseTile) {
        uint4 v[kLseLoads];
#pragma unroll
        for (int u = 0; u < kLseLoads; ++u) v[u] = ld_stream16(src + i + u * kLseThreads);
        add_tile<DT>(o, v, c1);
    }
    if (i < v1) {
        uint4 v[kLseLoads];
#pragma unroll
        for (int u = 0; u < kLseLoads; ++u) {
            v[u] = neg_inf_vec<DT>();
            if (i + u * kLseThreads < v1) v[u] = ld_stream16(src + i + u * kLseThreads);
        }
        add_tile<DT>(o, v, c1);
    }
    float zx = 0.f, qx = 0.f;
    bool owned = false;
    if (scout && x >= 0 && x < (long long)P.V) {
        const long long vec = x * E::kBytes < head ? -1 : (x * E::kBytes - head) >> 4;
        owned = (vec >= v0 && vec < v1) || (vec < 0 && run == 0) || (vec >= nvec && run + 1 == P.runs);
        if (owned) {
            zx = E::load(rowp, x);
            if (P.draft_q_rows) qx = ld_after(P.draft_q_rows + ((size_t)seq * P.gamma + pos) * (size_t)P.V + (size_t)x);
        }
    }
    add_extra(o, extra, c1);
    float R, s;  // the warp's, then the CTA's
    online_total(o, R, s);
    if ((tid & 31) == 0) s_warp[tid >> 5] = make_float2(R, s);
    __syncthreads();
    if (tid == 0) {
        float Rt = s_warp[0].x;
#pragma unroll
        for (int w = 1; w < kLseThreads / 32; ++w) Rt = fmaxf(Rt, s_warp[w].x);
        float t = 0.f;
#pragma unroll
        for (int w = 0; w < kLseThreads / 32; ++w) {
            const float2 c = s_warp[w];
            t += c.x == DSSD_NEG_INF ? (c.y != c.y ? c.y : 0.f) : c.y * ex2(c.x - Rt);
        }
        P.part[blockIdx.x] = (long long)row + 1 == P.test_drop_row_plus1 ? kNoPartial : partial_word(Rt, t);
        if (owned) {
            P.tokz[row] = zx;
            if (P.draft_q_rows) P.tokq[row] = qx;
        }
    }
}

// ---- emission (emit.cuh) ----------------------------------------------------------------------

// kWide: more than kFoldWide runs per row (B = 1 gamma = 2 float32, the edge call, eight threads per row / a warp: V = 16777216
// 189.6 / 67.8 us, V = 67108864 471 / 228, V = 1048576 18.8 / 9.7, V = 300000 11.4 / 8.5)
template <bool kWide>
__global__ void __launch_bounds__(kThreads) edge_fold_kernel(const __grid_constant__ EdgeParams P)
{
    __shared__ FoldShared sh;
    pdl_wait();
    pdl_trigger();
    fold_sequence<kWide>(P, blockIdx.x, true, sh);
}

// Bound by HBM: reads and writes mixed, 234 MB at B = 256 V = 151936 in 36.5 us.
// One CTA per (sequence, tile of row n), after a fold of its own or (kFold = false) the fold kernel's.
// The sequences run backwards: the rows that the log-sum-exp kernel read last are the ones still in L2.
template <int DT, bool kFold, bool kShift>
__global__ void __launch_bounds__(kThreads, 4) edge_emit_kernel(const __grid_constant__ EdgeParams P)
{
    const unsigned rb = blockIdx.x / (unsigned)P.emit_tiles;
    const int tile = (int)(blockIdx.x - rb * (unsigned)P.emit_tiles);
    const long long b = (long long)P.B - 1 - (long long)rb;
    pdl_wait();
    pdl_trigger();
    int n;
    float ref2, invS;
    if (kFold) {
        __shared__ FoldShared sh;
        fold_sequence<false>(P, b, tile == 0, sh);
        n = sh.n;
        ref2 = sh.ref2;
        invS = sh.invS;
    } else {
        const ReadySlot *s = P.ready + b;
        n = ld_after(&s->n);
        ref2 = ld_after(&s->ref2);
        invS = ld_after(&s->invS);
    }
    if (n < 0 || (P.skip_bonus_row && n == P.gamma)) return;
    const char *rowp = row_ptr<DT>(P, b * (P.gamma + 1) + n);
    if (P.p_row16) emit_tile<DT, kShift>(rowp, P.p_row16 + (size_t)b * P.V, P.V, tile, P.c1, ref2, invS);
    else emit_tile<DT, kShift>(rowp, P.p_row + (size_t)b * P.V, P.V, tile, P.c1, ref2, invS);
}

// ---- small launches: one cluster of CTAs per sequence ---------------------------------------------

// One warp's part of a row: the kLseLoads * 32 vectors from v0 on, and the entries outside the vectors that
// belong to them.  The result is the warp's (ref, sum), the same in all lanes.
template <int DT>
__device__ __forceinline__ void warp_lse(const char *rowp, int V, int seg, int segs, float c1, float &R, float &s)
{
    using E = Elem<DT>;
    const int lane = threadIdx.x & 31;
    const long long rowbytes = (long long)V * E::kBytes;
    int head = (int)((16u - (unsigned)(reinterpret_cast<uintptr_t>(rowp) & 15u)) & 15u);
    if (head > rowbytes) head = (int)rowbytes;
    const int nvec = (int)((rowbytes - head) >> 4);
    const uint4 *src = reinterpret_cast<const uint4 *>(rowp + head);
    const int i = seg * kSegVecs + lane;
    uint4 v[kLseLoads];
    if (seg * kSegVecs + kSegVecs <= nvec) {
#pragma unroll
        for (int u = 0; u < kLseLoads; ++u) v[u] = ld_stream16(src + i + 32 * u);
    } else {
#pragma unroll
        for (int u = 0; u < kLseLoads; ++u) {
            v[u] = neg_inf_vec<DT>();
            if (i + 32 * u < nvec) v[u] = ld_stream16(src + i + 32 * u);
        }
    }
    float extra = DSSD_NEG_INF;  // the up to seven entries before the vectors: lanes 0 .. 6; those after them: lanes 16 .. 22
    if (seg == 0 && lane < head / E::kBytes) extra = E::load(rowp, lane);
    if (seg + 1 == segs && lane >= 16) {
        const int e = (int)((head + ((long long)nvec << 4)) / E::kBytes) + lane - 16;
        if (e < V) extra = E::load(rowp, e);
    }
    Online o;
    o.m = DSSD_NEG_INF;
    o.ref = 0.f;
    o.s0 = o.s1 = o.s2 = o.s3 = 0ull;
    add_tile<DT>(o, v, c1);
    add_extra(o, extra, c1);
    online_total(o, R, s);
}

template <int DT, bool kShift, class OUT>
__device__ __forceinline__ void emit_pieces(const char *rowp, OUT *outp, int V, int g, int n_warps, float c1, float ref2, float invS)
{
    const long long lead = kShift ? emit_lead(outp) : 0;
    for (long long e = 128ll * kPieceQuads * g - lead; e < V; e += 128ll * kPieceQuads * n_warps)
        emit_piece<DT, kShift, kPieceQuads>(rowp, outp, V, e, c1, ref2, invS);
}

// The draw from row n of sequence b, by the cluster that has folded it: where its warps can hold the row (draw_held) as
// the kernel of small draws does it, else in turns (draw_streamed).
static_assert(kDrawSegs >= 2 * kEdgeClusterWide * kWarps, "draw_held keeps two sets of sums");
template <int DT, bool kShift, bool kHeld>
__device__ __forceinline__ void draw_here(const EdgeParams &P, long long b, const char *rowp, int n, float ref2, float invS, int n_warps,
                                          unsigned csize, unsigned rank, DrawShared &sh)
{
    const int warp = threadIdx.x >> 5, g = warp * (int)csize + (int)rank;
    const float *q = n < P.gamma ? P.draft_q_rows + ((size_t)b * P.gamma + n) * (size_t)P.V : nullptr;
    RowLogits<DT> row;
    row.row = rowp;
    row.c1 = P.c1;
    row.nref = -ref2;
    row.invS = invS;
    const float u = warp == 0 ? ld_after(P.draw_uniforms + b) : 0.f;
    WarpQuads<typename RowLogits<DT>::Q, 4, kShift> a;
    a.load(rowp, P.V, 512ll * g, RowLogits<DT>::kFill);
    uint32_t *flags = P.draw_flags ? P.draw_flags + b : nullptr;
    if constexpr (kHeld) draw_held<kShift>(row, a, q, P.V, g, n_warps, csize, rank, u, sh.sum, sh.pick, P.draw_token + b, flags);
    else draw_streamed<kShift>(row, a, q, P.V, g, n_warps, csize, rank, u, sh, P.draw_token + b, flags);
}

// One cluster of up to sixteen CTAs per sequence does the whole of it.  Warp g of the cluster's takes the segments
// g, g + warps, .. of the sequence's rows; every segment's (ref, sum) goes to every CTA's shared memory, and after
// one cluster barrier every CTA folds the sequence for itself and emits its part of row n.  kDraw = 1, 2: the call wants
// tokens too (of every sequence, or of the fully accepted ones); 2 holds the row in registers meanwhile, which
// saves fetching a segment again (B = 8 V = 32000 fused 7.9 us against 8.6) but costs half of the CTAs per SM.
// kCta: threads of a CTA, 0: as many as were launched (where they are known the shortest calls are 0.2 us shorter).
template <int DT, bool kShift, int kDraw, int kCta>
__global__ void __launch_bounds__(kCta ? kCta : kEdgeMostThreads, kDraw == 2 || !kCta ? 2 : 4) edge_cluster_kernel(const __grid_constant__ EdgeParams P)
{
    __shared__ unsigned long long s_part[kEdgeClusterParts];
    __shared__ Drafted s_draft[kFoldRows];
    __shared__ FoldShared sh;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, cta_warps = kCta ? kCta / 32 : (int)(blockDim.x >> 5);
    const unsigned csize = (unsigned)P.cluster, rank = csize > 1 ? cluster_rank() : 0u;
    const long long b = blockIdx.x / csize, row0 = b * (P.gamma + 1);
    const int g = warp * (int)csize + (int)rank, n_warps = (int)csize * cta_warps;
    if (csize > 1) {  // a CTA's shared memory may be written once it is known to run
        cluster_arrive();
        cluster_wait();
    }
    pdl_wait();
    pdl_trigger();
    // the last warp has the fewest segments: it looks the drafted tokens up
    if (warp == cta_warps - 1 && lane < P.gamma) {
        const size_t di = (size_t)b * P.gamma + lane;
        Drafted d;
        d.x = ld_after(P.draft_tokens + di);
        d.u = ld_after(P.uniforms + di);
        d.q = d.z = 0.f;
        if (!P.draft_q_rows) d.q = ld_after(P.draft_q_tok + di);
        if (d.x >= 0 && d.x < P.V) {
            d.z = Elem<DT>::load(row_ptr<DT>(P, row0 + lane), d.x);
            if (P.draft_q_rows) d.q = ld_after(P.draft_q_rows + di * (size_t)P.V + d.x);
        }
        s_draft[lane] = d;
    }
    for (int t = g; t < P.runs * (P.gamma + 1); t += n_warps) {
        const int i = t / P.runs;
        float R, s;
        warp_lse<DT>(row_ptr<DT>(P, row0 + i), P.V, t - i * P.runs, P.runs, P.c1, R, s);
        const unsigned long long word = row0 + i + 1 == P.test_drop_row_plus1 ? kNoPartial : partial_word(R, s);
        if (csize == 1) s_part[t] = word;
        else if (lane < (int)csize) cluster_store(&s_part[t], (unsigned)lane, word);
    }
    if (csize > 1) {
        cluster_arrive();
        cluster_wait();
    } else {
        __syncthreads();
    }
    fold_sequence<false, kCta>(P, b, rank == 0, sh, [&](int i, int k) { return s_part[i * P.runs + k]; }, [&](int i) { return s_draft[i]; });
    const int n = sh.n;
    if (kDraw) {
        __shared__ DrawShared sd;
        if (n == P.gamma || (n >= 0 && P.draw_rejected)) {
            draw_here<DT, kShift, kDraw == 2>(P, b, row_ptr<DT>(P, row0 + n), n, sh.ref2, sh.invS, n_warps, csize, rank, sd);
            return;
        }
        if (rank == 0 && threadIdx.x == 0) {  // no verdict, or a token that the device half draws
            P.draw_token[b] = -1;
            if (P.draw_flags) P.draw_flags[b] = n < 0 ? DSSD_RS_FLAG_INVALID : 0u;
        }
    }
    if (n < 0) return;
    const char *rowp = row_ptr<DT>(P, row0 + n);
    if (P.p_row16) emit_pieces<DT, kShift>(rowp, P.p_row16 + (size_t)b * P.V, P.V, g, n_warps, P.c1, sh.ref2, sh.invS);
    else if (P.p_row) emit_pieces<DT, kShift>(rowp, P.p_row + (size_t)b * P.V, P.V, g, n_warps, P.c1, sh.ref2, sh.invS);
}

// One shard of the vocabulary: the rows' sums and the drafted tokens' logits go out as they are.  kWide: a warp per row.
template <bool kWide>
__global__ void __launch_bounds__(kThreads) edge_partial_kernel(const __grid_constant__ EdgeParams P)
{
    constexpr int kLanes = kWide ? 32 : kFoldLanes;
    const long long rows = (long long)P.B * (P.gamma + 1);
    const long long row = (long long)blockIdx.x * (kThreads / kLanes) + threadIdx.x / kLanes;
    const int sub = threadIdx.x % kLanes;
    const bool live = row < rows;
    pdl_wait();
    pdl_trigger();
    const long long b = live ? row / (P.gamma + 1) : 0;
    const int i = (int)(row - b * (P.gamma + 1));
    long long x = -1;
    float zx = 0.f;
    if (live && sub == 0 && i < P.gamma) {
        x = (long long)ld_after(P.draft_tokens + (size_t)b * P.gamma + i) - (long long)P.v_begin;
        zx = ld_after(P.tokz + row);
    }
    float R;
    double S;
    bool missing;
    auto part = [&](int k) { return ld_after(P.part + (size_t)row * P.runs + k); };
    if (kWide) row_total_wide(part, live ? P.runs : 0, R, S, missing);
    else row_total(part, P.runs, sub, live, R, S, missing);
    if (live && sub == 0) {
        P.shard_ref[row] = R == DSSD_NEG_INF ? 0.f : R;
        P.shard_sum[row] = missing || S != S ? (double)__int_as_float(0x7fc00000) : S;
        if (i < P.gamma) P.shard_tok_logit[(size_t)b * P.gamma + i] = (x >= 0 && x < (long long)P.V) ? zx : __int_as_float(0x7fc00000);
    }
}

// The same in one launch, chosen as the cluster kernel is: the partial sums go to the first CTA's shared memory.
template <int DT, int kCta>
__global__ void __launch_bounds__(kCta ? kCta : kEdgeMostThreads, kCta ? 4 : 2) edge_partial_cluster_kernel(const __grid_constant__ EdgeParams P)
{
    __shared__ unsigned long long s_part[kEdgeClusterParts];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, cta_warps = kCta ? kCta / 32 : (int)(blockDim.x >> 5);
    const unsigned csize = (unsigned)P.cluster, rank = csize > 1 ? cluster_rank() : 0u;
    const long long b = blockIdx.x / csize, row0 = b * (P.gamma + 1);
    if (csize > 1) {  // the first CTA's shared memory may be written once it is known to run
        cluster_arrive();
        cluster_wait();
    }
    pdl_wait();
    pdl_trigger();
    if (rank == 0 && warp == cta_warps - 1 && lane < P.gamma) {
        const size_t di = (size_t)b * P.gamma + lane;
        const long long x = (long long)ld_after(P.draft_tokens + di) - (long long)P.v_begin;
        P.shard_tok_logit[di] = x >= 0 && x < (long long)P.V ? Elem<DT>::load(row_ptr<DT>(P, row0 + lane), x) : __int_as_float(0x7fc00000);
    }
    for (int t = warp * (int)csize + (int)rank; t < P.runs * (P.gamma + 1); t += cta_warps * (int)csize) {
        const int i = t / P.runs;
        float R, s;
        warp_lse<DT>(row_ptr<DT>(P, row0 + i), P.V, t - i * P.runs, P.runs, P.c1, R, s);
        const unsigned long long word = row0 + i + 1 == P.test_drop_row_plus1 ? kNoPartial : partial_word(R, s);
        if (lane == 0) {
            if (csize > 1) cluster_store(&s_part[t], 0u, word);
            else s_part[t] = word;
        }
    }
    if (csize > 1) {
        cluster_arrive();
        cluster_wait();
    } else {
        __syncthreads();
    }
    if (rank) return;
    auto total = [&](int i) {
        float R;
        double S;
        bool missing;
        row_total([&](int k) { return s_part[i * P.runs + k]; }, P.runs, tid % kFoldLanes, i <= P.gamma, R, S, missing);
        if (i <= P.gamma && tid % kFoldLanes == 0) {
            P.shard_ref[row0 + i] = R == DSSD_NEG_INF ? 0.f : R;
            P.shard_sum[row0 + i] = missing || S != S ? (double)__int_as_float(0x7fc00000) : S;
        }
    };
    if (kCta || tid < kThreads) total(tid / kFoldLanes);
    if (!kCta && blockDim.x < kThreads && kFoldRows / 2 <= P.gamma) total(tid / kFoldLanes + kFoldRows / 2);  // 128 threads: half of the rows at a time
}

}  // namespace

int edge_max_runs_per_row(int V)
{
    const long long n = ((long long)V * 4 / 16 + kLseTile - 1) / kLseTile;
    return (int)(n < 1 ? 1 : n);
}

size_t edge_workspace_layout(int B, int gamma, int runs_per_row, EdgeParams *P, char *base)
{
    const size_t R = (size_t)B * (size_t)(gamma + 1);
    size_t off = 0;
    auto take = [&](size_t bytes) {
        size_t o = off;
        off += (bytes + 255) & ~(size_t)255;
        return o;
    };
    const size_t o_ready = take((size_t)B * sizeof(ReadySlot));
    const size_t o_part = take(R * (size_t)runs_per_row * 8);
    const size_t o_tokz = take(R * 4);
    const size_t o_tokq = take(R * 4);
    if (P) {
        P->ready = reinterpret_cast<ReadySlot *>(base + o_ready);
        P->part = reinterpret_cast<unsigned long long *>(base + o_part);
        P->tokz = reinterpret_cast<float *>(base + o_tokz);
        P->tokq = reinterpret_cast<float *>(base + o_tokq);
    }
    return off;
}

namespace {

template <int DT, bool kShift>
cudaError_t launch_emit(const EdgeParams &P, unsigned ctas, bool fold, cudaStream_t stream)
{
    return fold ? launch_pdl(edge_emit_kernel<DT, true, kShift>, ctas, kThreads, stream, P)
                : launch_pdl(edge_emit_kernel<DT, false, kShift>, ctas, kThreads, stream, P);
}

template <int DT>
bool outputs_aligned(const EdgeParams &P)
{
    return emit_aligned(P.logits, P.row_stride, Elem<DT>::kBytes, P.p_row16 ? (const void *)P.p_row16 : P.p_row, P.V, P.p_row16 ? 2 : 4);
}

template <int DT, int kDraw, int kCta>
cudaError_t launch_cluster(const EdgeParams &P, cudaStream_t stream)
{
    const unsigned grid = (unsigned)P.B * (unsigned)P.cluster, threads = (unsigned)P.cta, cluster = (unsigned)P.cluster;
    const bool aligned = outputs_aligned<DT>(P) && (!P.draw_rejected || reinterpret_cast<uintptr_t>(P.draft_q_rows) % 16 == 0);
    return launch_pdl(aligned ? edge_cluster_kernel<DT, false, kDraw, kCta> : edge_cluster_kernel<DT, true, kDraw, kCta>, grid, threads, stream, P, 0, cluster);
}

// does a launch of this shape that draws hold the row in registers?
bool draws_held(const EdgeParams &P, int cta, long long cluster)
{
    return P.draw_token && cta == kThreads && P.B * cluster <= kEdgeHeldWave && P.V <= 512 * kWarps * cluster;
}

template <int DT>
cudaError_t launch_cluster(const EdgeParams &P, cudaStream_t stream)
{
    const bool usual = P.cta == kThreads;
    if (P.shard_sum)
        return launch_pdl(usual ? edge_partial_cluster_kernel<DT, kThreads> : edge_partial_cluster_kernel<DT, 0>, (unsigned)P.B * (unsigned)P.cluster,
                          (unsigned)P.cta, stream, P, 0, (unsigned)P.cluster);
    if (!P.draw_token) return usual ? launch_cluster<DT, 0, kThreads>(P, stream) : launch_cluster<DT, 0, 0>(P, stream);
    if (draws_held(P, P.cta, P.cluster)) return launch_cluster<DT, 2, kThreads>(P, stream);
    return usual ? launch_cluster<DT, 1, kThreads>(P, stream) : launch_cluster<DT, 1, 0>(P, stream);
}

template <int DT, int kDraw, int kCta>
bool wide_clusters()
{
    const unsigned threads = kCta ? kCta : kEdgeMostThreads;
    return allow_cluster(edge_cluster_kernel<DT, false, kDraw, kCta>, kEdgeClusterWide, threads) &&
           allow_cluster(edge_cluster_kernel<DT, true, kDraw, kCta>, kEdgeClusterWide, threads);
}
template <int DT>
bool wide_clusters()
{
    return wide_clusters<DT, 0, kThreads>() && wide_clusters<DT, 0, 0>() && wide_clusters<DT, 1, kThreads>() && wide_clusters<DT, 1, 0>() &&
           wide_clusters<DT, 2, kThreads>() && allow_cluster(edge_partial_cluster_kernel<DT, kThreads>, kEdgeClusterWide, kThreads) &&
           allow_cluster(edge_partial_cluster_kernel<DT, 0>, kEdgeClusterWide, kEdgeMostThreads);
}
int most_cluster_ctas()
{
    static PerContext most;
    return most.get([] {
        const bool wide = wide_clusters<DSSD_F32>() && wide_clusters<DSSD_BF16>();
        if (!wide) cudaGetLastError();
        return wide ? kEdgeClusterWide : kEdgeCluster;
    });
}

// at most c CTAs per sequence, no more than `wave` in all, at least one
long long fit(long long c, long long wave, int B)
{
    const long long most = wave / B;
    return c < most ? c : most > 1 ? most : 1;
}

// Threads per CTA and CTAs per sequence of the cluster kernel; false where the separate kernels are the better ones (edge_verify.h).
template <class Most>
bool cluster_shape(EdgeParams &P, int esz, long long segs, Most most_cluster_ctas)
{
    const long long parts = segs * (P.gamma + 1), B = P.B;
    if (P.gamma >= kFoldRows || parts > kEdgeClusterParts || (P.draw_token && P.V > 512 * kDrawSegs)) return false;
    const long long pieces = P.p_row || P.p_row16 || P.draw_token ? ((long long)P.V + 511) / 512 : 0, units = parts > pieces ? parts : pieces;
    const bool both = P.p_row && P.draw_token;
    const double work = (double)(parts * (esz == 2 ? 2 : 1)) + (pieces ? (double)P.V / 512.0 : 0.0), draw = both ? kEdgeDrawFactor : 1.0;
    auto is = [&](int cta, long long cluster) {
        P.cta = cta;
        P.cluster = (int)cluster;
        return true;
    };
    long long c = fit((units + kWarps - 1) / kWarps, kEdgeWave, P.B);
    if (c > kEdgeCluster) {
        const long long wide = fit(c, kEdgeWideWave, P.B);
        c = wide > kEdgeCluster ? wide : kEdgeCluster;
        if (c > kEdgeCluster && c > most_cluster_ctas()) c = most_cluster_ctas();
    }
    bool full = false;  // four or eight that find room as half as many CTAs of 512 threads
    while (c > 2 && c <= kEdgeCluster && B > kEdgeMostOf[c] && !full) {
        full = c % 4 == 0 && B * c <= kEdgeClusterWave && !P.draw_token;
        if (!full) --c;
    }
    if (c > 1 && 2 * c * B <= kEdgeSpread) {
        const long long most = most_cluster_ctas() < kEdgeSpreadCtas ? most_cluster_ctas() : kEdgeSpreadCtas, twice = 2 * c < most ? 2 * c : most;
        if (twice > c) c = twice;
    }
    if (c > kEdgeCluster && work > (P.shard_sum ? kEdgeWidePartial : kEdgeWideRounds) * (double)(kWarps * c)) c = kEdgeCluster;
    const bool held = draws_held(P, kThreads, c), draw_only = P.draw_token && !P.p_row;
    if (units > kEdgeBigUnits && kWarps * c < units && !held) {  // CTAs of 512 threads
        for (const auto &big : kEdgeBig) {
            if (B > (P.draw_token ? big.most_draw : big.most) || (big.ctas > kEdgeCluster && most_cluster_ctas() < big.ctas)) continue;
            const double warps = (double)(16 * big.ctas), limit = P.shard_sum ? big.shard : both ? big.both : draw_only ? big.draw : big.row;
            if (draw_only && c > kEdgeCluster && big.ctas > kEdgeCluster) break;
            if (2 * big.ctas > c && work <= limit * warps && (B > 1 || P.shard_sum || (double)parts <= (both ? 1.25 : 1.0) * warps))
                return is(kEdgeMostThreads, big.ctas);
            break;
        }
    }
    if (c > kEdgeCluster) return is(kThreads, c);
    if (!held && units >= (P.draw_token ? kEdgeSmallDrawUnits : kEdgeSmallUnits)) {  // CTAs of 128 threads
        for (const auto &small : kEdgeSmall) {
            if (B > small.most) continue;
            const double limit = P.shard_sum ? small.shard : both ? small.both : draw_only ? small.draw : small.row;
            if (units >= small.units && 4 * small.ctas > kWarps * c && work <= limit * (double)(4 * small.ctas)) return is(128, small.ctas);
            break;
        }
    }
    const long long ctas = B * c, waves = (ctas + kEdgeWave - 1) / kEdgeWave;
    const double fill = (double)ctas / (double)(waves * kEdgeWave);
    const double limit = P.shard_sum ? (fill >= 0.65 ? 8.0 : fill >= 0.5 ? 5.0 : 2.0)
                                     : (held || fill >= 0.65 ? draw : 1.0) * (fill >= 0.8 && c <= 4 ? 25.0 : fill >= 0.65 ? 14.0 : fill >= 0.5 ? 10.0 : 4.0);
    if (work > limit * (double)(kWarps * c)) return false;
    const bool pairs = P.shard_sum ? c % 2 == 0 : !P.draw_token && (full || (c == 2 && (B < kEdgeNoPairs || B > kEdgeNoPairsTo)));
    return pairs && ctas >= kEdgePairCtas ? is(kEdgeMostThreads, c / 2) : is(kThreads, c);
}

long long row_segments(int V, int esz)
{
    const long long nvec = (long long)V * esz / 16;
    return nvec > kSegVecs ? (nvec + kSegVecs - 1) / kSegVecs : 1;
}

template <int DT>
cudaError_t launch_edge(EdgeParams &P, unsigned lse_ctas, cudaStream_t stream)
{
    cudaError_t e = launch_pdl(edge_lse_kernel<DT>, lse_ctas, kLseThreads, stream, P);
    if (e != cudaSuccess) return e;
    const unsigned long long rows = (unsigned long long)P.B * (unsigned long long)(P.gamma + 1);
    const bool wide = P.runs > kFoldWide;
    if (P.shard_sum)
        return wide ? launch_pdl(edge_partial_kernel<true>, (unsigned)((rows + kWarps - 1) / kWarps), kThreads, stream, P)
                    : launch_pdl(edge_partial_kernel<false>, (unsigned)((rows + kFoldRows - 1) / kFoldRows), kThreads, stream, P);
    const bool emit = P.p_row || P.p_row16;
    const bool aligned = outputs_aligned<DT>(P);
    P.emit_tiles = emit_tiles(P.V, aligned);
    const unsigned long long ctas = (unsigned long long)P.B * (unsigned long long)P.emit_tiles;
    if (ctas > 0x7fffffffull) return cudaErrorInvalidConfiguration;
    const bool fold = emit && ctas <= kEmitFoldCtas && !wide;
    if (!fold) {
        e = wide ? launch_pdl(edge_fold_kernel<true>, (unsigned)P.B, kThreads, stream, P)
                 : launch_pdl(edge_fold_kernel<false>, (unsigned)P.B, kThreads, stream, P);
        if (e != cudaSuccess || !emit) return e;
    }
    return aligned ? launch_emit<DT, false>(P, (unsigned)ctas, fold, stream) : launch_emit<DT, true>(P, (unsigned)ctas, fold, stream);
}

}  // namespace

void edge_shape_chosen(EdgeParams &P, int dtype)
{
    const int esz = dtype == DSSD_BF16 ? 2 : 4;
    P.cta = P.cluster = 0;
    if (!cluster_shape(P, esz, row_segments(P.V, esz), [] { return kEdgeClusterWide; })) P.cta = P.cluster = 0;
}

cudaError_t edge_verify_launch(EdgeParams &P, int dtype, void *workspace, cudaStream_t stream)
{
    const int esz = dtype == DSSD_BF16 ? 2 : 4;
    const unsigned long long rows = (unsigned long long)P.B * (unsigned long long)(P.gamma + 1);
    P.c1 = (float)(1.4426950408889634 / (double)P.temperature);
    const long long nvec = (long long)P.V * esz / 16;
    const long long segs = row_segments(P.V, esz);
    P.cluster = 0;
    if (cluster_shape(P, esz, segs, most_cluster_ctas)) {
        edge_workspace_layout(P.B, P.gamma, 1, &P, static_cast<char *>(workspace));  // (the partial sums stay on the chip)
        P.runs = (int)segs;
        return dtype == DSSD_BF16 ? launch_cluster<DSSD_BF16>(P, stream) : launch_cluster<DSSD_F32>(P, stream);
    }
    const unsigned long long tiles = rows * (unsigned long long)((nvec + kLseTile - 1) / kLseTile);
    const long long per = tiles < kLseTwoTiles ? 1 : tiles < kLseFourTiles ? 2 : 4;
    long long runs = (nvec + per * kLseTile - 1) / (per * kLseTile);
    if (runs < 1) runs = 1;
    P.run_vecs = (int)(per * kLseTile);
    P.runs = (int)runs;
    if (rows * (unsigned long long)runs > 0x7fffffffull) return cudaErrorInvalidConfiguration;
    edge_workspace_layout(P.B, P.gamma, P.runs, &P, static_cast<char *>(workspace));
    const unsigned lse_ctas = (unsigned)(rows * (unsigned long long)runs);
    return dtype == DSSD_BF16 ? launch_edge<DSSD_BF16>(P, lse_ctas, stream) : launch_edge<DSSD_F32>(P, lse_ctas, stream);
}

}  // namespace dssd
