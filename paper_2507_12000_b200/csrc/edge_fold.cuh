// Folding a sequence: the runs' partial sums -> every row's log-sum-exp -> acceptance tests -> the
// first rejection.  Done by every CTA that needs the verdict on a sequence: it costs one round
// trip to L2 and a few hundred instructions, less than handing the verdict on in another launch.
#pragma once

#include "dssd_device.cuh"
#include "edge_judge.cuh"
#include "edge_verify.h"

namespace dssd {

constexpr unsigned long long kNoPartial = ~0ull;  // stored in place of a withheld partial sum (a sum is never this NaN)
constexpr int kFoldLanes = 8;                     // threads that add up one row's runs
constexpr int kFoldRows = kThreads / kFoldLanes;  // rows folded at a time
static_assert(kFoldRows == 32, "one lane of warp 0 per position");

struct FoldShared {
    float R[kFoldRows];
    double S[kFoldRows];
    int missing[kFoldRows];
    int n;                // accepted length; -1: no verdict
    float ref2, invS;     // row n
};

// The sum of one row, formed by kFoldLanes neighbouring threads (sub = 0 .. kFoldLanes - 1 within the row):
// the largest reference first, then float64 terms s * 2^(ref - R) by exponent arithmetic, added in a fixed
// order.  The result, sum_v 2^(l_v c1) = S * 2^R, is the same in all threads of the row; a NaN or an
// infinite sum stays one, a row without mass gives S = 0.  Short, because every emission CTA of a small
// launch runs it.  part(k) loads run k's word.
template <class Part>
__device__ __forceinline__ void row_total(Part part, int runs, int sub, bool live, float &R, double &S, bool &missing)
{
    constexpr int kHeld = 2;  // words in registers: rows of up to 16 runs need no second look
    unsigned long long w[kHeld];
    float top = DSSD_NEG_INF;
    missing = false;
    auto word = [&](int k) { return live && k < runs ? part(k) : 0ull; };
    auto look = [&](unsigned long long x) {
        missing |= x == kNoPartial;
        if (__uint_as_float((unsigned)(x >> 32)) > 0.f) top = fmaxf(top, __uint_as_float((unsigned)x));
    };
#pragma unroll
    for (int u = 0; u < kHeld; ++u) w[u] = word(u * kFoldLanes + sub);
#pragma unroll
    for (int u = 0; u < kHeld; ++u) look(w[u]);
    for (int k = kHeld * kFoldLanes + sub; k < runs; k += kFoldLanes) look(word(k));
#pragma unroll
    for (int o = 1; o < kFoldLanes; o <<= 1) top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, o));
    double s = 0.0;
    auto add = [&](unsigned long long x) {
        const float v = __uint_as_float((unsigned)(x >> 32));
        if (v > 0.f && v < INFINITY) s += scale_pow2((double)v, __uint_as_float((unsigned)x) - top);
        else if (v != 0.f) s += (double)v;
    };
#pragma unroll
    for (int u = 0; u < kHeld; ++u) add(w[u]);
    for (int k = kHeld * kFoldLanes + sub; k < runs; k += kFoldLanes) add(word(k));
#pragma unroll
    for (int o = 1; o < kFoldLanes; o <<= 1) {
        s += __shfl_xor_sync(0xffffffffu, s, o);
        missing |= __shfl_xor_sync(0xffffffffu, (int)missing, o) != 0;
    }
    R = top;
    S = s;
}

// The same by a whole warp, for rows of hundreds of runs: 256 words on their way at a time.
constexpr int kFoldWide = 64;  // runs beyond which it is used, by kernels of their own (edge_verify.cu: launch_edge)
template <class Part>
__device__ __forceinline__ void row_total_wide(Part part, int runs, float &R, double &S, bool &missing)
{
    const int lane = threadIdx.x & 31;
    float top = DSSD_NEG_INF;
    double s = 0.0;
    missing = false;
    auto all = [&](auto use) {
        for (int k0 = lane; k0 < runs; k0 += 256) {
            unsigned long long x[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) x[u] = k0 + 32 * u < runs ? part(k0 + 32 * u) : 0ull;
#pragma unroll
            for (int u = 0; u < 8; ++u) use(x[u]);
        }
    };
    all([&](unsigned long long x) {
        missing |= x == kNoPartial;
        if (__uint_as_float((unsigned)(x >> 32)) > 0.f) top = fmaxf(top, __uint_as_float((unsigned)x));
    });
    top = warp_max(top);
    all([&](unsigned long long x) {
        const float v = __uint_as_float((unsigned)(x >> 32));
        if (v > 0.f && v < INFINITY) s += scale_pow2((double)v, __uint_as_float((unsigned)x) - top);
        else if (v != 0.f) s += (double)v;
    });
    S = warp_sum(s);
    R = top;
    missing = __any_sync(0xffffffffu, missing);
}

// What the acceptance test of a position takes besides its row's sum.
struct Drafted {
    int x;          // the drafted token
    float z, q, u;  // its logit in the row, its draft probability, the position's uniform
};

// Run by all threads of a CTA, kCta of them (0: as many as were launched, 128 or at least kThreads); the results are in `sh` (n, ref2, invS)
// when it returns.
// `writer`: this CTA writes the sequence's accept_len, flags, lse, p_tok and `ready`.
// part(i, k) gives the partial sum of run k of row i of the sequence, drafted(i) what belongs to position i.
template <bool kWide, int kCta, class Part, class Draft>
__device__ __forceinline__ void fold_sequence(const EdgeParams &P, long long b, bool writer, FoldShared &sh, Part part, Draft drafted)
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int n = P.gamma;
    unsigned fl = 0;
    float ref2_n = 0.f, invS_n = 0.f;
    for (int base = 0; base <= P.gamma; base += kFoldRows) {
        if (base) __syncthreads();  // warp 0 has read the previous rows
        const int i = base + lane;
        const bool live = i <= P.gamma;
        Drafted d = {-1, 0.f, 0.f, 0.f};
        if (warp == 0 && i < P.gamma) d = drafted(i);
        if (kWide) {
            for (int w = warp; w < kFoldRows && base + w <= P.gamma; w += kWarps) {
                float R;
                double S;
                bool missing;
                row_total_wide([&](int k) { return part(base + w, k); }, P.runs, R, S, missing);
                if (lane == 0) {
                    sh.R[w] = R;
                    sh.S[w] = S;
                    sh.missing[w] = missing;
                }
            }
        } else {
            auto total = [&](int w) {
                const int r = base + w;
                float R;
                double S;
                bool missing;
                row_total([&](int k) { return part(r, k); }, P.runs, tid % kFoldLanes, r <= P.gamma, R, S, missing);
                if (tid % kFoldLanes == 0) {
                    sh.R[w] = R;
                    sh.S[w] = S;
                    sh.missing[w] = missing;
                }
            };
            if (kCta || tid < kThreads) total(tid / kFoldLanes);
            if (!kCta && blockDim.x < kThreads && base + kFoldRows / 2 <= P.gamma) total(tid / kFoldLanes + kFoldRows / 2);  // 128 threads: half of the rows at a time
        }
        __syncthreads();
        if (warp == 0) {
            if (P.draft_q_rows && (d.x < 0 || d.x >= P.V)) d.q = __int_as_float(0x7fc00000);  // nothing was looked up
            float Rs, invS;
            const unsigned bits = judge_position(P, b, i, live, writer, sh.R[lane], sh.S[lane], false, live && sh.missing[lane],
                                                 d.x, d.z, d.q, d.u, Rs, invS);
            const unsigned rej = __ballot_sync(0xffffffffu, live && i < P.gamma && !(bits & kBitAccept));
            if (rej && n == P.gamma) n = base + __ffs(rej) - 1;
            fl |= (__ballot_sync(0xffffffffu, bits & kBitBadToken) ? DSSD_EDGE_FLAG_BAD_TOKEN : 0u) |
                  (__ballot_sync(0xffffffffu, bits & kBitNonFinite) ? DSSD_EDGE_FLAG_NONFINITE : 0u) |
                  (__ballot_sync(0xffffffffu, bits & kBitTimeout) ? DSSD_EDGE_FLAG_TIMEOUT : 0u);
            if (n >= base && n < base + 32) {
                ref2_n = __shfl_sync(0xffffffffu, Rs, n - base);
                invS_n = __shfl_sync(0xffffffffu, invS, n - base);
            }
        }
    }
    if (tid == 0) {
        if (fl & DSSD_EDGE_FLAG_TIMEOUT) n = -1;
        sh.n = n;
        sh.ref2 = ref2_n;
        sh.invS = invS_n;
        if (writer) {
            P.accept_len[b] = n;
            if (P.accept_copy) P.accept_copy[b] = n;
            if (P.flags) P.flags[b] = fl;
            ReadySlot s;
            s.b = (int)b;
            s.n = n;
            s.ref2 = ref2_n;
            s.invS = invS_n;
            P.ready[b] = s;
        }
    }
    __syncthreads();
}

// The same with what the log-sum-exp kernel left in the workspace: one round trip to L2 for the partial sums,
// the drafted tokens' logits and the caller's arrays.
template <bool kWide>
__device__ __forceinline__ void fold_sequence(const EdgeParams &P, long long b, bool writer, FoldShared &sh)
{
    const long long row0 = b * (P.gamma + 1);
    fold_sequence<kWide, kThreads>(P, b, writer, sh, [&](int i, int k) { return ld_after(P.part + (size_t)(row0 + i) * P.runs + k); },
                  [&](int i) {
                      const size_t di = (size_t)b * P.gamma + i;
                      Drafted d;
                      d.x = ld_after(P.draft_tokens + di);
                      d.q = P.draft_q_rows ? ld_after(P.tokq + row0 + i) : ld_after(P.draft_q_tok + di);
                      d.u = ld_after(P.uniforms + di);
                      d.z = ld_after(P.tokz + row0 + i);
                      return d;
                  });
}

}  // namespace dssd
