// The vocabulary-sharded round: what happens between and after the shards' partial sums.
//
// Every shard runs the streaming edge kernel on its slice of the logits in "partial" mode and
// gets, per row, sum_v 2^(l_v c1) = part_sum * 2^part_ref over its slice, plus the logits of the
// drafted tokens it holds.  Once these small arrays have been exchanged (an all-gather of a few
// bytes per row), shard_combine_kernel - one warp per sequence, one lane per position - adds the
// shards' sums by exact power-of-two rescaling and evaluates the acceptance test and the
// first-rejection scan with the same arithmetic as the dense kernel's fold.  shard_emit_kernel
// then writes this shard's slice of row P_n.
#include "shard_verify.h"

#include "dssd_device.cuh"
#include "edge_judge.cuh"
#include "emit.cuh"
#include "launch.h"

namespace dssd {

namespace {

constexpr unsigned kFull = 0xffffffffu;

__global__ void __launch_bounds__(kThreads) shard_combine_kernel(const __grid_constant__ CombineParams P)
{
    const int lane = threadIdx.x & 31;
    const long long b = (long long)blockIdx.x * kWarps + (threadIdx.x >> 5);
    pdl_wait();
    pdl_trigger();
    if (b >= P.B) return;
    const size_t rows = (size_t)P.B * (size_t)(P.gamma + 1), toks = (size_t)P.B * (size_t)P.gamma;
    constexpr int kAtOnce = 8;  // shards whose values are requested together
    int n = P.gamma;
    unsigned fl = 0;
    float ref2_n = 0.f, invS_n = 0.f;
    for (int base = 0; base <= P.gamma; base += 32) {
        const int i = base + lane;
        const bool live = i <= P.gamma, tested = i < P.gamma;
        const size_t row = (size_t)b * (size_t)(P.gamma + 1) + (size_t)(live ? i : 0);
        const size_t di = (size_t)b * P.gamma + (tested ? i : 0);
        int x = -1;
        float zx = __int_as_float(0x7fc00000), qx = 0.f, ux = 0.f;
        if (tested) {
            x = ld_after(P.draft_tokens + di);
            qx = ld_after(P.draft_q_tok + di);
            ux = ld_after(P.uniforms + di);
        }
        float Rr = DSSD_NEG_INF;
        double S = 0.0;
        bool bad = false;
        for (int g0 = 0; g0 < P.G; g0 += kAtOnce) {
            float z[kAtOnce], r[kAtOnce];
            double s[kAtOnce];
#pragma unroll
            for (int k = 0; k < kAtOnce; ++k) {
                const size_t g = (size_t)(g0 + k);
                z[k] = __int_as_float(0x7fc00000);
                r[k] = 0.f;
                s[k] = 0.0;
                if (g0 + k < P.G && tested) z[k] = ld_after(P.tok_logit + g * toks + di);
                if (g0 + k < P.G && live) {
                    r[k] = ld_after(P.part_ref + g * rows + row);
                    s[k] = ld_after(P.part_sum + g * rows + row);
                }
            }
#pragma unroll
            for (int k = 0; k < kAtOnce; ++k) {  // shard order
                if (z[k] == z[k]) zx = z[k];     // the one shard that holds x reports its logit, the others NaN
                add_partial(Rr, S, bad, r[k], s[k]);
            }
        }
        float Rs, invS;
        const unsigned bits = judge_position(P, b, i, live, true, Rr, S, bad, false, x, zx, qx, ux, Rs, invS);
        const unsigned rej = __ballot_sync(kFull, live && i < P.gamma && !(bits & kBitAccept));
        if (rej && n == P.gamma) n = base + __ffs(rej) - 1;
        fl |= (__ballot_sync(kFull, bits & kBitBadToken) ? DSSD_EDGE_FLAG_BAD_TOKEN : 0u) |
              (__ballot_sync(kFull, bits & kBitNonFinite) ? DSSD_EDGE_FLAG_NONFINITE : 0u);
        if (n >= base && n < base + 32) {
            ref2_n = __shfl_sync(kFull, Rs, n - base);
            invS_n = __shfl_sync(kFull, invS, n - base);
        }
    }
    if (lane == 0) {
        P.accept_len[b] = n;
        if (P.flags) P.flags[b] = fl;
        P.row_scale[2 * b] = ref2_n;
        P.row_scale[2 * b + 1] = invS_n;
    }
}

// p_row[b, v] = 2^(l_{b,n,v} c1 - ref2) / S over this shard's slice of row n, one tile per CTA.
template <int DT, bool kShift>
__global__ void __launch_bounds__(kThreads) shard_emit_kernel(const __grid_constant__ EmitShardParams P)
{
    const long long b = blockIdx.x / (unsigned)P.tiles;
    const int tile = (int)(blockIdx.x - (unsigned)b * (unsigned)P.tiles);
    pdl_wait();
    pdl_trigger();
    const int n = ld_after(P.accept_len + b);
    const float ref2 = ld_after(P.row_scale + 2 * b), invS = ld_after(P.row_scale + 2 * b + 1);
    if (n < 0 || n > P.gamma) return;
    const char *rowp = static_cast<const char *>(P.logits) +
                       ((size_t)b * (size_t)(P.gamma + 1) + (size_t)n) * (size_t)P.row_stride * Elem<DT>::kBytes;
    emit_tile<DT, kShift>(rowp, P.p_row + (size_t)b * (size_t)P.p_stride, P.V, tile, P.c1, ref2, invS);
}

}  // namespace

cudaError_t shard_combine_launch(const CombineParams &P, cudaStream_t stream)
{
    return launch_pdl(shard_combine_kernel, (unsigned)((P.B + kWarps - 1) / kWarps), kThreads, stream, P);
}

template <int DT>
static cudaError_t emit_launch(EmitShardParams &P, cudaStream_t stream)
{
    const bool aligned = emit_aligned(P.logits, P.row_stride, Elem<DT>::kBytes, P.p_row, P.p_stride, 4);
    P.tiles = emit_tiles(P.V, aligned);
    const unsigned long long grid = (unsigned long long)P.B * (unsigned long long)P.tiles;
    if (grid > 0x7fffffffull) return cudaErrorInvalidConfiguration;
    return aligned ? launch_pdl(shard_emit_kernel<DT, false>, (unsigned)grid, kThreads, stream, P)
                   : launch_pdl(shard_emit_kernel<DT, true>, (unsigned)grid, kThreads, stream, P);
}

cudaError_t shard_emit_launch(EmitShardParams &P, int dtype, cudaStream_t stream)
{
    return dtype == DSSD_BF16 ? emit_launch<DSSD_BF16>(P, stream) : emit_launch<DSSD_F32>(P, stream);
}

}  // namespace dssd
