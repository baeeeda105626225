// Device half of the verification round: residual (or bonus) inverse-CDF draw, as two kernels, or as one where
// the batch is small (resample_cluster_kernel: a cluster of CTAs per sequence holds the row in registers) or of middle
// size (resample_stream_kernel: it goes over the row in turns).
//
//   resample_mass_kernel  one CTA per (sequence, one to four tiles of kTile entries): streams its part of
//                         p_row[b] and of Q_n[b], forms r = max(0, p - q) (or r = p for the bonus draw)
//                         and adds it up in float64: one sum per chunk of kResampleSub entries.
//   resample_draw_kernel  one CTA per sequence: a float64 prefix over the sequence's chunk sums gives Z
//                         and the chunk that holds u' * Z; every thread fetches its run of that chunk, a
//                         second prefix finds the thread and its run gives the token.
//
// Plain stores and the order of the launches (launch.h) connect them; nothing in the scratch has to be
// cleared.
// All sums are float64, so the token differs from an index-order float64 scan only when u' * Z
// lies within rounding (about 1e-13 relative) of a CDF step.
#include "device_resample.h"

#include <mutex>

#include <math.h>

#include "draw.cuh"
#include "dssd_device.cuh"
#include "launch.h"

namespace dssd {

namespace {

constexpr int kSub = kResampleSub;      // entries per chunk sum
constexpr int kRows = 4;                 // chunks per tile
constexpr int kTile = kRows * kSub;      // entries that a CTA streams at a time
static_assert(2 * kRows == kWarps && kSub == 2 * 512, "a warp of the mass kernel streams half a chunk, 512 entries");
// Tiles per CTA of the mass kernel.  Few tiles: one each, so that all SMs share them.  More than about
// one and a half waves of 740 resident CTAs: two, more than six waves: four, which pays for a CTA's
// start and its reduction less often.  Measured (us, mass kernel with the draw behind it; 1 / 2 / 4 tiles):
// B = 256 V = 151936 (9728 tiles) 45.7 / 45.0 / 41.7, B = 64 V = 128256 (2048) 21.4 / 21.4 / 32.1,
// B = 8 V = 32000 (64) 7.9 / 8.7 / 10.2.
constexpr unsigned long long kTwoTiles = 1200, kFourTiles = 4800;
constexpr int kClusterThreads = 512;     // most threads per CTA of the cluster kernel
constexpr int kClusterMax = 8;           // most CTAs per cluster: the portable size,
constexpr int kClusterWide = 16;         // and where the device has them
constexpr int kClusterSums = kClusterMax * kClusterThreads / 32;
// Small draws: one launch whose warps hold the row, 512 entries each (resample_cluster_kernel), while about one wave of the CTAs holds
// the batch; at 128 registers that is 2368 warps, less for large clusters, which do not pack the GPU's processing
// clusters completely.  The smallest CTAs that fit one cluster of sixteen leave the fewest warps idle and start soonest.
// Measured (us per call, this / the two kernels):
//   a CTA per sequence:  B = 1000 V = 1024 4.7 / 12.4, B = 1000 V = 2000 7.9 / 12.6, B = 600 V = 4001 10.7 / 11.9; beyond, B = 1000
//              V = 4001 16.1 / 15.1
//   clusters of 128 threads:  B = 168 V = 5460 (3 CTAs) 4.1 / 6.3, B = 59 V = 13786 (7) 4.2 / 6.7, B = 46 V = 16436 (9) 4.2 / 5.9;
//              beyond, B = 46 V = 28992 (15, 690 CTAs) 6.7 / 6.1, B = 175 V = 11384 (6) 7.8 / 6.1
//   of 256:  B = 7 V = 57700 (15) 4.3 / 6.1, of 512:  B = 2 V = 96209 (12) 4.3 / 5.9, B = 6 V = 105317 (13) 4.5 / 6.1, B = 4
//              V = 129300 (16) 4.6 / 5.1; beyond, B = 21 V = 82900 (11) 12.5 / 7.2.  In rounds too (a CTA of 512 threads has its SM to itself, so that a
//              cluster starts when up to sixteen SMs of one processing cluster are free): gamma = 4, B = 1 V = 96209 float32 11.3 / 13.4, B = 4 V = 128256 bf16
//              12.7 / 13.7, B = 8 V = 66000 12.4 / 14.5.  While another stream keeps the GPU busy a launch waits for its CTAs' room, one for
//              more of it, two twice (the latency of a round, B = 1 V = 96209, B = 2 V = 128256 and B = 4 V = 128256: beside products of 4096 x 4096 bf16 62 / 31, 67 / 41,
//              67 / 68 us, beside products of 2048 x 1024 19 / 22, 19 / 20, 21 / 22, beside copies of a GB 295 / 617, 297 / 618, 298 / 617).
constexpr long long kSingleThreads = 153600;
// More than eight CTAs of 128 threads only for a few sequences: many of them do not find room before the kernel before has drained (a round
// of B = 23 gamma = 7 V = 23912 bf16, twelve CTAs 13.0 us, six of 256 threads 12.5; B = 8 gamma = 4 V = 32000 bf16, sixteen 9.3, eight 9.5).
constexpr long long kHeldWideCtas = 148;
constexpr long long kHeldWarps = 2250, kHeldWideWarps = 1650, kHeldWidestWarps = 1250;  // up to eight CTAs, more, more of 512 threads
// Batches of middle size: the same in turns (resample_stream_kernel), in which a CTA's or cluster's start, its barrier and the walk are
// paid for once while the other CTAs on the SM stream.  For rows of up to kStreamSegs segments, at most kStreamTurns of them per warp:
// as many warps as there are segments while kStreamOne of them suffice, else as many as a wave of whole CTAs has (32 or 40 warps per
// SM: six CTAs of six warps, not seven: B = 915 V = 12480 in five turns by five warps, by six 20.8 us, two kernels 18.2), seven tenths of that in clusters.  Measured (us per call, this / the two kernels): B = 164 V = 9856
// 5.6 / 6.5, B = 331 V = 4384 binary16 6.7 / 10.6, B = 425 V = 5800 7.5 / 9.3, B = 714 V = 3728 6.4 / 9.1, B = 567 V = 11886 11.7 / 15.3,
// B = 665 V = 12640 12.8 / 15.6, B = 305 V = 15760 binary16 9.8 / 12.5, B = 143 V = 19400 7.8 / 9.4; beyond, B = 67 V = 32592 7.0 / 6.6,
// B = 100 V = 43015 13.3 / 12.2, B = 55 V = 124034 14.4 / 10.5.  The two kernels are the better ones for
//   clusters of more warps than kStreamClusters in all (B = 383 V = 23016 15.2 / 13.5, B = 290 V = 19376 by four CTAs 10.6 / 9.6, B = 195 V = 10576 by six 8.3 /
//   6.5; with fewer CTAs B = 330 V = 23040 11.9 / 13.1), of three CTAs from kStreamThrees sequences on (a round of B = 340 V = 15924 26.7, by one CTA of 256 threads 24.7, two
//   kernels 24.5) and of five of 256 threads (a round of B = 105 V = 17084 17.4, by five of 128 15.2, two kernels 14.9),
//   rows of more than kStreamTurnsFew turns by one CTA each that leave a third of the wave empty (B = 400 V = 18218 16.2 / 14.3, B = 352 V = 19047 17.3 / 13.6; in four
//   turns B = 416 V = 12881 12.4 / 14.2, B = 385 V = 15189 12.6 / 13.1, B = 421 V = 15520 11.7 / 10.5),
//   few long rows that need more than a segment per warp (B = 92 V = 20030 8.3 / 7.1 and B = 133 V = 15897 8.8 / 7.4 off the 16-byte boundaries, B = 107 V = 22920
//   7.2 / 6.4 on them), and most rows of more than 32 segments with one each (B = 105 V = 17034 9.0 / 7.5; B = 90 V = 18316 6.1 / 6.3).
// Up to sixteen segments by eight warps in two turns, not by as many warps as segments, from kStreamHalf sequences on: B = 340 V = 4608 6.5 / 8.0, B = 318 V =
// 4880 6.9 / 8.3; below, B = 290 V = 5120 6.3 / 5.9, B = 251 V = 4608 6.4 / 5.7.
constexpr int kStreamSegs = 45, kStreamTurns = 5, kStreamTurnsFew = 4;
constexpr long long kStreamOne = 3600, kStreamOneLong = 3300, kStreamHalf = 300, kStreamClusters = 4200, kStreamThrees = 333;
constexpr long long kStreamFew = 150;                              // sequences, of at most
constexpr int kStreamFewSegs = 41, kStreamFewSegsShifted = 29;     // segments, on and off the boundaries of 16 bytes
constexpr int kDrawThreads = 128;        // threads that draw for a sequence
constexpr int kDrawWarps = kDrawThreads / 32;
constexpr int kRun = kSub / kDrawThreads;  // entries of a chunk per thread

// r for thread t's run of the chunk that starts at entry e0: entries e0 + kRun * t + j in r[j]; 0 beyond the
// row's end.  All loads are requested before the first is used.
template <bool kHasQ, bool kShift, typename RV>
__device__ __forceinline__ void load_run(const RV &row, const float *q, int V, int e0, double (&r)[kRun])
{
    const long long first = (long long)e0 + kRun * (int)threadIdx.x;
    ThreadQuads<typename RV::Q, kRun / 4, kShift> a;
    ThreadQuads<Quads32, kRun / 4, kShift> b;
    a.load(row.row, V, first, RV::kFill);
    if (kHasQ) b.load(reinterpret_cast<const char *>(q), V, first, 0u);
#pragma unroll
    for (int u = 0; u < kRun / 4; ++u) {
        const float4 x = row.quad(a.at(u));
        const float4 y = kHasQ ? as_f4(b.at(u)) : make_float4(0.f, 0.f, 0.f, 0.f);
        r[4 * u] = kHasQ ? res(x.x, y.x) : (double)x.x;
        r[4 * u + 1] = kHasQ ? res(x.y, y.y) : (double)x.y;
        r[4 * u + 2] = kHasQ ? res(x.z, y.z) : (double)x.z;
        r[4 * u + 3] = kHasQ ? res(x.w, y.w) : (double)x.w;
    }
}

// is a sequence with accepted length n (0 <= n <= gamma) one this launch draws for?
__device__ __forceinline__ bool selected(const ResampleParams &P, int n)
{
    return P.select == 0 || (P.select == 1 ? n == P.gamma : n < P.gamma);
}

// The draw inside the picked chunk, which starts at entry e0, by the whole CTA: the token is the first entry whose
// running mass exceeds the target, else (rounding, or pk.beyond) the last one with mass; -1 when
// the chunk has none.  `base` moves on by the chunk's mass; `hit`: the target was exceeded.  The result is
// the same in all threads.  q == nullptr means r = p.
struct WalkShared {
    double sum[kDrawWarps];
    int tok[kDrawWarps];   // the warp's token; hit in bit 30
};
template <bool kShift, typename RV>
__device__ __forceinline__ int walk_chunk(const Pick &pk, const RV &row, const float *q, int V, int e0, double &base, bool &hit,
                                          WalkShared &sh)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double r[kRun], pre[kRun];
    if (q) load_run<true, kShift>(row, q, V, e0, r);
    else load_run<false, kShift>(row, q, V, e0, r);
    unsigned positive = 0;
    double mine = 0.0;
#pragma unroll
    for (int j = 0; j < kRun; ++j) {
        mine += r[j];
        pre[j] = mine;
        positive |= r[j] > 0.0 ? 1u << j : 0u;
    }
    const double incl = warp_scan(mine);
    __syncthreads();  // (an earlier chunk's results have been read)
    if (lane == 31) sh.sum[warp] = incl;
    __syncthreads();
    double before = base;
#pragma unroll
    for (int w = 0; w < kDrawWarps; ++w) {
        if (w == warp) before = base;
        base += sh.sum[w];
    }
    const double up = __shfl_up_sync(0xffffffffu, incl, 1);
    const double C = before + (lane ? up : 0.0);
    unsigned over = 0;
#pragma unroll
    for (int j = 0; j < kRun; ++j) over |= !pk.beyond && C + pre[j] > pk.target ? 1u << j : 0u;
    over &= positive;
    const unsigned cross = __ballot_sync(0xffffffffu, over != 0), mass = __ballot_sync(0xffffffffu, positive != 0);
    const int owner = cross ? __ffs(cross) - 1 : mass ? 31 - __clz(mass) : 0;
    int t = -1;
    if (positive) t = e0 + kRun * (int)threadIdx.x + (over ? __ffs(over) - 1 : 31 - __clz(positive));
    if (lane == owner) sh.tok[warp] = t < 0 ? -1 : cross ? t | (1 << 30) : t;
    __syncthreads();
    // the first warp that crosses, else the last with mass
    int tok = -1;
    hit = false;
#pragma unroll
    for (int w = 0; w < kDrawWarps; ++w) {
        const int x = sh.tok[w];
        if (x >= 0 && !hit) {
            tok = x & ~(1 << 30);
            hit = (x >> 30) & 1;
        }
    }
    return tok;
}

// The pick among n_sub chunks; kLong: there are many more than a warp's lanes keep.  (A draw of V = 300000, 293 sums: 7.5 us without,
// 7.9 with; V = 1048576, 1024 sums: 10.4 and 8.7.)
constexpr int kLongSums = 512;
template <bool kLong, class Sum, class Target>
__device__ __forceinline__ Pick pick_of(const LaneSums &L, Sum sum, bool beyond, Target target)
{
    if constexpr (kLong) return pick_long(L, sum, beyond, target);
    else return pick_chunk(L, sum, beyond, target);
}

// The draw for sequence b by one CTA; q == nullptr means r = p.
template <bool kLong, bool kShift, typename RV>
__device__ void draw(const ResampleParams &P, int64_t b, const RV &row, const float *q, unsigned fl, float u, LaneSums &L,
                     WalkShared &sh)
{
    const int tid = threadIdx.x, lane = tid & 31;
    const int width = P.rows_per_sum * kSub;  // entries per stored sum
    double *cs = P.chunk_sum + (size_t)b * P.n_sub;
    auto sum = [&](int c) { return ld_after(cs + c); };
    auto target = [&](double Z) { return (double)u * Z; };
    Pick pk = pick_of<kLong>(L, sum, false, target);
    if (!pk.ok && !pk.late && q) {
        // The residual has no mass (p == q): draw from p instead.  Rare, so its sums are formed here, a warp
        // at each, where the others were.
        q = nullptr;
        fl |= DSSD_RS_FLAG_FALLBACK;
        __syncthreads();  // every warp has read the sums that are replaced now
        for (int c = tid >> 5; c < P.n_sub; c += kDrawWarps) {
            double tot = 0.0, none;
            for (int e = 0; e < width; e += 512) tot += share_mass<false, false, kShift>(row, q, P.V, (long long)c * width + e, none);
            tot = warp_sum(tot);
            if (lane == 0) cs[c] = tot;
        }
        __syncthreads();
        load_sums(L, P.n_sub, sum);
        pk = pick_of<kLong>(L, sum, false, target);
    }
    int tok = -1;
    if (pk.ok && !pk.late) {
        double base = pk.base;
        bool hit = false;
        for (int k = 0; k < P.rows_per_sum && !hit; ++k) {
            const long long e0 = (long long)pk.chunk * width + k * kSub;
            if (e0 >= P.V) break;
            const int t = walk_chunk<kShift>(pk, row, q, P.V, (int)e0, base, hit, sh);
            if (t >= 0) tok = t;
        }
    }
    if (tid == 0) {
        P.token[b] = tok;
        if (P.flags) P.flags[b] = fl | (tok < 0 ? DSSD_RS_FLAG_INVALID : 0u) | (pk.late ? DSSD_RS_FLAG_TIMEOUT : 0u);
    }
}

// Bound by HBM and L2: 231 MB of rows at B = 256 V = 151936 in 32 us (a quarter of p_row from L2), where the
// persistent kernel it replaces, with tickets, a cleared scratch and the draws at its end, took 41 us
// with them; B = 1 V = 50272: 6.5 us for both kernels against 8.9.  48 registers, so five CTAs share an SM
// and one CTA's reduction lies under the others' loads (four: 36.1 us).
template <bool kShift, typename RV>
__global__ void __launch_bounds__(kThreads, kShift ? 4 : 5) resample_mass_kernel(const __grid_constant__ ResampleParams P)
{
    __shared__ double s_w[kResampleMaxTiles * kRows][2];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // in index order: the edge kernel emits the rows from the last sequence backwards, so the first ones
    // are still in L2 when they were written just before
    const unsigned t = blockIdx.x;
    const int64_t b = t / (unsigned)P.n_ctas;
    const int first = (int)(t - (unsigned)b * (unsigned)P.n_ctas) * P.tiles;  // the CTA's first tile
    pdl_wait();
    pdl_trigger();
    const int n = ld_after(P.accept_len + b);
    if (n < 0 || n > P.gamma || !selected(P, n)) return;  // the draw does not read this sequence's sums
    const RV row = RV::make(P, b, n);
    const float *q = n < P.gamma ? P.draft_q + ((size_t)b * P.gamma + n) * (size_t)P.V : nullptr;
    const int tiles = min(P.tiles, (P.V + kTile - 1) / kTile - first);
    for (int k = 0; k < tiles; ++k) {
        const long long base = (long long)(first + k) * kTile + warp * 512;
        double acc, none;
        if (q) acc = share_mass<true, false, kShift>(row, q, P.V, base, none);
        else acc = share_mass<false, false, kShift>(row, q, P.V, base, none);
        acc = warp_sum(acc);
        if (lane == 0) s_w[k * kRows + (warp >> 1)][warp & 1] = acc;
    }
    __syncthreads();
    const int sums = tiles * kRows / P.rows_per_sum;
    if (tid < sums) {
        const int c = first * kRows / P.rows_per_sum + tid;
        double tot = 0.0;
        for (int k = 0; k < P.rows_per_sum; ++k) tot += s_w[tid * P.rows_per_sum + k][0] + s_w[tid * P.rows_per_sum + k][1];
        if (b + 1 == (int64_t)P.test_drop_seq_plus1) tot = __longlong_as_double((long long)kNoSum);
        if (c < P.n_sub) P.chunk_sum[(size_t)b * P.n_sub + c] = tot;
    }
}

// One CTA per sequence.  Bound by latency: one round trip for the sums, one for the chunk, and the float64
// additions that depend on one another (4 us at B = 256; a chunk of 4096 entries instead of 1024 took 5.9,
// one warp per sequence with 32 entries per lane 6.0).  kLong: rows of many sums (the draw of B = 1 float32, V = 16777216
// 107 to 124 us where every lane added and searched its share one load after the other, now 37 to 39; V = 67108864 298 to 334, now 124).
template <bool kLong, bool kShift, typename RV>
__global__ void __launch_bounds__(kDrawThreads) resample_draw_kernel(const __grid_constant__ ResampleParams P)
{
    __shared__ WalkShared sh;
    const int64_t b = blockIdx.x;
    const double *cs = P.chunk_sum + (size_t)b * P.n_sub;
    pdl_wait();
    pdl_trigger();
    // one round trip for all that decides where to look
    const int n = ld_after(P.accept_len + b);
    const float u = ld_after(P.uniforms + b);
    LaneSums L;
    load_sums(L, P.n_sub, [&](int c) { return ld_after(cs + c); });
    if (n < 0 || n > P.gamma) {
        if (threadIdx.x == 0) {
            P.token[b] = -1;
            if (P.flags) P.flags[b] = DSSD_RS_FLAG_INVALID;
        }
    } else if (!selected(P, n)) {
        if (P.select == 1 && threadIdx.x == 0) {  // a rejected sequence: its token comes from the device half
            P.token[b] = -1;
            if (P.flags) P.flags[b] = 0u;
        }
    } else {
        const RV row = RV::make(P, b, n);
        const float *q = n < P.gamma ? P.draft_q + ((size_t)b * P.gamma + n) * (size_t)P.V : nullptr;
        draw<kLong, kShift>(P, b, row, q, q ? 0u : DSSD_RS_FLAG_BONUS, u, L, sh);
    }
}

// Small launches: one cluster of up to sixteen CTAs per sequence does the whole draw and reads every entry
// once (draw_held).
template <bool kShift, typename RV>
__global__ void __launch_bounds__(kClusterThreads) resample_cluster_kernel(const __grid_constant__ ResampleParams P)
{
    __shared__ double s_sum[2 * kClusterWide * kClusterThreads / 32];
    __shared__ Pick s_pick;
    const int warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
    const unsigned csize = (unsigned)P.n_ctas, rank = csize > 1 ? cluster_rank() : 0u;
    const int64_t b = blockIdx.x / csize;
    const int g = (int)rank * warps + warp;
    if (csize > 1) {  // a CTA's shared memory may be written once it is known to run
        cluster_arrive();
        cluster_wait();
    }
    pdl_wait();
    pdl_trigger();
    const int n = ld_after(P.accept_len + b);
    const float u = warp == 0 ? ld_after(P.uniforms + b) : 0.f;
    WarpQuads<typename RV::Q, 4, kShift> a;
    if (RV::kFixed) a.load(RV::make(P, b, 0).row, P.V, 512ll * g, RV::kFill);  // (on its way before n is back)
    const bool invalid = n < 0 || n > P.gamma;
    if (invalid || !selected(P, n)) {
        if (rank == 0 && threadIdx.x == 0 && (invalid || P.select == 1)) {  // (the bonus token drawn at the edge: the others get their token later)
            P.token[b] = -1;
            if (P.flags) P.flags[b] = invalid ? DSSD_RS_FLAG_INVALID : 0u;
        }
        return;
    }
    const RV row = RV::make(P, b, n);
    if (!RV::kFixed) a.load(row.row, P.V, 512ll * g, RV::kFill);
    const float *q = n < P.gamma ? P.draft_q + ((size_t)b * P.gamma + n) * (size_t)P.V : nullptr;
    draw_held<kShift>(row, a, q, P.V, g, (int)csize * warps, csize, rank, u, s_sum, s_pick, P.token + b, P.flags ? P.flags + b : nullptr);
}

// Batches of middle size (draw_streamed).  Bound by the chain of loads, sums, barrier and walk of each CTA, under which the others on
// the SM stream: 48 registers, so five CTAs of 256 threads share one, for 24 to 48 bytes per thread in local memory (64 and 8 to 48 off the 16-byte
// boundaries).
template <bool kShift, typename RV>
__global__ void __launch_bounds__(kThreads, kShift ? 4 : 5) resample_stream_kernel(const __grid_constant__ ResampleParams P)
{
    __shared__ DrawShared sh;
    const int warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
    const unsigned csize = (unsigned)P.n_ctas, rank = csize > 1 ? cluster_rank() : 0u;
    const int64_t b = blockIdx.x / csize;
    const int g = warp * (int)csize + (int)rank;
    if (csize > 1) {  // the first CTA's shared memory may be written once it is known to run
        cluster_arrive();
        cluster_wait();
    }
    pdl_wait();
    pdl_trigger();
    const int n = ld_after(P.accept_len + b);
    const float u = warp == 0 ? ld_after(P.uniforms + b) : 0.f;
    WarpQuads<typename RV::Q, 4, kShift> a;
    const bool early = RV::kFixed && P.select == 0;  // the row is on its way before n is back
    if (early) a.load(RV::make(P, b, 0).row, P.V, 512ll * g, RV::kFill);
    const bool invalid = n < 0 || n > P.gamma;
    if (invalid || !selected(P, n)) {
        if (rank == 0 && threadIdx.x == 0 && (invalid || P.select == 1)) {  // (the bonus token drawn at the edge: the others get their token later)
            P.token[b] = -1;
            if (P.flags) P.flags[b] = invalid ? DSSD_RS_FLAG_INVALID : 0u;
        }
        return;
    }
    const RV row = RV::make(P, b, n);
    if (!early) a.load(row.row, P.V, 512ll * g, RV::kFill);
    const float *q = n < P.gamma ? P.draft_q + ((size_t)b * P.gamma + n) * (size_t)P.V : nullptr;
    draw_streamed<kShift>(row, a, q, P.V, g, (int)csize * warps, csize, rank, u, sh, P.token + b, P.flags ? P.flags + b : nullptr);
}

// ---- one shard of the vocabulary ---------------------------------------------------------------
//
// The draw over a row that is spread over G shards takes two steps with one small exchange
// between them.  shard_mass_kernel streams this shard's slice of p_row and of Q_n once and leaves,
// per chunk of kSub entries, the residual mass sum max(0, p - q) (sum p for a bonus draw) and the
// plain mass sum p (needed if the residual turns out to have no mass anywhere);
// shard_total_kernel adds a sequence's chunks up.  After the masses of all shards have been
// gathered, shard_draw_kernel - one CTA per sequence - takes the same decisions on every shard
// (Z, fall-back, the shard that holds u' Z) and the owning shard walks its slice exactly as the
// dense kernel walks a row.  Plain stores and stream order connect the launches: no slot is read
// before the launch that wrote it has ended, so the scratch needs no fill.

__device__ __forceinline__ RowF32 shard_row(const ShardResampleParams &P, int64_t b)
{
    RowF32 r;
    r.row = reinterpret_cast<const char *>(P.p_row + (size_t)b * (size_t)P.p_stride);
    return r;
}

template <bool kShift>
__global__ void __launch_bounds__(kThreads, 4) shard_mass_kernel(const __grid_constant__ ShardResampleParams P)
{
    __shared__ double s_w[kWarps][2];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned n_tiles = (unsigned)((P.V + kTile - 1) / kTile);
    const int64_t b = blockIdx.x / n_tiles;
    const int tile = (int)(blockIdx.x - (unsigned)b * n_tiles);
    pdl_wait();
    pdl_trigger();
    const int n = ld_after(P.accept_len + b);
    const bool valid = n >= 0 && n <= P.gamma;
    double r = 0.0, p = 0.0;
    if (valid) {
        const RowF32 row = shard_row(P, b);
        const float *q = n < P.gamma ? P.draft_q + ((size_t)b * P.gamma + n) * (size_t)P.q_stride : nullptr;
        const long long base = (long long)tile * kTile + warp * 512;
        if (q) r = share_mass<true, true, kShift>(row, q, P.V, base, p);
        else r = share_mass<false, true, kShift>(row, q, P.V, base, p);
    }
    r = warp_sum(r);
    p = warp_sum(p);
    if (lane == 0) {
        s_w[warp][0] = r;
        s_w[warp][1] = p;
    }
    __syncthreads();
    if (tid < 2 * kRows) {
        const int k = tid >> 1, c = tile * kRows + k;
        double tot = s_w[2 * k][tid & 1] + s_w[2 * k + 1][tid & 1];
        if (!valid) tot = __longlong_as_double(0x7ff8000000000000ll);
        if (c < P.n_sub) P.chunk_sum[((size_t)b * P.n_sub + c) * 2 + (tid & 1)] = tot;
    }
}

// The same for slices that a cluster of CTAs holds at once (512 entries per warp): the sequence's totals are
// added up in the first CTA's shared memory, which saves the second launch.  For one wave of CTAs (a round of
// B = 8 V = 32000 in two shards 15.3 us against 15.8); in large launches the warps that stand idle beyond the
// slice's end and the barrier cost more (B = 256 V = 151936 in eight shards 39.4 against 36.4).
constexpr int kShardClusterWave = 200;  // CTAs
template <bool kShift>
__global__ void __launch_bounds__(kClusterThreads, 2) shard_mass_cluster_kernel(const __grid_constant__ ShardResampleParams P)
{
    __shared__ double s_all[2][kClusterSums];  // first CTA: every warp's sums
    __shared__ double s_w[kClusterThreads / 32][2];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, warps = blockDim.x >> 5;
    const unsigned csize = (unsigned)P.cluster, rank = csize > 1 ? cluster_rank() : 0u;
    const int64_t b = blockIdx.x / csize;
    const int g = (int)rank * warps + warp;
    if (csize > 1) cluster_arrive();  // the first CTA's shared memory may be written once it is known to run
    pdl_wait();
    pdl_trigger();
    const int n = ld_after(P.accept_len + b);
    const bool valid = n >= 0 && n <= P.gamma;
    double r = 0.0, p = 0.0;
    if (valid) {
        const RowF32 row = shard_row(P, b);
        const float *q = n < P.gamma ? P.draft_q + ((size_t)b * P.gamma + n) * (size_t)P.q_stride : nullptr;
        if (q) r = share_mass<true, true, kShift>(row, q, P.V, 512ll * g, p);
        else r = share_mass<false, true, kShift>(row, q, P.V, 512ll * g, p);
    }
    r = warp_sum(r);
    p = warp_sum(p);
    if (csize > 1) cluster_wait();
    if (lane == 0) {
        s_w[warp][0] = r;
        s_w[warp][1] = p;
        if (csize > 1) {
            cluster_store(&s_all[0][g], 0u, r);
            cluster_store(&s_all[1][g], 0u, p);
        } else {
            s_all[0][g] = r;
            s_all[1][g] = p;
        }
    }
    if (csize > 1) {
        cluster_arrive();
        cluster_wait();
    } else {
        __syncthreads();
    }
    const double nan = __longlong_as_double(0x7ff8000000000000ll);
    if (csize > 1) __syncthreads();
    for (int i = tid; i < warps; i += blockDim.x) {  // chunk i / 2 of this CTA, column i % 2
        const int k = i >> 1, c = (int)rank * (warps / 2) + k;
        const double tot = s_w[2 * k][i & 1] + s_w[2 * k + 1][i & 1];
        if (c < P.n_sub) P.chunk_sum[((size_t)b * P.n_sub + c) * 2 + (i & 1)] = valid ? tot : nan;
    }
    if (rank == 0 && warp < 2) {
        double tot = 0.0;
        for (int i = lane; i < (int)csize * warps; i += 32) tot += s_all[warp][i];
        tot = warp_sum(tot);
        if (lane == 0) P.mass[2 * b + warp] = valid ? tot : nan;
    }
}

// one warp per sequence: the chunk sums in a fixed order
__global__ void __launch_bounds__(kThreads) shard_total_kernel(const __grid_constant__ ShardResampleParams P)
{
    const int lane = threadIdx.x & 31;
    const long long b = (long long)blockIdx.x * kWarps + (threadIdx.x >> 5);
    pdl_wait();
    pdl_trigger();
    if (b >= P.B) return;
    const double *cs = P.chunk_sum + (size_t)b * P.n_sub * 2;
    double r = 0.0, p = 0.0;
    for (int c = lane; c < P.n_sub; c += 32) {
        r += ld_after(cs + 2 * c);
        p += ld_after(cs + 2 * c + 1);
    }
    r = warp_sum(r);
    p = warp_sum(p);
    if (lane == 0) {
        P.mass[2 * b] = r;
        P.mass[2 * b + 1] = p;
    }
}

// one CTA per sequence; kLong: slices of many chunks
template <bool kLong, bool kShift>
__global__ void __launch_bounds__(kDrawThreads) shard_draw_kernel(const __grid_constant__ ShardResampleParams P)
{
    __shared__ WalkShared sh;
    const int64_t b = blockIdx.x;
    pdl_wait();
    pdl_trigger();
    // one round trip for what every sequence needs: the first 32 shards' residual masses (one per lane) and this
    // shard's residual chunk sums
    const int lane = threadIdx.x & 31;
    const int n = ld_after(P.accept_len + b);
    const float u = ld_after(P.uniforms + b);
    const double *masses = P.masses + 2 * b;
    const size_t step = 2 * (size_t)P.B;  // between shards
    const double mass0 = lane < P.G ? ld_after(masses + lane * step) : 0.0;
    const double *cs = P.chunk_sum + (size_t)b * P.n_sub * 2;
    LaneSums L;
    load_sums(L, P.n_sub, [&](int c) { return ld_after(cs + 2 * c); });
    int tok = -1;
    unsigned fl = DSSD_RS_FLAG_INVALID;
    if (n >= 0 && n <= P.gamma) {
        // The verdict on the sequence, from all shards' masses: every thread of every shard takes the
        // same steps in the same order.
        fl = n == P.gamma ? DSSD_RS_FLAG_BONUS : 0u;
        // sum over the shards in their order; `first`: the first shard whose inclusive sum exceeds t (-1: none),
        // `before` the sum before it, `last` the last shard with mass.  32 shards' masses at a time, one per lane.
        auto over_shards = [&](int col, double t, int &first, double &before, int &last) {
            double C = 0.0;
            first = last = -1;
            before = 0.0;
            for (int h0 = 0; h0 < P.G; h0 += 32) {
                double mine = mass0;
                if (h0 || col) mine = h0 + lane < P.G ? ld_after(masses + (h0 + lane) * step + col) : 0.0;
                for (int h = h0; h < P.G && h < h0 + 32; ++h) {
                    const double m = shfl_f64(mine, h - h0);
                    if (m > 0.0) last = h;
                    if (first < 0 && C + m > t) {
                        first = h;
                        before = C;
                    }
                    C += m;
                }
            }
            return C;
        };
        int col = 0, owner, last_mass;
        double before;
        double Z = over_shards(0, INFINITY, owner, before, last_mass);
        bool ok = (Z > 0.0) && (Z < INFINITY);
        if (!ok && n < P.gamma) {  // no residual mass anywhere: draw from p instead
            fl |= DSSD_RS_FLAG_FALLBACK;
            col = 1;
            Z = over_shards(1, INFINITY, owner, before, last_mass);
            ok = (Z > 0.0) && (Z < INFINITY);
        }
        const double t = (double)u * Z;
        over_shards(col, t, owner, before, last_mass);
        const bool beyond = owner < 0;  // rounding left no shard above t: the last shard with mass, its last positive entry
        if (beyond) owner = last_mass;
        if (!ok) {
            fl |= DSSD_RS_FLAG_INVALID;
        } else if (owner == P.g) {
            // this shard holds the target: the chunk first, then the walk inside it
            auto sum = [&](int c) { return ld_after(cs + 2 * c + col); };
            if (col) load_sums(L, P.n_sub, sum);
            const Pick pk = pick_of<kLong>(L, sum, beyond, [&](double) { return t - before; });
            const RowF32 row = shard_row(P, b);
            const float *q = (col == 0 && n < P.gamma) ? P.draft_q + ((size_t)b * P.gamma + n) * (size_t)P.q_stride : nullptr;
            double base = pk.base;
            bool hit;
            tok = walk_chunk<kShift>(pk, row, q, P.V, pk.chunk * kSub, base, hit, sh);
            if (tok < 0) fl |= DSSD_RS_FLAG_INVALID;
            else tok += P.v_begin;
        }
    }
    if (threadIdx.x == 0) {
        P.token[b] = tok;
        if (P.flags) P.flags[b] = fl;
    }
}

}  // namespace

size_t resample_workspace_layout(int B, int V, ResampleParams *P, char *base)
{
    // one sum per chunk; rows of more than 1024 chunks, and batches whose sums would take more than the built-in scratch of
    // dssd_device_resample_static, keep one per two chunks or per tile, which the draw then looks at in turn
    int rows = 1;
    auto sums = [&]() { return ((size_t)V + (size_t)(rows * kSub) - 1) / (size_t)(rows * kSub); };
    while (rows < kRows && (sums() > 1024 || (size_t)B * sums() * sizeof(double) > (size_t)DSSD_STATIC_SCRATCH_BYTES)) rows *= 2;
    const size_t n_sub = sums();
    if (P) {
        P->chunk_sum = reinterpret_cast<double *>(base);
        P->n_sub = (int)n_sub;
        P->rows_per_sum = rows;
    }
    // The size is enough for every smaller batch and vocabulary too, also where those keep more sums per row: they do
    // so up to that scratch's size only.
    const size_t need = (size_t)B * n_sub * sizeof(double), finest = (size_t)B * (((size_t)V + kSub - 1) / kSub) * sizeof(double);
    const size_t smaller = finest < (size_t)DSSD_STATIC_SCRATCH_BYTES ? finest : (size_t)DSSD_STATIC_SCRATCH_BYTES;
    return ((need > smaller ? need : smaller) + 255) & ~(size_t)255;
}

namespace {

// do the rows of an array start on boundaries of four entries?
bool quads_aligned(const void *base, int64_t stride, int esz)
{
    return reinterpret_cast<uintptr_t>(base) % (4 * esz) == 0 && stride % 4 == 0;
}

template <typename RV, bool kShift>
cudaError_t launch_resample_as(const ResampleParams &P, unsigned grid, cudaStream_t stream)
{
    if (P.cluster_threads)
        return launch_pdl(P.streamed ? resample_stream_kernel<kShift, RV> : resample_cluster_kernel<kShift, RV>, (unsigned)(P.B * P.n_ctas),
                          (unsigned)P.cluster_threads, stream, P, 0, (unsigned)P.n_ctas);
    const cudaError_t e = launch_pdl(resample_mass_kernel<kShift, RV>, grid, kThreads, stream, P);
    if (e != cudaSuccess) return e;
    return P.n_sub > kLongSums ? launch_pdl(resample_draw_kernel<true, kShift, RV>, (unsigned)P.B, kDrawThreads, stream, P)
                                : launch_pdl(resample_draw_kernel<false, kShift, RV>, (unsigned)P.B, kDrawThreads, stream, P);
}

template <typename RV>
bool wide_clusters()
{
    return allow_cluster(resample_cluster_kernel<false, RV>, kClusterWide, kClusterThreads) &&
           allow_cluster(resample_cluster_kernel<true, RV>, kClusterWide, kClusterThreads);
}
int most_cluster_ctas()
{
    static PerContext most;
    return most.get([] {
        const bool wide = wide_clusters<RowF32>() && wide_clusters<RowF16>() && wide_clusters<RowLogits<DSSD_F32>>() &&
                          wide_clusters<RowLogits<DSSD_BF16>>();
        if (!wide) cudaGetLastError();
        return wide ? kClusterWide : kClusterMax;
    });
}

// Threads and CTAs per sequence of the kernels that draw in one launch; false where the two kernels are the better ones.
template <class Most>
bool one_launch(ResampleParams &P, bool aligned, Most most_cluster_ctas)
{
    const int segs = (P.V + 511) / 512;
    const long long B = P.B;
    auto is = [&](int threads, long long ctas, bool streamed) {
        P.cluster_threads = threads;
        P.n_ctas = (int)ctas;
        P.streamed = streamed;
        return true;
    };
    if (segs <= 8) {
        if (B * 32 * segs <= kSingleThreads) return is(32 * segs, 1, false);
    } else if (segs <= kClusterWide * kClusterThreads / 32 && B * segs <= kHeldWarps) {
        for (int warps = 4; warps <= kClusterThreads / 32; warps *= 2) {
            const long long ctas = (segs + warps - 1) / warps;
            if (ctas > kClusterWide || (ctas > kClusterMax && (most_cluster_ctas() < kClusterWide || (warps == 4 && B * ctas > kHeldWideCtas)))) continue;
            if (B * ctas * warps <= (ctas <= kClusterMax ? kHeldWarps : warps < 16 ? kHeldWideWarps : kHeldWidestWarps)) return is(32 * warps, ctas, false);
            break;
        }
    }
    if (segs > kStreamSegs) return false;
    const long long sm_warps = aligned ? 40 : 32;  // that the registers of an SM hold, a quarter of them in each of its parts
    const long long wave = 148 * sm_warps;
    long long warps = segs, most_turns = kStreamTurns;
    auto even = [&](long long w) {  // no more than w warps, with even shares
        const long long turns = (segs + w - 1) / w;
        return (segs + turns - 1) / turns;
    };
    if (B * segs <= (segs <= 32 ? kStreamOne : kStreamOneLong)) {
        if (segs <= 2 * kWarps && B >= kStreamHalf) warps = kWarps;
    } else if (B * 10 > wave) {
        for (warps = kWarps; warps >= 4 && B > 148 * (sm_warps / warps);) --warps;
        if (warps < 4) return false;
    } else {
        if (B < kStreamFew && segs > (aligned ? kStreamFewSegs : kStreamFewSegsShifted)) return false;
        warps = even(wave * 7 / 10 / B);
        long long most = kStreamClusters / B / 4 * 4;  // whole CTAs of four warps
        if (most > 4 * kClusterMax) most = 4 * kClusterMax;
        if (most < kWarps || B > kStreamThrees) most = kWarps;
        if (warps > kWarps && (warps + 3) / 4 * 4 > most) warps = even(most);
    }
    if (warps <= kWarps && 10 * kWarps * B < 7 * wave) most_turns = kStreamTurnsFew;
    if (warps > segs) warps = segs;
    if (segs > most_turns * warps) return false;
    if (warps <= kWarps) return is(32 * (int)warps, 1, true);
    return warps <= 4 * kClusterMax ? is(128, (warps + 3) / 4, true) : is(kThreads, (warps + kWarps - 1) / kWarps, true);
}

template <typename RV>
cudaError_t launch_resample(ResampleParams &P, unsigned grid, cudaStream_t stream)
{
    const bool aligned = (P.logits ? quads_aligned(P.logits, P.row_stride, RV::Q::kBytes) : quads_aligned(P.p_row, P.V, RV::Q::kBytes)) &&
                         (!P.draft_q || quads_aligned(P.draft_q, P.V, 4));
    if (!P.test_drop_seq_plus1) one_launch(P, aligned, most_cluster_ctas);
    return aligned ? launch_resample_as<RV, false>(P, grid, stream) : launch_resample_as<RV, true>(P, grid, stream);
}

}  // namespace

void resample_shape_chosen(ResampleParams &P, bool aligned)
{
    P.cluster_threads = P.n_ctas = 0;
    P.streamed = false;
    one_launch(P, aligned, [] { return kClusterWide; });
}

cudaError_t resample_launch(ResampleParams &P, void *workspace, cudaStream_t stream)
{
    resample_workspace_layout(P.B, P.V, &P, static_cast<char *>(workspace));
    const unsigned long long n_tiles = ((unsigned long long)P.V + kTile - 1) / kTile;
    const unsigned long long total = (unsigned long long)P.B * n_tiles;
    P.tiles = total < kTwoTiles ? 1 : total < kFourTiles ? 2 : kResampleMaxTiles;
    P.n_ctas = (int)((n_tiles + P.tiles - 1) / P.tiles);
    const unsigned long long grid = (unsigned long long)P.B * (unsigned long long)P.n_ctas;
    if (grid > 0x7fffffffull) return cudaErrorInvalidConfiguration;
    P.cluster_threads = 0;
    if (P.logits) {
        return P.logits_dtype == DSSD_BF16 ? launch_resample<RowLogits<DSSD_BF16>>(P, (unsigned)grid, stream)
                                           : launch_resample<RowLogits<DSSD_F32>>(P, (unsigned)grid, stream);
    }
    return P.p_half ? launch_resample<RowF16>(P, (unsigned)grid, stream) : launch_resample<RowF32>(P, (unsigned)grid, stream);
}

size_t shard_resample_workspace_bytes(int B, int V)
{
    const size_t n_sub = ((size_t)V + kSub - 1) / kSub;
    return (((size_t)B * n_sub * 2 * sizeof(double)) + 255) & ~(size_t)255;
}

static bool shard_aligned(const ShardResampleParams &P)
{
    return quads_aligned(P.p_row, P.p_stride, 4) && (!P.draft_q || quads_aligned(P.draft_q, P.q_stride, 4));
}

cudaError_t shard_mass_launch(ShardResampleParams &P, void *workspace, cudaStream_t stream)
{
    P.n_sub = (int)(((size_t)P.V + kSub - 1) / kSub);
    P.chunk_sum = static_cast<double *>(workspace);
    const long long warps = ((long long)P.V + 511) / 512;
    const int per_cta = warps <= 8 * kClusterMax ? 8 : 16;
    const long long ctas = (warps + per_cta - 1) / per_cta;
    if (ctas <= kClusterMax && P.B * ctas <= kShardClusterWave) {
        P.cluster = (int)ctas;
        const unsigned block = 32u * (unsigned)per_cta, cgrid = (unsigned)(P.B * ctas);
        return shard_aligned(P) ? launch_pdl(shard_mass_cluster_kernel<false>, cgrid, block, stream, P, 0, (unsigned)ctas)
                                : launch_pdl(shard_mass_cluster_kernel<true>, cgrid, block, stream, P, 0, (unsigned)ctas);
    }
    const unsigned long long grid = (unsigned long long)P.B * (((unsigned long long)P.V + kTile - 1) / kTile);
    if (grid > 0x7fffffffull) return cudaErrorInvalidConfiguration;
    const cudaError_t e = shard_aligned(P) ? launch_pdl(shard_mass_kernel<false>, (unsigned)grid, kThreads, stream, P)
                                           : launch_pdl(shard_mass_kernel<true>, (unsigned)grid, kThreads, stream, P);
    return e != cudaSuccess ? e : launch_pdl(shard_total_kernel, (unsigned)((P.B + kWarps - 1) / kWarps), kThreads, stream, P);
}

cudaError_t shard_draw_launch(ShardResampleParams &P, const void *workspace, cudaStream_t stream)
{
    P.n_sub = (int)(((size_t)P.V + kSub - 1) / kSub);
    P.chunk_sum = const_cast<double *>(static_cast<const double *>(workspace));
    if (P.n_sub > kLongSums)
        return shard_aligned(P) ? launch_pdl(shard_draw_kernel<true, false>, (unsigned)P.B, kDrawThreads, stream, P)
                                : launch_pdl(shard_draw_kernel<true, true>, (unsigned)P.B, kDrawThreads, stream, P);
    return shard_aligned(P) ? launch_pdl(shard_draw_kernel<false, false>, (unsigned)P.B, kDrawThreads, stream, P)
                            : launch_pdl(shard_draw_kernel<false, true>, (unsigned)P.B, kDrawThreads, stream, P);
}

}  // namespace dssd

// ---- dssd_device_resample_static: the same draw, with its scratch inside the library ----------
//
// The scratch of this entry point is a fixed array in the library's device image.  Host code
// cannot use the array's name as an address: the address is looked up once per device with
// cudaGetSymbolAddress, with that device current, and handed to the kernel like any workspace.

static __device__ __align__(256) unsigned char g_static_scratch[DSSD_STATIC_SCRATCH_BYTES];

namespace {
std::mutex g_static_mutex;
void *g_static_ptr[64];  // per device, filled on the first call made with that device current
}  // namespace

extern "C" dssd_status dssd_device_resample_static(const float *p_row, const float *draft_q,
                                                   const int32_t *accept_len, const float *uniforms, int B,
                                                   int gamma, int V, int32_t *token, uint32_t *flags,
                                                   void *cuda_stream)
{
    dssd::set_last_cuda_error(0);
    if (B < 1 || gamma < 0 || V < 1) return DSSD_ERR_INVALID_ARG;
    if (V > DSSD_MAX_V || (long long)B * ((long long)gamma + 1) > (long long)DSSD_MAX_ROWS) return DSSD_ERR_UNSUPPORTED;
    if (!p_row || !accept_len || !uniforms || !token) return DSSD_ERR_INVALID_ARG;
    if (gamma > 0 && !draft_q) return DSSD_ERR_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(p_row) % 4) || (reinterpret_cast<uintptr_t>(draft_q) % 4)) return DSSD_ERR_INVALID_ARG;
    // the built-in scratch has a fixed size: larger batches must use dssd_device_resample
    if (dssd::resample_workspace_layout(B, V, nullptr, nullptr) > (size_t)DSSD_STATIC_SCRATCH_BYTES) return DSSD_ERR_UNSUPPORTED;

    cudaError_t e;
    int dev = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) {
        dssd::set_last_cuda_error((int)e);
        return DSSD_ERR_CUDA;
    }
    if (dev < 0 || dev >= 64) return DSSD_ERR_UNSUPPORTED;
    void *scratch = nullptr;
    {
        std::lock_guard<std::mutex> lock(g_static_mutex);
        if (!g_static_ptr[dev]) {
            void *ptr = nullptr;
            e = cudaGetSymbolAddress(&ptr, g_static_scratch);
            if (e == cudaSuccess && !ptr) e = cudaErrorInvalidSymbol;  // a look-up that gives no address is a failed one
            if (e != cudaSuccess) {
                dssd::set_last_cuda_error((int)e);
                return DSSD_ERR_CUDA;
            }
            g_static_ptr[dev] = ptr;
        }
        scratch = g_static_ptr[dev];
    }

    dssd::ResampleParams P{};
    P.p_row = p_row;
    P.draft_q = draft_q;
    P.accept_len = accept_len;
    P.uniforms = uniforms;
    P.B = B;
    P.gamma = gamma;
    P.V = V;
    P.token = token;
    P.flags = flags;
    // every sum that the draw reads has been written by the same call, so what the previous call left
    // behind does not matter
    e = dssd::resample_launch(P, scratch, static_cast<cudaStream_t>(cuda_stream));
    if (e != cudaSuccess) {
        dssd::set_last_cuda_error((int)e);
        return DSSD_ERR_CUDA;
    }
    return DSSD_OK;
}
