// Host-side interface of the edge verification kernels (internal to the library).
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

namespace dssd {

constexpr int kLseThreads = 128;                     // threads per CTA of the log-sum-exp kernel
constexpr int kLseLoads = 8;                         // 16-byte loads a thread has in flight
constexpr int kLseTile = kLseThreads * kLseLoads;    // 16-byte vectors of one pass over the CTA (16 KB)
// Tiles per CTA of the log-sum-exp kernel: one in small launches, so that all SMs share the work; from about
// three waves of 1184 resident CTAs on two, from sixteen on four, so that a CTA's start and reduction are
// paid for less often.  Measured (us, partial sums of a shard, 1 / 2 / 4 tiles): 256 x 5 rows of 151936 bf16
// (24 320 tiles) 74.1 / 66.2 / 62.3, 64 x 9 of 128256 bf16 (9216) 31.3 / 29.2 / 28.7, 300 x 5 of 30011 bf16 (6000)
// 22.5 / 21.4 / 21.9, 256 x 5 of 18992 bf16 (3840) 16.0 / 15.4 / 15.9, 64 x 5 of 50256 float32 (4160) 14.0 / 14.0 /
// 14.6, 30 x 5 of 128256 bf16 (2400) 11.8 / 11.7 / 12.2.  Runs of equal length instead of full tiles and a rest
// are slower (24 320 tiles: 66.0 with four).
constexpr unsigned long long kLseTwoTiles = 3000, kLseFourTiles = 19000;
// Where the separate kernels run, up to one wave of emission CTAs (four per SM) each fold their sequence themselves, which
// saves a launch (B = 1 V = 50272: 0.5 to 1 us on the GPU and 3 us of host time); beyond that a fold per wave costs
// more than a kernel that folds every sequence once (B = 256 V = 151936: emission 49.9 us against 3.1 + 36.5).
constexpr unsigned long long kEmitFoldCtas = 592;

// The cluster kernel does the log-sum-exps, the fold and the emission in one launch.  A unit of its work is a segment (4 KB) of
// logits summed or a piece (512 entries) of the row emitted or drawn from by a warp.  It takes CTAs of 256 threads, as many per
// sequence as give every warp one segment and one piece, as a cluster can have - eight, or sixteen while a warp's work stays
// below kEdgeWideRounds - and as fit a wave: four CTAs per SM, somewhat less for clusters of three and more, which
// do not pack the GPU's processing clusters completely and find no room while the kernel before drains.  From there:
//   * Launches that leave most SMs idle spread over twice the CTAs, so that fewer warps share an SM (us per call, default / spread):
//     B = 13 gamma = 7 V = 42256 / 8 bf16 3.07 / 2.63, B = 3 gamma = 15 V = 4160 bf16 4.50 / 4.23, B = 23 gamma = 8 V = 3200 4.49 / 4.21.
//   * Sequences of more units than such a cluster has warps, few at a time: CTAs of 512 threads, as many as a wave has room for, while
//     a warp's work stays below kEdgeBig's.  One sequence alone leaves SMs idle that the separate kernels use, and pays up to a segment per warp
//     (a round, CTAs of 512 / separate: B = 1 gamma = 8 V = 50272 float32 11.1 / 10.35); two to eight up to two units (B = 2 gamma = 5 V = 48272 float32 10.3 /
//     11.1, B = 4 gamma = 15 V = 29151 12.3 / 13.3, B = 8 gamma = 7 V = 50272 12.5 / 13.0; beyond, B = 5 gamma = 2 V = 133456 15.9 / 15.3, B = 2 gamma = 8 V = 56240 11.6 / 11.2);
//     more sequences by 16 CTAs: B = 14 gamma = 2 V = 83517 float32, a call, 8.5 / 10.2; beyond, B = 12 gamma = 5 V = 90108 bf16 9.7 / 8.7; 12 CTAs: B = 18
//     gamma = 11 V = 34312 float32 10.6 / 11.4; beyond, B = 19 gamma = 8 V = 100000 bf16 15.2 / 14.0; 8: B = 29 gamma = 3 V = 63728 float32 10.4 / 11.5; beyond, B = 30
//     gamma = 11 V = 100000 bf16 23.3 / 21.1; 6: B = 45 gamma = 6 V = 127696 bf16 25.4 / 29.8, B = 35 gamma = 2 V = 140736 float32 19.8 / 20.7; beyond, a round of B = 33 gamma = 11
//     V = 68752 bf16 30.3 / 27.4; 5: B = 48 gamma = 6 V = 115296 float32 34.4 / 35.3.  With a draw as well (five separate kernels): B = 7 gamma = 1 V = 128512 float32
//     10.0 / 13.7, B = 27 gamma = 2 V = 64064 bf16 10.0 / 14.0, a round of B = 6 gamma = 2 V = 109056 float32 17.0 / 19.4; beyond, B = 1 gamma = 4 V = 121880 float32 9.3 / 7.9.
//     A draw alone: B = 17 gamma = 6 V = 54992 float32 13.7 / 16.3, B = 14 gamma = 8 V = 74608 16.4 / 18.9; beyond, B = 44 gamma = 14 V = 57719 float32 41.8 / 38.3.  Not
//     where CTAs of 256 hold the row that is drawn from (fused B = 1 gamma = 12 V = 13930 float32 8.4, of 512 9.9).
//   * A batch that leaves each sequence one or two CTAs and half of the SM's room idle: three to six of 128 threads (kEdgeSmall), which find
//     room in one wave while they are about nine tenths of the clusters that the GPU holds.  B = 303 gamma = 2 V = 24064 float32 22.5 / 25.6, B = 190 gamma = 1
//     V = 34288 bf16 14.5 / 16.7, fused B = 178 gamma = 3 V = 25552 float32 23.7 / 27.5; beyond, the round of B = 213 gamma = 5 V = 7568 float32 23.2 / 18.8, of B = 220 gamma = 2
//     V = 90976 106.7 / 87.1.  Near the last cluster, from 326 sequences on, only with less work per warp: rounds of B = 359 gamma = 7 V = 4993 float32 25.3 / 26.9, B = 367 gamma = 8
//     V = 8080 bf16 26.0 / 29.5, with a draw as well B = 350 gamma = 13 V = 11171 45.7 / 54.3; beyond, B = 327 gamma = 9 V = 11968 float32 51.8 / 45.1, B = 333 gamma = 10 V = 12288
//     54.9 / 46.0, fused B = 349 gamma = 3 V = 12233 32.5 / 27.5.  From 17 units on (five CTAs 24: a round of B = 204 gamma = 6 V = 5721 bf16, 21 units, 18.5 / 17.5), with a draw
//     from 30 on (fused B = 332 gamma = 13 V = 1360, 28 units, 20.2 / 14.9).  Beyond the limits on the work: fused B = 187 gamma = 2 V = 72378 bf16 (18 per warp) 45.1 / 40.9 in
//     separate kernels, a shard of B = 190 gamma = 5 V = 49424 bf16 (15) 26.9 / 23.7, B = 370 gamma = 12 V = 20480 float32 (25) 91.2 / 76.1, a round of B = 300 gamma = 4 V = 30011
//     bf16 (17.4) 49.8 / 49.5.
//   * Otherwise a sequence's two CTAs are one of 512 threads, which needs no cluster, where they are many: B = 117 gamma = 2 V = 6656 bf16 5.0 / 5.4, a round of B = 225
//     gamma = 11 V = 1520 float32 11.3 / 11.7; not from 150 to 203 sequences, where the draw's clusters that follow find less room (a round of B = 175 gamma = 4 V = 5280 bf16
//     13.2 / 11.6).  Not four or six, which as two or three of 512 threads find less room: a round of B = 92 gamma = 14 V = 10400 float32 20.4 us with six of 256, 28.7 with
//     three of 512; B = 49 gamma = 9 V = 5242 bf16 10.9 and 12.2 with two.  Eight from 66 sequences and four from 137 sequences on (a round of B = 137 gamma = 14 V = 44928 bf16 55.5, with four of 256 threads 59.6; of B = 69 gamma = 1 V = 95104 float32 26.7, with seven of 256
//     threads 28.2, with eight 35.2), and a shard's, whose next kernel has few CTAs (the calls of B = 61 gamma = 6 V = 10528 17.4 / 19.2, of B = 90 gamma = 7 V = 16752
//     26.2 / 29.5; of B = 57 gamma = 13 V = 1088 level).
// Near the last cluster that the GPU holds, a launch in a pipeline waits for the one before it to drain (kEdgeMostOf).  Rounds, with one CTA less: B = 70 gamma = 2 V = 42528 float32
// by eight 28.8, by seven 22.2; B = 75 gamma = 2 V = 84960 by seven 39.1, by six 33.6; B = 91 gamma = 3 V = 17695 by six 18.2, by five 17.7; B = 108 gamma = 3 V = 61178 bf16 by five
// 40.2, by four 36.0; fused B = 169 gamma = 2 V = 6224 float32 by three 13.2, by two 10.9.
// How much work per warp still pays depends on how full the wave is, since a
// warp's loads wait for one another from segment to segment and only other CTAs on the SM fill the gaps.  Measured (us per
// call, cluster kernel / separate kernels):
//   few CTAs:  B = 1 gamma = 8 V = 2176 bf16 4.2 / 6.1, B = 8 gamma = 4 V = 32000 bf16 4.8 / 6.5, B = 16 5.4 / 7.0
//   one CTA per sequence:  B = 520 gamma = 1 V = 1172 bf16 5.0 / 11.6, B = 979 gamma = 1 V = 4880 bf16 11.8 / 17.5,
//              B = 318 gamma = 4 V = 9792 bf16 16.3 / 20.2; beyond B = 661 gamma = 1 V = 72431 bf16 110 / 86
//   full wave:  B = 89 gamma = 4 V = 18896 float32 9.6 / 13.0, B = 64 gamma = 4 V = 128256 bf16 26.5 / 29.7,
//              B = 128 gamma = 4 V = 50272 float32 30.7 / 32.3; beyond B = 166 gamma = 11 V = 53648 bf16 52.8 / 48.8.
// A shard's partial sums have no emission to share a launch with and pay off up to less work per warp.  By up to sixteen CTAs of 512 threads the kernel is slower than the two
// from about one unit per warp on (B = 5 gamma = 6 V = 18928 float32 3.5 / 3.9; B = 1 gamma = 8 V = 50272 5.2 / 3.7), but a round is seven launches, which the host
// enqueues in 20 us, and so one less is quicker up to two units, except from a CUDA graph (the calls of B = 1 gamma = 8 V = 50272 17.5 / 20.0, from a graph 15.9 / 14.3; of B = 2 gamma = 7
// V = 36176 18.1 / 20.6 and 15.2 / 14.4, of B = 2 gamma = 9 V = 55623 bf16 17.7 / 21.5 and 15.6 / 14.3); beyond, B = 19 gamma = 8 V = 50272 11.5 / 9.5, B = 40 gamma = 16 V = 76000 bf16 25.0 / 22.6, a round of B = 7 gamma = 13 V = 58416 1.05 of it;
// in smaller ones more: B = 256 gamma = 4 V = 18992
// bf16 13.5 / 14.2, B = 503 gamma = 3 V = 5936 float32 8.5 / 11.1, B = 620 gamma = 15 V = 792 bf16 9.7 / 28.4; beyond B = 173 gamma = 3
// V = 67023 float32 40.5 / 30.5, B = 2 gamma = 2 V = 79648 float32 5.4 / 4.6.  Where the edge draws bonus tokens the separate kernels are
// five and the cluster kernel pays for longer (kEdgeDrawFactor; B = 33 gamma = 10 V = 32480 bf16 11.7 / 16.5), unless it leaves SMs idle and does not hold
// the row (B = 1 gamma = 5 V = 57440 float32 11.4 / 7.5, B = 9 gamma = 4 V = 64935 13.3 / 12.8; held, B = 2 gamma = 10 V = 31702 bf16 9.3 / 10.4).
constexpr int kEdgeCluster = 8, kEdgeClusterWide = 16;  // most CTAs per cluster: portable, and where the device has them
constexpr int kEdgeMostThreads = 512;                    // per CTA
constexpr long long kEdgeWave = 592, kEdgeClusterWave = 552, kEdgeWideWave = 400;  // CTAs: up to two per sequence, up to eight, more
constexpr int kEdgeMostOf[] = {0, 0, 0, 166, 136, 106, 92, 74, 65};  // sequences by so many CTAs each
constexpr long long kEdgeSpread = 140, kEdgeSpreadCtas = 12;  // CTAs, in all and per sequence
constexpr long long kEdgeBigUnits = 64;
struct EdgeBig {  // up to so many sequences (with a draw) so many CTAs of 512 threads each; most work per warp: a row, a draw, both, a shard
    long long most, most_draw;
    int ctas;
    double row, draw, both, shard;
};
constexpr EdgeBig kEdgeBig[] = {{1, 1, 16, 2.0, 2.0, 2.6, 2.2},     {8, 8, 16, 2.08, 2.05, 3.5, 2.2},  {14, 14, 16, 2.0, 3.3, 6.5, 1.4},   {19, 19, 12, 3.0, 2.7, 5.4, 1.05},
                                {30, 30, 8, 5.0, 7.6, 8.0, 1.05}, {39, 39, 6, 8.0, 10.0, 14.5, 3.0}, {45, 43, 6, 12.0, 10.0, 25.0, 3.0}, {52, 50, 5, 13.0, 4.0, 14.5, 3.0}};
struct EdgeSmall {  // up to so many sequences of so many units so many CTAs of 128 threads each; most work per warp as above
    long long most, units;
    int ctas;
    double row, draw, both, shard;
};
constexpr EdgeSmall kEdgeSmall[] = {{181, 17, 6, 15.0, 15.0, 35.0, 8.0}, {204, 24, 5, 15.0, 13.0, 35.0, 8.0}, {325, 17, 3, 15.0, 13.0, 35.0, 8.0},
                                    {335, 17, 3, 9.0, 13.0, 35.0, 8.0},  {350, 17, 3, 9.0, 0.0, 35.0, 8.0},   {370, 17, 3, 9.0, 0.0, 0.0, 0.0}};
constexpr long long kEdgeSmallUnits = 17, kEdgeSmallDrawUnits = 30;  // units of a sequence; with a draw
constexpr long long kEdgePairCtas = 150, kEdgeNoPairs = 150, kEdgeNoPairsTo = 203;
constexpr double kEdgeWideRounds = 2.8, kEdgeWidePartial = 1.6, kEdgeDrawFactor = 1.8;
constexpr int kEdgeHeldWave = 200;                       // CTAs of a launch that draws with the row in registers (two per SM)
constexpr int kEdgeClusterParts = 1024;                  // segments of a sequence (8 KB of shared memory).  It ends the calls by CTAs of 512 threads; the other limits allow 900

// What the draw needs to know about a folded sequence when no row is written.
struct ReadySlot {
    int b;       // sequence
    int n;       // accepted length, or -1 if the sequence has no verdict
    float ref2;  // row n's integer-valued reference exponent: terms are 2^(l * c1 - ref2); never NaN
    float invS;  // 1 / sum_v 2^(l_v * c1 - ref2)   (NaN for a row without finite log-sum-exp)
};

struct EdgeParams {
    // caller's arrays
    const void *logits;
    int64_t row_stride;
    const int32_t *draft_tokens;
    const float *draft_q_tok;
    const float *draft_q_rows;  // instead of draft_q_tok: the full rows [B, gamma, V]; q_i(x_i) is read out of them
    const float *uniforms;
    float temperature;
    float c1;  // log2(e) / T, rounded to float32; the kernels' temperature scaling throughout
    int B, gamma, V;
    int32_t *accept_len;
    int32_t *accept_copy;  // optional second copy of accept_len (in host memory that the GPU reaches)
    float *p_row;          // float32 payload, or
    uint16_t *p_row16;     // IEEE binary16 payload (at most one of the two is set)
    float *p_tok;
    float *lse;
    uint32_t *flags;
    int skip_bonus_row;    // 1: no row is emitted for fully accepted sequences (n == gamma)
    // a token per sequence as well, if the cluster kernel runs (P.cluster != 0 after the launch; otherwise the caller draws):
    // from row gamma for fully accepted sequences and, with draw_rejected, from max(0, p - q) of row n for the others,
    // which get token -1 and flags 0 without it.  draw_rejected needs draft_q_rows.
    int32_t *draw_token;
    uint32_t *draw_flags;
    const float *draw_uniforms;  // [B]
    int draw_rejected;
    // one shard of the vocabulary (entries v_begin .. v_begin + V - 1 of every row): when shard_sum is
    // set only each row's partial sum is formed, sum_v 2^(l_v c1) = shard_sum * 2^shard_ref, and the
    // logits of the drafted tokens the shard holds are looked up; nothing is tested or emitted
    float *shard_ref;         // [B, gamma+1]
    double *shard_sum;        // [B, gamma+1]
    float *shard_tok_logit;   // [B, gamma]; NaN where the token lies outside the shard
    int v_begin;
    // geometry
    int runs;                 // runs per row (one CTA of the log-sum-exp kernel each), segments in the cluster kernel
    int run_vecs;             // 16-byte vectors per run
    int cluster;              // CTAs per sequence of the cluster kernel (0: separate kernels)
    int cta;                  // threads of each
    int emit_tiles;           // tiles (emission CTAs) per sequence
    // test hook (0: off): the partial sums of row test_drop_row_plus1 - 1 are formed but never stored
    long long test_drop_row_plus1;
    // workspace (no initial contents needed: every word that is read has been written by the call)
    unsigned long long *part;        // [rows, runs] (ref2, sum) of one run
    float *tokz;                     // [rows] logit of the row's drafted token (where it lies in the row)
    float *tokq;                     // [rows] its draft probability (draft_q_rows only)
    ReadySlot *ready;                // [B]
};

// Most runs a row can have for a vocabulary of V entries (any dtype, any launch size).
int edge_max_runs_per_row(int V);

// Threads per CTA and CTAs per sequence (P.cta, P.cluster) of the kernel that a call takes where clusters of sixteen CTAs are to be had;
// 0, 0: the separate kernels.  For the tests.
void edge_shape_chosen(EdgeParams &P, int dtype);

// Carves the workspace for `runs_per_row` partial slots per row; returns the bytes needed.
// With P == nullptr only computes the size.
size_t edge_workspace_layout(int B, int gamma, int runs_per_row, EdgeParams *P, char *base);

// Fills the geometry fields of P and launches the kernels on `stream`.
cudaError_t edge_verify_launch(EdgeParams &P, int dtype, void *workspace, cudaStream_t stream);

}  // namespace dssd
