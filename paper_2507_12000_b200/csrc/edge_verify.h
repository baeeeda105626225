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
// Up to one wave of emission CTAs (four per SM) each folds its sequence itself, which saves a launch (B = 8
// V = 32000: 12.1 us a round against 13.3); beyond that a fold per wave costs more than a kernel that
// folds every sequence once (B = 256 V = 151936: emission 49.9 us against 3.1 + 36.5).
constexpr unsigned long long kEmitFoldCtas = 592;

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
    // one shard of the vocabulary (entries v_begin .. v_begin + V - 1 of every row): when shard_sum is
    // set only each row's partial sum is formed, sum_v 2^(l_v c1) = shard_sum * 2^shard_ref, and the
    // logits of the drafted tokens the shard holds are looked up; nothing is tested or emitted
    float *shard_ref;         // [B, gamma+1]
    double *shard_sum;        // [B, gamma+1]
    float *shard_tok_logit;   // [B, gamma]; NaN where the token lies outside the shard
    int v_begin;
    // geometry
    int runs;                 // runs per row (one CTA of the log-sum-exp kernel each)
    int run_vecs;             // 16-byte vectors per run
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

// Carves the workspace for `runs_per_row` partial slots per row; returns the bytes needed.
// With P == nullptr only computes the size.
size_t edge_workspace_layout(int B, int gamma, int runs_per_row, EdgeParams *P, char *base);

// Fills the geometry fields of P and launches the kernels on `stream`.
cudaError_t edge_verify_launch(EdgeParams &P, int dtype, void *workspace, cudaStream_t stream);

}  // namespace dssd
