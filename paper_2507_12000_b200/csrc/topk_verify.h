// Host-side interface of the truncated-support (top-k) kernels (internal to the library).
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

namespace dssd {

struct TopkParams {
    // caller's arrays
    const void *logits;
    int64_t row_stride;
    const int32_t *draft_tokens;
    const float *draft_q_tok;
    const float *uniforms;
    float temperature;
    int B, gamma, V, k;
    int32_t *accept_len;
    int32_t *p_idx;
    float *p_val;
    float *p_tok;
    uint32_t *flags;
    // geometry
    int runs;                         // runs per row (one CTA of the selection kernel each)
    int run_vecs;                     // 16-byte vectors per run
    // workspace (no initial contents needed: every word that is read has been written by the call)
    unsigned long long *lists;        // [rows, runs, k] the run's k best keys, best first, 0 where it has fewer
    uint32_t *verdict;                // [rows] many positions only: the row's verdict
};

size_t topk_workspace_bytes(int B, int gamma, int V, int k);

// Fills the geometry and launches the kernels on `stream`.
cudaError_t topk_verify_launch(TopkParams &P, int dtype, void *workspace, cudaStream_t stream);

struct TopkResampleParams {
    const int32_t *p_idx;
    const float *p_val;
    const int32_t *q_idx;
    const float *q_val;
    const int32_t *accept_len;
    const float *uniforms;
    int B, gamma, k;
    int32_t *token;
    uint32_t *flags;
};

cudaError_t topk_resample_launch(const TopkResampleParams &P, cudaStream_t stream);

}  // namespace dssd
