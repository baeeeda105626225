/*
 * dssd_test_hooks.h - entry points for the library's own tests.  NOT part of the product API:
 * they exist so that a sum that a kernel hands on can be made to go missing on purpose, in
 * a way that cannot hang or fault a GPU, and the outcome be checked, and so that the choice of a
 * kernel by size can be looked at.  (The paper has no
 * counterpart: its link model of Section 2.2 has no loss or failure term.)
 *
 * The dense kernels hand sums on from one launch to the next; a sum that has not arrived is reported
 * per sequence (DSSD_EDGE_FLAG_TIMEOUT with accept_len = -1, DSSD_RS_FLAG_TIMEOUT |
 * DSSD_RS_FLAG_INVALID with token = -1) and the kernel ends normally.  The first two calls below provoke
 * exactly that by withholding ONE store; nothing else about the launch changes, no address is wrong
 * and nothing waits without a bound.
 */
#ifndef DSSD_TEST_HOOKS_H
#define DSSD_TEST_HOOKS_H

#include "dssd.h"

#ifdef __cplusplus
extern "C" {
#endif

/*
 * dssd_edge_verify in which the partial sum of target row `drop_row` (0 <= drop_row < B * (gamma + 1))
 * is formed but never stored.  (The sums are read after the kernel that forms them has ended, so a
 * missing one is seen at the first look; `poll_limit` is not used.)  The sequence that owns the row
 * ends with accept_len = -1 and DSSD_EDGE_FLAG_TIMEOUT and its p_row is not written; every other
 * sequence is verified as usual.  Arguments otherwise as dssd_edge_verify.
 */
dssd_status dssd_test_edge_verify_wait_runs_out(const void *target_logits, dssd_dtype dtype,
                                                int64_t row_stride, const int32_t *draft_tokens,
                                                const float *draft_q_tok, const float *uniforms,
                                                float temperature, int B, int gamma, int V,
                                                int32_t *accept_len, float *p_row, uint32_t *flags,
                                                void *workspace, size_t workspace_bytes,
                                                long long drop_row, unsigned poll_limit,
                                                void *cuda_stream);

/*
 * dssd_device_resample, always by its mass and its draw kernel (small batches otherwise take one launch, which hands
 * no sum on through memory), in which the chunk sums of sequence `drop_seq` (0 <= drop_seq < B) are
 * computed but never stored.  (The sums are read after the kernel that forms them has ended, so a
 * missing one is seen at the first look; `poll_limit` is not used.)  That sequence ends with token = -1 and DSSD_RS_FLAG_TIMEOUT | DSSD_RS_FLAG_INVALID; every other
 * sequence is drawn for as usual.  Arguments otherwise as dssd_device_resample.
 */
dssd_status dssd_test_device_resample_wait_runs_out(const float *p_row, const float *draft_q,
                                                    const int32_t *accept_len,
                                                    const float *uniforms, int B, int gamma, int V,
                                                    int32_t *token, uint32_t *flags,
                                                    void *workspace, size_t workspace_bytes,
                                                    int drop_seq, unsigned poll_limit,
                                                    void *cuda_stream);

/*
 * Which kernels a call of these sizes takes on a device that has clusters of sixteen CTAs: threads per CTA and CTAs per
 * sequence of the kernel that does it in one launch, 0 and 0 where several do it.  They need no GPU.
 *   edge: form 0 dssd_edge_verify, 1 dssd_edge_verify_bonus, 2 dssd_dsd_verify, 3 dssd_edge_partial of a slice of V entries
 *   draw: dssd_device_resample of float32 rows on 16-byte boundaries; *turns = 1 where the kernel goes over the row in turns
 */
void dssd_test_edge_shape(dssd_dtype dtype, int form, int B, int gamma, int V, int *threads, int *ctas);
void dssd_test_draw_shape(int B, int V, int *threads, int *ctas, int *turns);

#ifdef __cplusplus
}
#endif
#endif /* DSSD_TEST_HOOKS_H */
