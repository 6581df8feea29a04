// What the Python binding's native code calls beside the C ABI in npas.h.
//
// Packing without the read-back: for callers that have counted the very masks they pass, so that the blob's size is right by
// construction and nothing has to be asked of the device.
//
// Chains: several compute calls that one caller makes in a row, with nothing in between that could write one of their blobs.
// The first is launched after everything ahead of it in the stream has ended; the others may then fetch their weights while
// the kernel ahead of them still runs (the rule is at launch_pdl in tc_common.cuh).  A call on another stream belongs to the
// chain when that stream has waited for an event recorded after the chain's first call.
#pragma once
#include "npas.h"

#ifdef __cplusplus
extern "C" {
#endif
// size of the blob with n_pairs kept (block, tap) pairs / n_vals stored values (each block's rounded up to 8) and max_cols
// kept columns in the fullest block
npas_status npas_internal_bp_size(const npas_bp_desc *d, uint64_t n_pairs, size_t *blob_bytes);
npas_status npas_internal_bb_size(const npas_bb_desc *d, uint64_t n_vals, uint32_t max_cols, size_t *blob_bytes);
// The plan of a blob: mask words on the device, each read once, to scratch memory (16-byte aligned, as many bytes as the first
// call says) together with the prefix sums, and the counts that the blob's size follows from to a word of page-locked memory,
// zero before: bit 63 set, above bit 32 the fullest block's taps / columns, below it the kept pairs / stored values.
npas_status npas_internal_plan_bp_bytes(const npas_bp_desc *d, size_t *bytes);
npas_status npas_internal_plan_bp(const npas_bp_desc *d, const uint64_t *words, void *scratch, uint64_t *host, void *stream);
npas_status npas_internal_plan_bb_bytes(const npas_bb_desc *d, size_t *bytes);
npas_status npas_internal_plan_bb(const npas_bb_desc *d, const uint64_t *rows, const uint64_t *cols, void *scratch, uint64_t *host, void *stream);
// the blob of a plan, on the same stream, with the counts it posted
npas_status npas_internal_pack_bp_planned(const npas_bp_desc *d, const void *w, void *scratch, uint64_t n_pairs, void *blob, size_t blob_bytes, void *stream);
npas_status npas_internal_pack_bb_planned(const npas_bb_desc *d, const void *w, void *scratch, uint64_t n_vals, uint32_t max_cols, void *blob,
                                          size_t blob_bytes, void *stream);
// the pack calls up to, but without, their synchronisation
npas_status npas_internal_pack_bp(const npas_bp_desc *d, const void *w, const uint64_t *tap_mask, void *blob, size_t blob_bytes, void *stream);
npas_status npas_internal_pack_bb(const npas_bb_desc *d, const void *w, const uint64_t *rk, const uint64_t *ck, void *blob,
                                  size_t blob_bytes, void *stream);
enum { NPAS_CHAIN_NONE = 0, NPAS_CHAIN_FIRST = 1, NPAS_CHAIN_LATER = 2 };
npas_status npas_internal_conv2d_bp(const npas_conv_desc *d, const npas_bp_desc *bp, const void *x, const void *blob, const float *bias,
                                    const void *residual, void *y, void *ws, size_t ws_bytes, int32_t chain, void *stream);
npas_status npas_internal_conv2d_bp_maxpool(const npas_conv_desc *d, const npas_bp_desc *bp, int32_t pool_r, int32_t pool_stride,
                                            int32_t pool_pad, const void *x, const void *blob, const float *bias, void *y_pooled,
                                            void *ws, size_t ws_bytes, int32_t chain, void *stream);
npas_status npas_internal_linear_bb(const npas_linear_desc *d, const npas_bb_desc *bb, const void *x, const void *blob, const float *bias,
                                    const void *residual, void *y, void *ws, size_t ws_bytes, int32_t chain, void *stream);
// Two GEMMs behind one another, b's input being a's output (which is written all the same), as one launch: whether that is the
// faster way, and the call.  None of y1, y2 may lie on x or the residual.
int32_t npas_internal_linear_two_preferred(const npas_linear_desc *a, const npas_linear_desc *b);
npas_status npas_internal_linear_two(const npas_linear_desc *a, const npas_bb_desc *bba, const npas_linear_desc *b, const npas_bb_desc *bbb,
                                     const void *x, const void *blob1, const float *bias1, const void *residual, void *y1, const void *blob2,
                                     const float *bias2, void *y2, void *ws, size_t ws_bytes, int32_t chain, void *stream);
// Which of the two ways is the faster one on the caller's buffers, for layers whose descriptors name their own measured plans (like the
// tuners in npas.h; not supported where the launch is not preferred): *together, and the microseconds of that way.
npas_status npas_internal_tune_linear_two(const npas_linear_desc *a, const npas_bb_desc *bba, const npas_linear_desc *b, const npas_bb_desc *bbb,
                                          const void *x, const void *blob1, const float *bias1, const void *residual, void *y1, const void *blob2,
                                          const float *bias2, void *y2, void *ws, size_t ws_bytes, int32_t reps, int32_t *together, float *us, void *stream);
// The plan of the pair convolution (path 7) for a call, as a forced `variant` restricts it: filters per item, position tiles per CTA,
// rows of a slab, bytes of a slab stage and of a weight stage, stages of each, bytes of shared memory.
npas_status npas_internal_conv_d2_plan(const npas_conv_desc *d, const npas_bp_desc *bp, int32_t shape[8]);
#ifdef __cplusplus
}
#endif
