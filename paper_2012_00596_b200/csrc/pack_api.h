// Packing without the read-back: for callers that have counted the very masks they pass (the Python binding), so that the
// blob's size is right by construction and nothing has to be asked of the device.  Not part of the C ABI in npas.h.
#pragma once
#include "npas.h"

#ifdef __cplusplus
extern "C" {
#endif
// size of the blob with n_pairs kept (block, tap) pairs / n_vals stored values (each block's rounded up to 8) and max_cols
// kept columns in the fullest block
npas_status npas_internal_bp_size(const npas_bp_desc *d, uint64_t n_pairs, size_t *blob_bytes);
npas_status npas_internal_bb_size(const npas_bb_desc *d, uint64_t n_vals, uint32_t max_cols, size_t *blob_bytes);
// the pack calls up to, but without, their synchronisation
npas_status npas_internal_pack_bp(const npas_bp_desc *d, const void *w, const uint64_t *tap_mask, void *blob, size_t blob_bytes, void *stream);
npas_status npas_internal_pack_bb(const npas_bb_desc *d, const void *w, const uint64_t *rk, const uint64_t *ck, void *blob,
                                  size_t blob_bytes, void *stream);
#ifdef __cplusplus
}
#endif
