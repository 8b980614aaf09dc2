/*
 * hkv_layers.h — calls of the HeadKV C-ABI (hkv.h) that take every layer of
 * the model at once, for callers that hold all layers' inputs together.
 * Conventions, types and statuses are those of hkv.h.
 */
#ifndef HKV_LAYERS_H
#define HKV_LAYERS_H

#include "hkv.h"

#ifdef __cplusplus
extern "C" {
#endif

/* hkv_repack for every layer in one launch (one CTA per head of the model):
 * the same results, checks and errors as a call per layer. Asynchronous on
 * `stream`; a decode step with HKV_STEP_PREFETCH may follow it directly. */
hkv_status hkv_repack_all(const hkv_config *cfg, const hkv_cache *dense, const hkv_cache *ragged,
                          hkv_stream_t stream);

/* One token through every layer: hkv_decode_step for layers 0 .. L-1 in
 * order, or hkv_decode_step_identify where label_out is given, with the same
 * launches, results, checks and errors as the L calls. q, k, v and out hold
 * all layers' rows ([L][S][H][head_dim]). flags as for hkv_decode_step, for
 * every layer: HKV_STEP_PREFETCH says that the kernel before the call does
 * not write layer 0's cache and, between the layers, that L >= 2. A failure
 * leaves the layers before it launched. */
hkv_status hkv_decode_step_layers(const hkv_config *cfg, const hkv_cache *cache, const void *q,
                                  const void *k, const void *v, float *out, uint8_t *label_out,
                                  void *workspace, size_t ws_bytes, int flags,
                                  hkv_stream_t stream);

#ifdef __cplusplus
}
#endif

#endif /* HKV_LAYERS_H */
