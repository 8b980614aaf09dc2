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
 * `stream`. */
hkv_status hkv_repack_all(const hkv_config *cfg, const hkv_cache *dense, const hkv_cache *ragged,
                          hkv_stream_t stream);

#ifdef __cplusplus
}
#endif

#endif /* HKV_LAYERS_H */
