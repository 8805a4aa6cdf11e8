/*
 * wnw_debug.h -- test and measurement hooks of the WnW library (not part of the decode path's interface).
 *
 * Same conventions as wnw.h.  Production code needs none of these: the bounded-wait test hook, per-kernel event
 * timing, and the host-link probe the benchmark reports recall traffic against.
 */
#ifndef WNW_DEBUG_H_
#define WNW_DEBUG_H_

#include "wnw.h"

#ifdef __cplusplus
extern "C" {
#endif

/* Test hook for the bounded waits: adds `delta` to the device's step-epoch word, so that the tidal CTAs of the next
 * replayed step wait for a recall epoch that nothing will publish.  Every such wait gives up after about a second of
 * SM clocks, the kernel finishes on what it has and sets the sticky status that wnw_sync reports as WNW_ERR_TIMEOUT.
 * The cache's results are meaningless afterwards; destroy it.  Not for production use. */
wnw_status_t wnw_debug_advance_step_epoch(wnw_cache_t *cache, int32_t delta);

/* Chunks of a size that is no multiple of 16 tokens are stored padded to whole granules of 16 rows.  On the device the
 * padding rows of a slot are zero; those of the pinned host mirror are neither written nor read.  Test hooks for that:
 * fill sets every byte of the mirror's padding rows of a placed sequence; get copies the padding rows of one slot, head
 * and K|V (which = 0|1) as stored: (chunk_tokens rounded up to 16, minus chunk_tokens) rows of head_dim elements, two
 * bytes each (one in an e4m3 tidal tier).  Both drain the cache's work. */
wnw_status_t wnw_debug_fill_mirror_padding(wnw_cache_t *cache, int32_t seq, int32_t byte);
wnw_status_t wnw_debug_get_slot_padding(wnw_cache_t *cache, int32_t seq, int32_t layer, int32_t kv_head, int32_t slot,
                                        int32_t which, void *rows);

/* How wnw_attend_static cuts the heads of such a call: *cluster = CTAs of the thread-block cluster in which a head's pieces
 * meet, 0 if they meet in global memory.  The answer is the call's own, whatever the process did before. */
wnw_status_t wnw_debug_attend_static_cluster(int32_t device, int32_t n_tokens, int32_t n_q_heads, int32_t n_kv_heads,
                                             int32_t head_dim, int32_t *cluster);

/* How the step issued last cuts a layer: cut[0] the attention kernel, cut[1] CTAs of a thread-block cluster (0: no clusters),
 * cut[2] 1 if a head takes several clusters.  Valid from wnw_step_begin or wnw_graph_begin on until a sequence is placed or
 * grows. */
typedef enum {
  WNW_DEBUG_CUT_PERSISTENT = 0,  /* CTAs that work through several items */
  WNW_DEBUG_CUT_CLUSTER = 1,     /* the pieces of a head in a cluster */
  WNW_DEBUG_CUT_SHORT = 2,       /* ... short pieces, one CTA to an SM */
  WNW_DEBUG_CUT_SHORT_DENSE = 3, /* ... two CTAs to an SM */
  WNW_DEBUG_CUT_ONE_SHOT = 4,    /* CTAs of one item, eight warps */
  WNW_DEBUG_CUT_NARROW = 5,      /* ... four warps */
  WNW_DEBUG_CUT_PACKED = 6       /* eight warps, several heads to a CTA */
} wnw_debug_cut_t;
wnw_status_t wnw_debug_get_layer_cut(wnw_cache_t *cache, int32_t layer, int32_t cut[3]);

/* Optional per-kernel timing: when enabled the library brackets its attention-kernel launches with CUDA events
 * on the launching stream; wnw_get_kernel_time returns the accumulated milliseconds and launch count since the
 * last call (drains the stream).  Off by default. */
wnw_status_t wnw_set_kernel_timing(wnw_cache_t *cache, int32_t enable);
wnw_status_t wnw_get_kernel_time(wnw_cache_t *cache, float *attn_ms, int32_t *attn_launches);

/* Host-link probe used by the benchmark: copies `bytes` from pinned host memory into device memory `reps` times
 * (a) with cudaMemcpyAsync and (b) with the library's recall kernel on a synthetic plan, and returns GB/s of each. */
wnw_status_t wnw_measure_host_link(int32_t device, int64_t bytes, int32_t reps, double *memcpy_gbs, double *kernel_gbs);

#ifdef __cplusplus
}
#endif
#endif /* WNW_DEBUG_H_ */
