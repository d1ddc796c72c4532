// Interface of the expert step on tokens ordered by the experts they keep (see moe_sorted.cu).
#pragma once

#include "d2d_common.cuh"

// Where things lie in the form's scratch (byte offsets)
struct d2d_sorted_layout {
    size_t xs, order, smask, keyrank, base, up_items, down_items, n_items, total;
};

// Whether layers of this shape can take the form at T tokens at all (d2d_api.cu decides when they do)
bool d2d_sorted_supports(const d2d_layer_desc &D, int T);
d2d_sorted_layout d2d_sorted_layout_for(const d2d_layer_desc &D, int T);
// Buckets of the order, and the device ints the kernels need zeroed at creation (and leave zeroed)
constexpr int D2D_SORTED_BUCKETS = 1024, D2D_SORTED_CTR_WORDS = 2 * D2D_SORTED_BUCKETS + 64;

// y = the expert step of the batch: buckets, row copies, up projection, down projection, all of which return at once unless *n_sel is at
// most n_sel_max (n_sel NULL: always work).  H: [T, d_ff] bf16 scratch, ws: d2d_sorted_layout_for(...).total bytes, both the
// caller's; ctr: D2D_SORTED_CTR_WORDS layer-owned ints, tile_counters: two.
d2d_status d2d_moe_sorted(const d2d_layer *L, const void *x, int T, const d2d_routing *r, void *y, void *H, void *ws, int *ctr, int *tile_counters,
                          const int32_t *n_sel, long long n_sel_max, cudaStream_t st);
