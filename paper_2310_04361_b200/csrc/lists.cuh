// Per-expert lists (counts, offsets, tokens in ascending order) of a batch small enough for one CTA per mask word to look at all
// of the mask: shared by lists_kernel (select.cu) and the down projection's idle epilogue warps (gemm_tc.cu).
#pragma once

#include "d2d_common.cuh"

struct d2d_list_io {
    const uint32_t *mask;
    int32_t *k, *counts, *offsets, *perm, *n_sel, *status;       // k: wanted too (with the status word), or NULL
    long long capacity;
};
// The lists of up to MAX_N layers of one shape; n = 0: none
template <int MAX_N> struct d2d_list_jobs {
    int n, T, E, W;
    d2d_list_io l[MAX_N];
};
typedef d2d_list_jobs<D2D_MAX_GROUP> d2d_list_job;
d2d_list_job d2d_list_job_for(const d2d_routing *r, int n, int T, int E, bool with_k);      // select.cu

#ifdef __CUDACC__
namespace d2d_lists {

// Lane j returns the bitmap, over this warp's 32 tokens, of bit j of `word`.
__device__ __forceinline__ uint32_t transpose_bits(uint32_t word, int lane)
{
    uint32_t col = 0;
#pragma unroll
    for (int j = 0; j < 32; ++j) {
        const uint32_t b = __ballot_sync(0xffffffffu, (word >> j) & 1u);
        if (lane == j) col = b;
    }
    return col;
}

// Mask word w of one layer (32 experts) by NWARP warps that meet at `sync`: adds up the pairs of the words before its own (what
// its first list starts at), counts its experts per warp (a warp has a contiguous range of 32-token groups), scans, and writes.
// At most GROUPS * 32 * NWARP tokens.  cnt: [NWARP * 32], sums: [NWARP], shared.
template <int NWARP, int GROUPS, typename Sync>
__device__ __forceinline__ void lists_of_word(const d2d_list_io &io, int w, int T, int E, int W, int warp, int lane, uint16_t *cnt, int *sums, Sync sync)
{
    constexpr int N = NWARP * 32;
    const uint32_t *__restrict__ mask = io.mask;
    const int per = (T + N - 1) / N * 32;                 // tokens of a warp
    const int t0 = warp * per, e = w * 32 + lane;
    uint32_t col[GROUPS];                                 // per group of 32 tokens: which of them keep expert e
#pragma unroll
    for (int i = 0; i < GROUPS; ++i) {
        const int t = t0 + i * 32 + lane;
        col[i] = i * 32 < per && t < T ? __ldg(mask + (size_t)t * W + w) : 0u;
    }
    int before = 0;
    for (int t = warp * 32 + lane; t < T; t += N) {
        const uint32_t *row = mask + (size_t)t * W;
        int n = 0;
        for (int i0 = 0; i0 < w; i0 += 8) {                     // eight loads in flight: one after the other they were most of the time
            uint32_t v[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) v[i] = i0 + i < w ? __ldg(row + i0 + i) : 0u;
#pragma unroll
            for (int i = 0; i < 8; ++i) n += __popc(v[i]);
        }
        before += n;
        if (io.k && w == W - 1) io.k[t] = n + __popc(__ldg(row + w));
    }
    before = __reduce_add_sync(0xffffffffu, before);
    int mine = 0;
#pragma unroll
    for (int i = 0; i < GROUPS; ++i) {
        col[i] = transpose_bits(col[i], lane);
        if (e >= E) col[i] = 0u;
        mine += __popc(col[i]);
    }
    cnt[warp * 32 + lane] = (uint16_t)mine;
    if (lane == 0) sums[warp] = before;
    sync();
    int total = 0, earlier = 0;
    before = 0;
#pragma unroll
    for (int i = 0; i < NWARP; ++i) {
        const int c = cnt[i * 32 + lane];
        if (i < warp) earlier += c;
        total += c;
        before += sums[i];
    }
    int inc = total;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += v;
    }
    const int first = before + inc - total;
    if (warp == 0 && e < E) {
        io.counts[e] = total;
        io.offsets[e] = first;
        if (e == E - 1) {
            const int all = first + total;
            io.offsets[E] = all;
            *io.n_sel = all;
            const int over = (long long)all > io.capacity ? (int)D2D_ERR_CAPACITY : 0;
            if (io.k) *io.status = over;
            else if (over) atomicMax(io.status, over);
        }
    }
    int pos = first + earlier;
#pragma unroll
    for (int i = 0; i < GROUPS; ++i) {
        if (i * 32 >= per) break;
#pragma unroll 4
        for (int j = 0; j < 32; ++j) {
            const uint32_t b = __shfl_sync(0xffffffffu, col[i], j);
            const int at = __shfl_sync(0xffffffffu, pos, j) + __popc(b & ((1u << lane) - 1u));
            if (((b >> lane) & 1u) && at < io.capacity) io.perm[at] = t0 + i * 32 + lane;
        }
        pos += __popc(col[i]);
    }
}

}  // namespace d2d_lists
#endif
