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

// Mask word w of one layer (32 experts) by NWARP warps that meet at `sync`: adds up the pairs of the words before its own (what
// its first list starts at), counts its experts per warp (a warp has a contiguous range of 32-token groups), scans, and writes.
// At most 65535 tokens a warp.  cnt: [NWARP * 32], sums: [NWARP], shared.  A warp sees a group's holders of an expert as one ballot.
// Loops are kept short: this runs once per launch, and code that an SM runs for the first time is slow (with the groups' words
// in registers and the loops over them unrolled eight times, a layer call of 64 tokens took 4 us longer).
// FRESH: the mask was written by this very launch (other CTAs of it), so it is read from L2.
template <int NWARP, bool FRESH = false, typename Sync>
__device__ __forceinline__ void lists_of_word(const d2d_list_io &io, int w, int T, int E, int W, int warp, int lane, uint16_t *cnt, int *sums, Sync sync)
{
    constexpr int N = NWARP * 32;
    const uint32_t *mask = io.mask;
    auto load = [](const uint32_t *p) { return FRESH ? __ldcg(p) : __ldg(p); };
    const int per = (T + N - 1) / N * 32;                 // tokens of a warp
    const int t0 = warp * per, t1 = min(T, t0 + per), e = w * 32 + lane;
    const uint32_t valid = E - w * 32 >= 32 ? 0xffffffffu : (1u << (E - w * 32)) - 1u, lower = (1u << lane) - 1u;
    auto word_of = [&](int t) { return t < t1 ? load(mask + (size_t)t * W + w) & valid : 0u; };
    uint32_t word = word_of(t0 + lane);
    int before = 0;
#pragma unroll 1
    for (int t = warp * 32 + lane; t < T; t += N) {
        const uint32_t *row = mask + (size_t)t * W;
        int n = 0;
#pragma unroll 1
        for (int i0 = 0; i0 < w; i0 += 4) {
            uint32_t v[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) v[i] = i0 + i < w ? load(row + i0 + i) : 0u;
            n += __popc(v[0]) + __popc(v[1]) + __popc(v[2]) + __popc(v[3]);
        }
        before += n;
        if (io.k && w == W - 1) io.k[t] = n + __popc(load(row + w));
    }
    before = __reduce_add_sync(0xffffffffu, before);
    int mine = 0;
#pragma unroll 1
    for (int t = t0; t < t1; t += 32) {
        const uint32_t now = word;
        word = word_of(t + 32 + lane);
#pragma unroll 4
        for (int j = 0; j < 32; ++j) {
            const uint32_t b = __ballot_sync(0xffffffffu, (now >> j) & 1u);
            if (lane == j) mine += __popc(b);
        }
    }
    cnt[warp * 32 + lane] = (uint16_t)mine;
    if (lane == 0) sums[warp] = before;
    sync();
    word = word_of(t0 + lane);
    int total = 0, earlier = 0;
    before = 0;
#pragma unroll 4
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
#pragma unroll 1
    for (int t = t0; t < t1; t += 32) {
        const uint32_t now = word;
        word = word_of(t + 32 + lane);
#pragma unroll 4
        for (int j = 0; j < 32; ++j) {
            const uint32_t b = __ballot_sync(0xffffffffu, (now >> j) & 1u);
            const int at = __shfl_sync(0xffffffffu, pos, j) + __popc(b & lower);
            if (((now >> j) & 1u) && at < io.capacity) io.perm[at] = t + lane;
            if (lane == j) pos += __popc(b);
        }
    }
}

}  // namespace d2d_lists
#endif
