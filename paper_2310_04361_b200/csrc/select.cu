// select_dynk (Eq. 4) and the routing metadata of Listing 1, all integer work after one
// float32 multiply per token, built from warp ballots, popcounts and prefix scans so that
// every output is unique and bit-exact: no sort, no order-dependent atomic.
//
//   mask kernel     one warp per token: row max, thr = tau*max (one fp32 RN multiply),
//                   ballot -> packed mask words, popcount -> k
//   count kernel    256 tokens per CTA; each warp turns its 32 tokens x 32 experts bit tile
//                   into per-expert token bitmaps with 32 ballots (a register transpose);
//                   the CTA that finishes last scans: per expert over the token blocks, then
//                   over the experts -> counts, offsets, n_sel
//   fill kernel     same tiling as the count kernel; rank of a token inside its expert's
//                   list = block base + popcounts of the warps before it + popcount of the
//                   lower lanes: tokens come out in ascending order
//   dual kernels    exclusive scan of k -> tok_off; one warp per token writes tok_exp
#include "d2d_common.cuh"
#include "lists.cuh"

namespace {

constexpr int TOKB = 256;         // tokens per CTA in the count / fill kernels (8 warps x 32 tokens)
constexpr unsigned FULL = 0xffffffffu;

__device__ __forceinline__ bool is_finite_f32(float v) { return (__float_as_uint(v) & 0x7f800000u) != 0x7f800000u; }

// ---------------------------------------------------------------------------- mask kernels

// ksum (optional): [0] running sum of k over the CTAs, [1] exit ticket, [2] largest condition (all zero at launch and left at
// zero), [4] receives the total = number of selected (token, expert) pairs, for the density-adaptive dispatch of the
// expert step; the last CTA then also writes *status (otherwise the caller has cleared it).
__global__ void __launch_bounds__(256)
dynk_mask_kernel(const float *__restrict__ R, int T, int E, int W, float tau,
                 uint32_t *__restrict__ mask, int32_t *__restrict__ k, int32_t *__restrict__ status, int32_t *ksum)
{
    __shared__ int block_k;
    if (ksum) {
        if (threadIdx.x == 0) block_k = 0;
        __syncthreads();
    }
    const int lane = threadIdx.x & 31;
    const int t = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (t < T) {
        const float *row = R + (size_t)t * E;
        float m = -INFINITY;
        bool bad = false;
        for (int i = lane; i < E; i += 32) {
            const float v = __ldg(row + i);
            bad |= !is_finite_f32(v);
            m = v > m ? v : m;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float other = __shfl_xor_sync(FULL, m, o);
            m = other > m ? other : m;
        }
        bad = __any_sync(FULL, bad);
        const float thr = __fmul_rn(tau, m);     // the one rounding the rule is defined with
        int kt = 0;
        for (int w = 0; w < W; ++w) {
            const int i = w * 32 + lane;
            const bool keep = (i < E) && (bad || __ldg(row + i) >= thr);
            const uint32_t word = __ballot_sync(FULL, keep);
            if (lane == 0) mask[(size_t)t * W + w] = word;
            kt += __popc(word);
        }
        if (lane == 0) {
            k[t] = kt;
            if (bad) atomicMax(ksum ? ksum + 2 : status, (int32_t)D2D_ERR_NONFINITE);
            if (ksum) atomicAdd(&block_k, kt);
        }
    }
    if (!ksum) return;
    __syncthreads();
    if (threadIdx.x == 0) {
        atomicAdd(ksum, block_k);
        __threadfence();
        if (atomicAdd(ksum + 1, 1) == (int)gridDim.x - 1) {          // the last CTA publishes the total and resets
            __threadfence();
            ksum[4] = atomicExch(ksum, 0);
            *status = atomicExch(ksum + 2, 0);
            ksum[1] = 0;
        }
    }
}

// Static top-k: kk rounds of a warp arg-max over the not yet chosen experts; equal scores
// resolve to the lower expert index.  Lane l owns experts l, l+32, ... (bit j of `chosen`
// = expert l + 32 j), so the ballot of bit j over the lanes is exactly mask word j.
__global__ void __launch_bounds__(256)
topk_mask_kernel(const float *__restrict__ R, int T, int E, int W, int kk,
                 uint32_t *__restrict__ mask, int32_t *__restrict__ k, int32_t *__restrict__ status)
{
    const int lane = threadIdx.x & 31;
    const int t = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (t >= T) return;
    const float *row = R + (size_t)t * E;
    bool bad = false;
    for (int i = lane; i < E; i += 32) bad |= !is_finite_f32(__ldg(row + i));
    bad = __any_sync(FULL, bad);
    unsigned long long chosen = 0ull;        // W <= 64 is checked on the host
    const int keep_n = bad ? E : min(kk, E);
    if (bad) {
        chosen = ~0ull;
    } else {
        for (int round = 0; round < keep_n; ++round) {
            float best = -INFINITY;
            int best_i = 0x7fffffff;
            for (int j = 0; j < W; ++j) {
                const int i = j * 32 + lane;
                if (i < E && !((chosen >> j) & 1ull)) {
                    const float v = __ldg(row + i);
                    if (v > best || (v == best && i < best_i)) { best = v; best_i = i; }
                }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const float ov = __shfl_xor_sync(FULL, best, o);
                const int oi = __shfl_xor_sync(FULL, best_i, o);
                if (ov > best || (ov == best && oi < best_i)) { best = ov; best_i = oi; }
            }
            if ((best_i & 31) == lane && best_i < E) chosen |= 1ull << (best_i >> 5);
        }
    }
    for (int w = 0; w < W; ++w) {
        const bool keep = (w * 32 + lane < E) && ((chosen >> w) & 1ull);
        const uint32_t word = __ballot_sync(FULL, keep);
        if (lane == 0) mask[(size_t)t * W + w] = word;
    }
    if (lane == 0) {
        k[t] = keep_n;
        if (bad) atomicMax(status, (int32_t)D2D_ERR_NONFINITE);
    }
}

// k from a caller-supplied mask (override protocol of Sec. 4.4); also clears what the kernels behind it add to (a memset each took
// as long as this kernel).
__global__ void __launch_bounds__(256)
k_from_mask_kernel(const uint32_t *__restrict__ mask, int T, int W, int32_t *__restrict__ k, unsigned int *ticket, int32_t *status)
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (blockIdx.x == 0 && threadIdx.x == 0) { *ticket = 0u; *status = 0; }
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= T) return;
    int kt = 0;
    for (int w = 0; w < W; ++w) kt += __popc(__ldg(mask + (size_t)t * W + w));
    k[t] = kt;
}

// ---------------------------------------------------------------------------- bucketing

// Lane j returns the bitmap, over this warp's 32 tokens, of bit j of `word`.
__device__ __forceinline__ uint32_t transpose_bits(uint32_t word, int lane)
{
    uint32_t col = 0;
#pragma unroll
    for (int j = 0; j < 32; ++j) {
        const uint32_t b = __ballot_sync(FULL, (word >> j) & 1u);
        if (lane == j) col = b;
    }
    return col;
}

// Exclusive scan of one int per thread over a 256-thread CTA; returns the exclusive prefix and
// leaves the CTA total in *total_out (shared).
__device__ __forceinline__ int block_exscan_256(int v, int *warp_sums /*[8]*/, int *total_out)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int n = __shfl_up_sync(FULL, inc, o);
        if (lane >= o) inc += n;
    }
    if (lane == 31) warp_sums[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        const int ws = lane < 8 ? warp_sums[lane] : 0;
        int winc = ws;
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) {
            const int n = __shfl_up_sync(FULL, winc, o);
            if (lane >= o) winc += n;
        }
        if (lane < 8) warp_sums[lane] = winc - ws;
        if (lane == 7) *total_out = winc;
    }
    __syncthreads();
    const int res = warp_sums[warp] + inc - v;
    __syncthreads();
    return res;
}

// Lists of a batch small enough for every CTA to look at all of the mask: one CTA per mask word (32 experts) and layer, no
// order between CTAs, so counts, offsets and lists take one launch and no scratch (lists.cuh).  k != NULL: k and the status word
// are wanted too.  Bound by latency; as small as bucket_count_scan_kernel, for the same reason.  What it saves is the host's time
// (two launches, a memset and, for a mask that is given, two more): see d2d_launch_select for the line.
constexpr int LISTS_MAX_T = 4 * TOKB;

__global__ void __launch_bounds__(TOKB, 6)
lists_kernel(const __grid_constant__ d2d_list_job g)
{
    __shared__ uint16_t cnt[TOKB];
    __shared__ int sums[TOKB / 32];
    d2d_lists::lists_of_word<TOKB / 32>(g.l[blockIdx.y], blockIdx.x, g.T, g.E, g.W, threadIdx.x >> 5, threadIdx.x & 31, cnt, sums,
                                                      [] { __syncthreads(); });
}

// Per-expert token counts of each 256-token block (8 warps x 32 tokens; a warp turns its
// 32 x 32 bit tile into per-expert bitmaps with 32 ballots).  The CTA that finishes last (ticket
// counter) then scans: per expert the exclusive prefix over the blocks, and over the experts the
// exclusive prefix of the totals -> counts, offsets, n_sel.  Integer sums only: the result does
// not depend on which CTA is last.
// The scan is a chain of L2 latencies: a thread takes an expert and reads eight blocks' counts at a time before it writes
// their prefixes back (one at a time: 25 us for 197 blocks); few experts (at most 64) are cut into segments of blocks, a
// thread per (expert, segment).  Shared memory is kept below 700 bytes: these CTAs run beside the persistent GEMM CTAs,
// which leave 1.8 KB of an SM's shared memory (1 KB of it reserved per CTA) and 10 K registers (40 per thread here).
constexpr int SCAN_BATCH = 8, SCAN_SEGS = 128;

__global__ void __launch_bounds__(TOKB, 6)
bucket_count_scan_kernel(const uint32_t *__restrict__ mask, int T, int E, int W, int nblk,
                         int32_t *__restrict__ blockcounts, unsigned int *__restrict__ ticket,
                         int32_t *__restrict__ counts, int32_t *__restrict__ offsets, int32_t *__restrict__ n_sel,
                         int32_t *__restrict__ status, long long capacity)
{
    __shared__ union { uint16_t cnt[TOKB / 32][33]; int seg[SCAN_SEGS]; } sh;
    __shared__ int warp_sums[8];
    __shared__ int chunk_total;
    __shared__ unsigned int my_ticket;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int t = blockIdx.x * TOKB + threadIdx.x;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    {
        const int w = blockIdx.y;                // one 32-expert mask word per CTA
        const uint32_t word = (t < T) ? __ldg(mask + (size_t)t * W + w) : 0u;
        sh.cnt[warp][lane] = (uint16_t)__popc(transpose_bits(word, lane));
        __syncthreads();
        if (warp == 0) {
            int total = 0;
#pragma unroll
            for (int i = 0; i < TOKB / 32; ++i) total += sh.cnt[i][lane];
            const int e = w * 32 + lane;
            if (e < E) blockcounts[(size_t)blockIdx.x * E + e] = total;
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        // releases the whole CTA's counts (the barrier before it); the last one acquires everybody's
        asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;" : "=r"(my_ticket) : "l"(ticket) : "memory");
        if (my_ticket == (unsigned int)(nblk * W - 1)) *ticket = 0u;      // ready for the next call
    }
    __syncthreads();
    if (my_ticket != (unsigned int)(nblk * W - 1)) return;
    const int nseg = E * 2 <= SCAN_SEGS ? SCAN_SEGS / E : 1, per = (nblk + nseg - 1) / nseg;
    const int sg = nseg > 1 ? (int)threadIdx.x / E : 0;
    const int b_begin = sg * per, b_end = min(nblk, b_begin + per);
    int carry = 0;
    for (int e0 = 0; e0 < E; e0 += TOKB) {
        const int e = nseg > 1 ? (int)threadIdx.x % E : e0 + (int)threadIdx.x;
        const bool on = e < E && sg < nseg;
        int run = 0;
        if (nseg > 1) {
            // totals of the segments before this one
            if (on)
                for (int b0 = b_begin; b0 < b_end; b0 += SCAN_BATCH) {
#pragma unroll
                    for (int i = 0; i < SCAN_BATCH; ++i)
                        if (b0 + i < b_end) run += __ldcg(blockcounts + (size_t)(b0 + i) * E + e);
                }
            if (on) sh.seg[sg * E + e] = run;
            __syncthreads();
            run = 0;
            if (on)
                for (int i = 0; i < sg; ++i) run += sh.seg[i * E + e];
            __syncthreads();
        }
        if (on) {
            for (int b0 = b_begin; b0 < b_end; b0 += SCAN_BATCH) {
                int c[SCAN_BATCH];
#pragma unroll
                for (int i = 0; i < SCAN_BATCH; ++i) c[i] = b0 + i < b_end ? __ldcg(blockcounts + (size_t)(b0 + i) * E + e) : 0;
#pragma unroll
                for (int i = 0; i < SCAN_BATCH; ++i) {
                    if (b0 + i < b_end) blockcounts[(size_t)(b0 + i) * E + e] = run;      // exclusive prefix over the token blocks
                    run += c[i];
                }
            }
        }
        // the last segment's run is the expert's total; experts in the order of their threads
        int total = run;
        if (nseg > 1) {
            if (on && sg == nseg - 1) sh.seg[e] = run;
            __syncthreads();
            total = (int)threadIdx.x < E ? sh.seg[threadIdx.x] : 0;
        } else if (!on) {
            total = 0;
        }
        const int ee = nseg > 1 ? (int)threadIdx.x : e;
        const int ex = block_exscan_256(total, warp_sums, &chunk_total);
        if (ee < E) {
            counts[ee] = total;
            offsets[ee] = carry + ex;
        }
        carry += chunk_total;
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        offsets[E] = carry;
        *n_sel = carry;
        if ((long long)carry > capacity) atomicMax(status, (int32_t)D2D_ERR_CAPACITY);
    }
}

// Writes the per-expert token lists.  Position of token t in expert e's list = offsets[e]
// + tokens of earlier blocks + tokens of earlier warps of this block + tokens of lower lanes,
// so lists come out in ascending token order.  For each expert bit the lanes that hold it write
// consecutive entries (a coalesced store).
__global__ void __launch_bounds__(TOKB)
bucket_fill_kernel(const uint32_t *__restrict__ mask, int T, int E, int W,
                   const int32_t *__restrict__ blockbase, const int32_t *__restrict__ offsets,
                   int32_t *__restrict__ perm, long long capacity)
{
    __shared__ uint16_t cnt[TOKB / 32][33];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int t = blockIdx.x * TOKB + threadIdx.x;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const uint32_t lower = (1u << lane) - 1u;
    {
        const int w = blockIdx.y;                // one 32-expert mask word per CTA
        const int e = w * 32 + lane;
        // start of this CTA's run inside expert e's list (lane = expert); issued early to hide the latency
        const long long cta_base = e < E ? (long long)__ldg(offsets + e) + __ldg(blockbase + (size_t)blockIdx.x * E + e) : 0;
        const uint32_t word = (t < T) ? __ldg(mask + (size_t)t * W + w) : 0u;
        cnt[warp][lane] = (uint16_t)__popc(transpose_bits(word, lane));
        __syncthreads();
        int before = 0;
        for (int i = 0; i < warp; ++i) before += cnt[i][lane];
        const long long base = cta_base + before;
#pragma unroll 4
        for (int j = 0; j < 32; ++j) {
            const uint32_t holders = __ballot_sync(FULL, (word >> j) & 1u);
            const long long bj = __shfl_sync(FULL, base, j);
            if ((word >> j) & 1u) {
                const long long idx = bj + __popc(holders & lower);
                if (idx < capacity) perm[idx] = t;
            }
        }
    }
}

// A mask that is given, in two kernels without a ticket.  The first has everything a 256-token block yields by itself: k, its tokens per
// expert, and on request a copy of the mask and a cleared perm; the second's CTAs each add up the counts of all blocks before
// they fill their part of the lists (as bucket_fill_kernel does), so no CTA scans for the others: a chain of latencies shorter by the
// last CTA's scan, for reading the counts once per CTA (up to SUMS_MAX of them).  50432 tokens x 24 experts, from the first start to the
// last end: 16 us where clearing perm, copying the mask, k, count with scan, and fill took 24.5; the call 16 us instead of 30 at 200 to
// 12608 tokens, where that is the host's time.
constexpr int SUMS_MAX = 16384;

__global__ void __launch_bounds__(TOKB)
mask_count_kernel(const uint32_t *__restrict__ mask, uint32_t *__restrict__ copy, int T, int E, int W, int32_t *__restrict__ k,
                  int32_t *__restrict__ blockcounts, int32_t *__restrict__ perm, long long clear, int32_t *status)
{
    __shared__ uint16_t cnt[TOKB / 32][33];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, w = blockIdx.y;
    const int t = blockIdx.x * TOKB + threadIdx.x, e = w * 32 + lane;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const uint32_t valid = E - w * 32 >= 32 ? FULL : (1u << (E - w * 32)) - 1u;
    uint32_t word = t < T ? __ldg(mask + (size_t)t * W + w) : 0u;
    if (copy && t < T) copy[(size_t)t * W + w] = word;
    word &= valid;
    if (w == 0 && t < T) {
        int kt = __popc(word);
        for (int i = 1; i < W; ++i) kt += __popc(__ldg(mask + (size_t)t * W + i) & (E - i * 32 >= 32 ? FULL : (1u << (E - i * 32)) - 1u));
        k[t] = kt;
    }
    if (blockIdx.x == 0 && w == 0 && threadIdx.x == 0) *status = 0;
    // this CTA's share of perm, in whole 16-byte pieces (perm is 16-byte aligned where it is cleared)
    const long long per = (clear / ((long long)gridDim.x * gridDim.y) + 4) / 4 * 4, at = per * ((long long)w * gridDim.x + blockIdx.x);
    const long long end = at + per < clear ? at + per : clear;
    for (long long i = at + threadIdx.x * 4; i + 4 <= end; i += TOKB * 4) *reinterpret_cast<int4 *>(perm + i) = make_int4(0, 0, 0, 0);
    if (at < end && threadIdx.x < (end & 3)) perm[(end & ~3ll) + threadIdx.x] = 0;
    cnt[warp][lane] = (uint16_t)__popc(transpose_bits(word, lane));
    __syncthreads();
    if (warp == 0 && e < E) {
        int total = 0;
#pragma unroll
        for (int i = 0; i < TOKB / 32; ++i) total += cnt[i][lane];
        blockcounts[(size_t)blockIdx.x * E + e] = total;
    }
}

__global__ void __launch_bounds__(TOKB)
mask_fill_kernel(const uint32_t *__restrict__ mask, int T, int E, int W, int nblk, const int32_t *__restrict__ blockcounts,
                 int32_t *__restrict__ counts, int32_t *__restrict__ offsets, int32_t *__restrict__ n_sel, int32_t *__restrict__ status,
                 int32_t *__restrict__ perm, long long capacity)
{
    constexpr int NW = TOKB / 32;
    __shared__ uint16_t cnt[NW][33];
    __shared__ int earlier[NW][32], all[NW][32], front[NW];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, w = blockIdx.y, b = blockIdx.x;
    const int t = b * TOKB + threadIdx.x, e = w * 32 + lane;
    const uint32_t lower = (1u << lane) - 1u, valid = E - w * 32 >= 32 ? FULL : (1u << (E - w * 32)) - 1u;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const uint32_t word = t < T ? __ldg(mask + (size_t)t * W + w) & valid : 0u;
    // this word's experts: tokens in the blocks before this one, and in all; and all pairs of the words before
    int sum_b = 0, sum_all = 0, sum_f = 0;
    if (e < E)
#pragma unroll 8
        for (int i = warp; i < nblk; i += NW) {
            const int c = __ldcg(blockcounts + (size_t)i * E + e);
            sum_all += c;
            sum_b += i < b ? c : 0;
        }
    for (int i = warp; i < nblk; i += NW)
        for (int j = lane; j < w * 32; j += 32) sum_f += __ldcg(blockcounts + (size_t)i * E + j);
    sum_f = __reduce_add_sync(FULL, sum_f);
    cnt[warp][lane] = (uint16_t)__popc(transpose_bits(word, lane));
    earlier[warp][lane] = sum_b;
    all[warp][lane] = sum_all;
    if (lane == 0) front[warp] = sum_f;
    __syncthreads();
    int total = 0, before = 0, offset = 0;
#pragma unroll
    for (int i = 0; i < NW; ++i) {
        total += all[i][lane];
        before += earlier[i][lane] + (i < warp ? cnt[i][lane] : 0);
        offset += front[i];
    }
    int inc = total;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int n = __shfl_up_sync(FULL, inc, o);
        if (lane >= o) inc += n;
    }
    offset += inc - total;                                    // where expert e's list begins
    if (b == 0 && warp == 0 && e < E) {
        counts[e] = total;
        offsets[e] = offset;
        if (e == E - 1) {
            offsets[E] = offset + total;
            *n_sel = offset + total;
            if ((long long)offset + total > capacity) atomicMax(status, (int32_t)D2D_ERR_CAPACITY);
        }
    }
    const long long base = (long long)offset + before;
#pragma unroll 4
    for (int j = 0; j < 32; ++j) {
        const uint32_t holders = __ballot_sync(FULL, (word >> j) & 1u);
        const long long bj = __shfl_sync(FULL, base, j);
        if ((word >> j) & 1u) {
            const long long idx = bj + __popc(holders & lower);
            if (idx < capacity) perm[idx] = t;
        }
    }
}

// Exclusive scan of one int per thread over a 1024-thread CTA (used by the token-major dual).
__device__ __forceinline__ int block_exscan_1024(int v, int *warp_sums /*[32]*/, int *total_out)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int n = __shfl_up_sync(FULL, inc, o);
        if (lane >= o) inc += n;
    }
    if (lane == 31) warp_sums[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        const int ws = warp_sums[lane];
        int winc = ws;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int n = __shfl_up_sync(FULL, winc, o);
            if (lane >= o) winc += n;
        }
        warp_sums[lane] = winc - ws;
        if (lane == 31) *total_out = winc;
    }
    __syncthreads();
    const int res = warp_sums[warp] + inc - v;
    __syncthreads();
    return res;
}

// ---------------------------------------------------------------------------- token-major dual

__global__ void __launch_bounds__(1024)
tok_scan_kernel(const int32_t *__restrict__ k, int T, int32_t *__restrict__ tok_off)
{
    __shared__ int warp_sums[32];
    __shared__ int chunk_total;
    int carry = 0;
    for (int t0 = 0; t0 < T; t0 += 1024) {
        const int t = t0 + threadIdx.x;
        const int v = (t < T) ? k[t] : 0;
        const int ex = block_exscan_1024(v, warp_sums, &chunk_total);
        if (t < T) tok_off[t] = carry + ex;
        carry += chunk_total;
        __syncthreads();
    }
    if (threadIdx.x == 0) tok_off[T] = carry;
}

__global__ void __launch_bounds__(256)
tok_fill_kernel(const uint32_t *__restrict__ mask, int T, int W, const int32_t *__restrict__ tok_off,
                int32_t *__restrict__ tok_exp, long long capacity)
{
    const int lane = threadIdx.x & 31;
    const int t = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (t >= T) return;
    long long base = tok_off[t];
    for (int w = 0; w < W; ++w) {
        const uint32_t word = __ldg(mask + (size_t)t * W + w);
        if ((word >> lane) & 1u) {
            const long long idx = base + __popc(word & ((1u << lane) - 1u));
            if (idx < capacity) tok_exp[idx] = w * 32 + lane;
        }
        base += __popc(word);
    }
}

}  // namespace

size_t d2d_select_ws_bytes(int T, int E)
{
    // [ticket counter, padded to 256 bytes | per-block, per-expert counters]
    const size_t nblk = (size_t)d2d_cdiv(T > 0 ? T : 1, TOKB);
    return 256 + d2d_align_up(nblk * (size_t)E * sizeof(int32_t), 256);
}

// One launch for the lists of batches whose time is the host's.  A CTA's work grows with the whole mask: up to 1024 tokens
// where nothing runs beside it, up to 512 beside the experts, whose persistent CTAs it competes with for issue slots in longer
// batches (at 1749 tokens it took the BERT-shaped layer from 41 to 57 us, at 1000 the Llama-shaped one from 231 to 244).
static bool lists_in_one_launch(int T, int E, bool alone)
{
    return T <= (alone ? LISTS_MAX_T : LISTS_MAX_T / 2) && (long long)T * ((E + 31) / 32) <= 16384;
}

d2d_list_job d2d_list_job_for(const d2d_routing *r, int n, int T, int E, bool with_k)
{
    d2d_list_job g = {};
    g.n = n; g.T = T; g.E = E; g.W = (E + 31) / 32;
    for (int l = 0; l < n; ++l)
        g.l[l] = {r[l].mask, with_k ? r[l].k : nullptr, r[l].counts, r[l].offsets, r[l].perm, r[l].n_sel, r[l].status,
                  (long long)r[l].perm_capacity};
    return g;
}

static void launch_lists(const d2d_routing *r, int n, int T, int E, bool with_k, cudaStream_t st)
{
    lists_kernel<<<dim3((E + 31) / 32, n), TOKB, 0, st>>>(d2d_list_job_for(r, n, T, E, with_k));
    D2D_LAUNCHED(1);
}

// Token-major dual, where the caller wants it
static void launch_dual(const d2d_routing *out, int T, int W, cudaStream_t st)
{
    if (!out->tok_off || !out->tok_exp) return;
    D2D_LAUNCHED(2);
    tok_scan_kernel<<<1, 1024, 0, st>>>(out->k, T, out->tok_off);
    tok_fill_kernel<<<d2d_cdiv(T, 8), 256, 0, st>>>(out->mask, T, W, out->tok_off, out->tok_exp, (long long)out->perm_capacity);
}

// Lists of n layers of one shape whose masks, k and status words are there.  ws: n workspaces of ws_each bytes
d2d_status d2d_launch_lists(const d2d_routing *r, int n, int T, int E, void *ws, size_t ws_each, cudaStream_t st)
{
    if (lists_in_one_launch(T, E, false)) {
        launch_lists(r, n, T, E, false, st);
        for (int l = 0; l < n; ++l) launch_dual(&r[l], T, (E + 31) / 32, st);
        return cudaGetLastError() == cudaSuccess ? D2D_OK : D2D_ERR_CUDA;
    }
    for (int l = 0; l < n; ++l) {
        const d2d_status rc = d2d_launch_select(nullptr, T, E, 0.0f, 0, &r[l], (char *)ws + (size_t)l * ws_each, st, 1);
        if (rc != D2D_OK) return rc;
    }
    return D2D_OK;
}

// Mask, k and status only (Eq. 4), T > 0; the sum of k is published through ksum (see the kernel).  The per-expert
// lists can be built afterwards, on any stream ordered behind this one, with d2d_launch_select(nullptr, ..., mask_ready = 1).
d2d_status d2d_launch_dynk_mask(const float *R, int T, int E, float tau, const d2d_routing *out, int32_t *ksum, cudaStream_t st)
{
    dynk_mask_kernel<<<d2d_cdiv(T, 8), 256, 0, st>>>(R, T, E, (E + 31) / 32, tau, out->mask, out->k, out->status, ksum);
    D2D_LAUNCHED(1);
    return cudaGetLastError() == cudaSuccess ? D2D_OK : D2D_ERR_CUDA;
}

// k, status and lists from a mask, by mask_count_kernel and mask_fill_kernel.  copy: the mask is to be copied to out->mask, perm cleared
static bool mask_pair_fits(int T, int E) { return (long long)d2d_cdiv(T, TOKB) * E <= SUMS_MAX; }
static d2d_status launch_mask_pair(const uint32_t *mask, int T, int E, const d2d_routing *out, bool copy, void *ws, cudaStream_t st)
{
    const int W = (E + 31) / 32, nblk = d2d_cdiv(T, TOKB);
    int32_t *blockcounts = (int32_t *)((char *)ws + 256);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(nblk, W, 1);
    cfg.blockDim = dim3(TOKB, 1, 1);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = d2d_tc_pdl_enabled() ? 1 : 0;
    const long long capacity = (long long)out->perm_capacity;
    D2D_CUDA_TRY(cudaLaunchKernelEx(&cfg, mask_count_kernel, mask, copy ? out->mask : (uint32_t *)nullptr, T, E, W, out->k, blockcounts, out->perm,
                                    copy ? capacity : 0ll, out->status));
    D2D_CUDA_TRY(cudaLaunchKernelEx(&cfg, mask_fill_kernel, mask, T, E, W, nblk, (const int32_t *)blockcounts, out->counts, out->offsets, out->n_sel,
                                    out->status, out->perm, capacity));
    D2D_LAUNCHED(2);
    launch_dual(out, T, W, st);
    return cudaGetLastError() == cudaSuccess ? D2D_OK : D2D_ERR_CUDA;
}

d2d_status d2d_launch_select_mask_of(const uint32_t *mask, int T, int E, const d2d_routing *out, void *ws, cudaStream_t st)
{
    if (T > 64 && mask_pair_fits(T, E) && (reinterpret_cast<uintptr_t>(out->perm) & 15) == 0) return launch_mask_pair(mask, T, E, out, true, ws, st);
    D2D_CUDA_TRY(cudaMemcpyAsync(out->mask, mask, (size_t)T * ((E + 31) / 32) * 4, cudaMemcpyDeviceToDevice, st));
    D2D_CUDA_TRY(cudaMemsetAsync(out->perm, 0, (size_t)out->perm_capacity * 4, st));
    return d2d_launch_select(nullptr, T, E, 0.0f, 0, out, ws, st);
}

d2d_status d2d_launch_select(const float *R, int T, int E, float tau, int topk, const d2d_routing *out,
                             void *ws, cudaStream_t st, int mask_ready, unsigned int *zero_ticket)
{
    const int W = (E + 31) / 32;
    // a mask that is given, lists in one launch: that kernel writes k and the status word as well
    const bool one = T > 0 && lists_in_one_launch(T, E, !mask_ready), given = !R && !mask_ready;
    const bool small = topk == 0 && d2d_small_select_supports(T, E);
    if (!mask_ready && !(given && T > 0 && !small)) D2D_CUDA_TRY(cudaMemsetAsync(out->status, 0, sizeof(int32_t), st));
    if (T == 0) {
        D2D_CUDA_TRY(cudaMemsetAsync(out->counts, 0, sizeof(int32_t) * (size_t)E, st));
        D2D_CUDA_TRY(cudaMemsetAsync(out->offsets, 0, sizeof(int32_t) * (size_t)(E + 1), st));
        D2D_CUDA_TRY(cudaMemsetAsync(out->n_sel, 0, sizeof(int32_t), st));
        if (out->tok_off) D2D_CUDA_TRY(cudaMemsetAsync(out->tok_off, 0, sizeof(int32_t), st));
        return D2D_OK;
    }
    if (small) return d2d_small_select(R, T, E, tau, out, st, mask_ready);
    if (given && !one && mask_pair_fits(T, E)) return launch_mask_pair(out->mask, T, E, out, false, ws, st);
    const int nblk = d2d_cdiv(T, TOKB);
    // the ticket must start at zero (the kernel leaves it there): a word the caller keeps, or cleared on every call
    unsigned int *ticket = zero_ticket ? zero_ticket : (unsigned int *)ws;
    int32_t *blockcounts = (int32_t *)((char *)ws + 256);
    const int warps_per_cta = 8;
    const int grid_tok = d2d_cdiv(T, warps_per_cta);
    if (R) {
        if (topk > 0)
            topk_mask_kernel<<<grid_tok, 256, 0, st>>>(R, T, E, W, topk, out->mask, out->k, out->status);
        else
            dynk_mask_kernel<<<grid_tok, 256, 0, st>>>(R, T, E, W, tau, out->mask, out->k, out->status, nullptr);
    } else if (given && !one) {
        k_from_mask_kernel<<<nblk, 256, 0, st>>>(out->mask, T, W, out->k, ticket, out->status);
    }
    if (one) {
        D2D_LAUNCHED(R ? 1 : 0);
        launch_lists(out, 1, T, E, given, st);
        launch_dual(out, T, W, st);
        return cudaGetLastError() == cudaSuccess ? D2D_OK : D2D_ERR_CUDA;
    }
    if (!zero_ticket && !given) D2D_CUDA_TRY(cudaMemsetAsync(ticket, 0, sizeof(unsigned int), st));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(nblk, W, 1);
    cfg.blockDim = dim3(TOKB, 1, 1);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = !mask_ready && d2d_tc_pdl_enabled() ? 1 : 0;      // (on a side stream they would only sit on the experts' SMs earlier)
    D2D_CUDA_TRY(cudaLaunchKernelEx(&cfg, bucket_count_scan_kernel, (const uint32_t *)out->mask, T, E, W, nblk, blockcounts, ticket, out->counts,
                                    out->offsets, out->n_sel, out->status, (long long)out->perm_capacity));
    D2D_CUDA_TRY(cudaLaunchKernelEx(&cfg, bucket_fill_kernel, (const uint32_t *)out->mask, T, E, W, (const int32_t *)blockcounts,
                                    (const int32_t *)out->offsets, out->perm, (long long)out->perm_capacity));
    D2D_LAUNCHED(mask_ready ? 2 : 3);
    launch_dual(out, T, W, st);
    return cudaGetLastError() == cudaSuccess ? D2D_OK : D2D_ERR_CUDA;
}

// ------------------------------------------------------------------------------------------
// d2d_select_dynk_static: the same selection + metadata, for callers that are not allowed to
// allocate device memory (and therefore cannot provide the workspace).  The per-block counter
// scratch lives in this file-scope device array instead.  Every GPU that loads the library
// holds these 512 KiB until the process exits.
//
// The name of a __device__ array is only a host-side stand-in in host code, not an address a
// kernel can use; the device address is fetched once per device with cudaGetSymbolAddress
// (with that device current) and cached.
// ------------------------------------------------------------------------------------------
#include <mutex>

#define D2D_STATIC_SCRATCH_INTS (128 * 1024)          /* 512 KiB: 64 + ceil(T/256) * E must not exceed this */
static __device__ __align__(256) int32_t d2d_select_static_scratch[D2D_STATIC_SCRATCH_INTS];

namespace {
constexpr int kMaxDevices = 64;
std::mutex g_scratch_mutex;
int32_t *g_scratch_ptr[kMaxDevices] = {};
}

extern "C" D2D_API d2d_status d2d_select_dynk_static(const float *R, int32_t T, int32_t E, float tau,
                                                     d2d_routing *out, void *stream)
{
    if (T < 0 || E <= 0 || !out || !out->mask || !out->k || !out->counts || !out->offsets || !out->perm ||
        !out->n_sel || !out->status || out->perm_capacity < 0)
        return D2D_ERR_INVALID_ARG;
    if ((out->tok_off == nullptr) != (out->tok_exp == nullptr)) return D2D_ERR_INVALID_ARG;
    if (T > 0 && (!R || (reinterpret_cast<uintptr_t>(R) & 15u))) return D2D_ERR_INVALID_ARG;
    if (!(tau >= 0.0f && tau <= 1.0f)) return D2D_ERR_INVALID_ARG;
    // the scratch holds a ticket counter (64 ints reserved) and one counter per (block of 256 tokens, expert)
    const long long need = 64 + (long long)d2d_cdiv(T > 0 ? T : 1, TOKB) * (long long)E;
    if (need > (long long)D2D_STATIC_SCRATCH_INTS) return D2D_ERR_UNSUPPORTED;

    int dev = -1;
    D2D_CUDA_TRY(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kMaxDevices) return D2D_ERR_UNSUPPORTED;
    int32_t *scratch = nullptr;
    {
        std::lock_guard<std::mutex> lock(g_scratch_mutex);
        if (!g_scratch_ptr[dev]) {
            // first call on this device: resolve the device address of the array (not capturable work)
            void *p = nullptr;
            if (cudaGetSymbolAddress(&p, d2d_select_static_scratch) != cudaSuccess || !p) return D2D_ERR_CUDA;
            g_scratch_ptr[dev] = static_cast<int32_t *>(p);
        }
        scratch = g_scratch_ptr[dev];
    }
    // the ticket counter at the front must start at zero and is cleared by the launch sequence on
    // every call; the block counters need no clearing (each is written before it is read)
    return d2d_launch_select(R, T, E, tau, 0, out, scratch, (cudaStream_t)stream);
}
