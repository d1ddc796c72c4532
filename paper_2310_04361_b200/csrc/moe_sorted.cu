// Expert step on tokens ordered by the experts they keep, for bf16 layers of at most 32 experts.
//
// A tensor-core tile is 128 token rows.  In the caller's order every expert is kept by some token of a tile, so the masked dense
// pair multiplies everything, and the gathered pair saves in the up projection only.  Tokens whose masks are alike, side by side,
// make tiles that need few experts: the up projection then skips column tiles, the down projection k-blocks, nothing is merged and
// nothing is executed twice.  The fraction of (tile, expert) pairs left is bounded by how many patterns of kept experts the tiles can
// tell apart, so this is for few experts and many tokens: 24 experts, 50432 tokens, independent decisions with probability 0.02 /
// 0.05 / 0.1 / 0.2 / 0.3 / 0.5: 0.06 / 0.15 / 0.30 / 0.56 / 0.70 / 0.83 (in the order of the mask as a number 0.07 / 0.20 / 0.40 /
// 0.65 / 0.76 / 0.86); at 128 experts and 4096 tokens it would be nearly all.
//
//   sort_bucket_kernel   a bucket for each token (1024 of them), its rank in the bucket, the union of the masks of each bucket; the last
//                        CTA turns the counts into positions
//   sort_rows_kernel     copies the token rows (and masks) to their places; one CTA lists the work of the two projections
//   gemm_tc.cu           both projections, from the lists (d2d_gemm_args::sorted)
// Which place a token gets inside its bucket is left to chance; y is not: a token's sums run over k in
// ascending order, and the experts its neighbours brought in contribute exact zeros (finite weights: an infinity or NaN in W2 of an expert
// that a token does not keep reaches it where a neighbour keeps that expert; in the dense pair it reaches every token).
#include "gemm_tc.cuh"
#include "moe_sorted.cuh"
#include "tc_common.cuh"

namespace {

constexpr int N_BUCKETS = D2D_SORTED_BUCKETS, RANK_SHIFT = 10, LOW_BITS = 4;
static_assert(N_BUCKETS == 1 << RANK_SHIFT && RANK_SHIFT == 6 + LOW_BITS, "bucket numbers");
constexpr int THREADS = 512;                // = tokens of a CTA of the bucket kernel
constexpr int TILE = 128;                   // rows of an output tile
constexpr int BN = 256;                     // columns of an output tile of both projections
constexpr int MAX_TILES = D2D_SORTED_MAX_TOKENS / TILE;       // unions of the tiles, in shared memory of the CTA that lists the work

// Which bucket a mask belongs to.  Buckets with similar unions of experts should lie side by side: the upper six bits say which of six
// blocks of adjacent experts have a kept one, in the order of a Gray code (neighbours differ in one block), the lower four are the
// leading bits of the mask without its empty blocks (six of them: 0.305 instead of 0.309 of the pairs left at 50432 tokens, p = 0.1).
__device__ __forceinline__ uint32_t bucket_of(uint32_t mask, int w)
{
    const uint32_t block = w >= 32 ? 0xffffffffu : (1u << w) - 1u;
    uint32_t any = 0u, packed = 0u;
    int used = 0;
#pragma unroll
    for (int i = 5; i >= 0; --i) {
        const uint32_t q = (mask >> (w * i)) & block;             // w * i <= 30
        if (q) {
            any |= 1u << i;
            packed = (packed << w) | q;
            used += w;
        }
    }
    packed = used >= LOW_BITS ? packed >> (used - LOW_BITS) : packed << (LOW_BITS - used);
    any ^= any >> 1; any ^= any >> 2; any ^= any >> 4;            // position in the Gray code
    return any << LOW_BITS | (packed & ((1u << LOW_BITS) - 1u));
}

struct SortArgs {
    const uint4 *x;
    uint4 *xs;
    const uint32_t *mask;
    uint32_t *smask;                        // [T] masks in the new order
    int *order;                             // [T] token of each place
    uint32_t *keyrank;                      // [T] bucket | rank << RANK_SHIFT
    int *base;                              // [N_BUCKETS] first place of a bucket
    uint32_t *up_items;                     // row tile << 8 | column tile
    uint2 *down_items;                      // (row tile, union of its masks), those with most experts first
    int *n_items;                           // number of up_items
    int *ctr;                               // [N_BUCKETS] counts | [N_BUCKETS] unions | ticket: zero at launch and behind the rows kernel
    const int32_t *n_sel;
    long long n_sel_max;
    int T, row16;                           // row16: 16-byte pieces of a token row
    int w, s, up_cols;                      // experts per block; expert size; column tiles of the up projection
};

// exclusive prefix sum over the CTA's THREADS values; total in `total`
__device__ __forceinline__ int block_scan(int v, int *scratch, int &total)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += u;
    }
    __syncthreads();
    if (lane == 31) scratch[warp] = inc;
    __syncthreads();
    int before = 0, all = 0;
#pragma unroll
    for (int i = 0; i < THREADS / 32; ++i) {
        const int c = scratch[i];
        before += i < warp ? c : 0;
        all += c;
    }
    total = all;
    return before + inc - v;
}

// Bound by a chain of latencies (mask, shared and global atomics, ticket, scan), not by its traffic.
__global__ void __launch_bounds__(THREADS) sort_bucket_kernel(const SortArgs a)
{
    __shared__ int cnt[N_BUCKETS];
    __shared__ uint32_t uni[N_BUCKETS];
    __shared__ int scratch[THREADS / 32], last;
    const int tid = threadIdx.x;
    for (int i = tid; i < N_BUCKETS; i += THREADS) { cnt[i] = 0; uni[i] = 0u; }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (a.n_sel && (long long)__ldcg(a.n_sel) > a.n_sel_max) return;
    const int t = (int)blockIdx.x * THREADS + tid;
    const bool in = t < a.T;
    const uint32_t m = in ? __ldg(a.mask + t) : 0u;
    const uint32_t b = in ? bucket_of(m, a.w) : N_BUCKETS;
    __syncthreads();
    // one addition per bucket and warp (a bucket may hold most of the batch)
    const uint32_t peers = __match_any_sync(0xffffffffu, b);
    const uint32_t peer_or = __reduce_or_sync(peers, m);
    const int lane = tid & 31, lead = __ffs(peers) - 1;
    int rank = 0;
    if (in && lane == lead) {
        rank = atomicAdd(&cnt[b], __popc(peers));
        atomicOr(&uni[b], peer_or);
    }
    rank = __shfl_sync(0xffffffffu, rank, lead) + __popc(peers & ((1u << lane) - 1u));
    __syncthreads();
    if (in && rank == 0) {                                        // the bucket's first token in this CTA
        atomicOr(reinterpret_cast<unsigned int *>(a.ctr) + N_BUCKETS + b, uni[b]);
        cnt[b] = atomicAdd(a.ctr + b, cnt[b]);
    }
    __syncthreads();
    if (in) a.keyrank[t] = b | (uint32_t)(cnt[b] + rank) << RANK_SHIFT;
    if (tid == 0) {
        // releases the whole CTA's additions (the barrier before it); the last one acquires everybody's
        int n;
        asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;" : "=r"(n) : "l"(a.ctr + 2 * N_BUCKETS) : "memory");
        last = n == (int)gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    // the last CTA: places of the buckets
    static_assert(N_BUCKETS == 2 * THREADS, "two buckets a thread");
    int2 *const ctr2 = reinterpret_cast<int2 *>(a.ctr) + tid;
    const int2 c = __ldcg(ctr2);
    *ctr2 = make_int2(0, 0);
    int total;
    const int at = block_scan(c.x + c.y, scratch, total);
    reinterpret_cast<int2 *>(a.base)[tid] = make_int2(at, at + c.x);
    if (tid == 0) a.ctr[2 * N_BUCKETS] = 0;
}

// The union of the masks of each tile, and from them the work of the projections.  A tile gets what the buckets that reach into it
// have: where buckets begin or end inside a tile that may be more than its own tokens keep (their experts are multiplied for nothing,
// with masks that say so).
__device__ __forceinline__ void list_work(const SortArgs &a)
{
    __shared__ int first[N_BUCKETS + 1];
    __shared__ uint32_t uni[N_BUCKETS], tile_or[MAX_TILES];
    __shared__ int scratch[THREADS / 32], by_size[33];
    const int tid = threadIdx.x;
    const int n_tiles = (a.T + TILE - 1) / TILE;
    for (int i = tid; i < N_BUCKETS; i += THREADS) {
        first[i] = __ldcg(a.base + i);
        uni[i] = __ldcg(reinterpret_cast<const unsigned int *>(a.ctr) + N_BUCKETS + i);
        a.ctr[N_BUCKETS + i] = 0;
    }
    if (tid == 0) first[N_BUCKETS] = a.T;
    for (int i = tid; i < n_tiles; i += THREADS) tile_or[i] = 0u;
    if (tid < 33) by_size[tid] = 0;
    __syncthreads();
    for (int i = tid; i < N_BUCKETS; i += THREADS) {
        const int lo = first[i], hi = first[i + 1];
        if (hi > lo) {
            atomicOr(&tile_or[lo / TILE], uni[i]);
            atomicOr(&tile_or[(hi - 1) / TILE], uni[i]);
        }
    }
    for (int i = tid; i < n_tiles; i += THREADS) {                // tiles that lie inside one bucket
        int lo = 0, hi = N_BUCKETS - 1;                           // the last bucket that begins at or before the tile
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (first[mid] <= i * TILE) lo = mid; else hi = mid - 1;
        }
        if (first[lo + 1] >= (i + 1) * TILE) atomicOr(&tile_or[i], uni[lo]);
    }
    __syncthreads();
    // bits of the union that column tile c of the up projection needs
    const int per_col = BN / a.s;
    auto bits = [&](int c) { return ((1u << per_col) - 1u) << (c * per_col); };
    int n_up = 0;
    for (int i0 = 0; i0 < n_tiles; i0 += THREADS) {
        const int i = i0 + tid;
        const uint32_t u = i < n_tiles ? tile_or[i] : 0u;
        if (i < n_tiles) atomicAdd(&by_size[32 - __popc(u)], 1);
        int n = 0, all;
        for (int c = 0; c < a.up_cols; ++c) n += u & bits(c) ? 1 : 0;
        int to = n_up + block_scan(n, scratch, all);
        for (int c = 0; c < a.up_cols; ++c)
            if (u & bits(c)) a.up_items[to++] = (uint32_t)i << 8 | (uint32_t)c;
        n_up += all;
    }
    __syncthreads();
    if (tid < 32) {
        const int n = by_size[tid];
        int inc = n;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, inc, o);
            if (tid >= o) inc += u;
        }
        by_size[tid] = inc - n;
        if (tid == 31) by_size[32] = inc;
        if (tid == 0) *a.n_items = n_up;
    }
    __syncthreads();
    for (int i = tid; i < n_tiles; i += THREADS)
        a.down_items[atomicAdd(&by_size[32 - __popc(tile_or[i])], 1)] = make_uint2((uint32_t)i, tile_or[i]);
}

// Token rows to their places: a warp per row, four rows at once.  Bound by memory: reads and writes T d 2 bytes (50432 rows of 768: 23 us
// = 6.7 TB/s).  Rows of tokens that keep nothing are left out: whatever the tile then multiplies is masked.
constexpr int ROWS_AT_ONCE = 4;
__global__ void __launch_bounds__(THREADS) sort_rows_kernel(const SortArgs a)
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (a.n_sel && (long long)__ldcg(a.n_sel) > a.n_sel_max) return;
    if (blockIdx.x == 0) {
        list_work(a);
        return;
    }
    const int lane = threadIdx.x & 31;
    constexpr int WARPS = THREADS / 32;
    const int n_warps = (int)(gridDim.x - 1) * WARPS;
    for (int t0 = (((int)blockIdx.x - 1) * WARPS + (threadIdx.x >> 5)) * ROWS_AT_ONCE; t0 < a.T; t0 += n_warps * ROWS_AT_ONCE) {
        const int mine = t0 + (lane & (ROWS_AT_ONCE - 1));
        int p = -1;
        if (mine < a.T) {
            const uint32_t kr = __ldcg(a.keyrank + mine), m = __ldg(a.mask + mine);
            p = __ldcg(a.base + (kr & (N_BUCKETS - 1))) + (int)(kr >> RANK_SHIFT);
            if (lane < ROWS_AT_ONCE) {
                a.order[p] = mine;
                a.smask[p] = m;
            }
            if (m == 0u) p = -1;
        }
        int pos[ROWS_AT_ONCE];
#pragma unroll
        for (int j = 0; j < ROWS_AT_ONCE; ++j) pos[j] = __shfl_sync(0xffffffffu, p, j);
        for (int c = lane; c < a.row16; c += 32) {
            uint4 v[ROWS_AT_ONCE];
#pragma unroll
            for (int j = 0; j < ROWS_AT_ONCE; ++j)
                if (pos[j] >= 0) v[j] = __ldg(a.x + (size_t)(t0 + j) * a.row16 + c);
#pragma unroll
            for (int j = 0; j < ROWS_AT_ONCE; ++j)
                if (pos[j] >= 0) a.xs[(size_t)pos[j] * a.row16 + c] = v[j];
        }
    }
}

template <typename K, typename A> d2d_status launch_pdl(K kern, int grid, int block, const A &a, cudaStream_t st)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid, 1, 1);
    cfg.blockDim = dim3(block, 1, 1);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = d2d_tc_pdl_enabled() ? 1 : 0;
    const cudaError_t err = cudaLaunchKernelEx(&cfg, kern, a);
    D2D_LAUNCHED(1);
    return err == cudaSuccess ? D2D_OK : D2D_ERR_CUDA;
}

}  // namespace

// At most one mask word; column tiles of 256 that hold whole experts and k-blocks of 64 that lie inside one (expert sizes 64 and 128: no
// layer has larger ones); whole column tiles in both projections; weights that stay in L2 beside the rows (the lists are walked row
// tile by row tile).
bool d2d_sorted_supports(const d2d_layer_desc &D, int T)
{
    const bool size_ok = D.expert_size == 64 || D.expert_size == 128;
    return D.dtype == D2D_BF16 && !D.gated && D.n_experts <= 32 && size_ok && D.d % BN == 0 && D.d_ff % BN == 0 && D.d_ff / BN <= 256 &&
           2.0 * D.d * D.d_ff < 48e6 && T > 0 && T <= D2D_SORTED_MAX_TOKENS;
}

d2d_sorted_layout d2d_sorted_layout_for(const d2d_layer_desc &D, int T)
{
    d2d_sorted_layout l;
    size_t off = 0;
    auto take = [&](size_t bytes) { const size_t o = off; off += d2d_align_up(bytes, 256); return o; };
    const size_t tiles = (size_t)d2d_cdiv(T, TILE);
    l.xs = take((size_t)T * D.d * 2);
    l.order = take((size_t)T * 4);
    l.smask = take((size_t)T * 4);
    l.keyrank = take((size_t)T * 4);
    l.base = take(N_BUCKETS * 4);
    l.up_items = take(tiles * (D.d_ff / BN) * 4);
    l.down_items = take(tiles * 8);
    l.n_items = take(4);
    l.total = off;
    return l;
}

d2d_status d2d_moe_sorted(const d2d_layer *L, const void *x, int T, const d2d_routing *r, void *y, void *H, void *ws, int *ctr, int *tile_counters,
                          const int32_t *n_sel, long long n_sel_max, cudaStream_t st)
{
    const d2d_layer_desc &D = L->desc;
    const d2d_sorted_layout l = d2d_sorted_layout_for(D, T);
    char *base = (char *)ws;
    SortArgs s = {};
    s.x = (const uint4 *)x; s.xs = (uint4 *)(base + l.xs); s.mask = r->mask; s.smask = (uint32_t *)(base + l.smask); s.order = (int *)(base + l.order);
    s.keyrank = (uint32_t *)(base + l.keyrank); s.base = (int *)(base + l.base);
    s.up_items = (uint32_t *)(base + l.up_items); s.down_items = (uint2 *)(base + l.down_items); s.n_items = (int *)(base + l.n_items);
    s.ctr = ctr; s.n_sel = n_sel; s.n_sel_max = n_sel_max;
    s.T = T; s.row16 = D.d / 8; s.w = d2d_cdiv(D.n_experts, 6); s.s = D.expert_size; s.up_cols = D.d_ff / BN;
    d2d_status rc = launch_pdl(sort_bucket_kernel, d2d_cdiv(T, THREADS), THREADS, s, st);
    if (rc != D2D_OK) return rc;
    const int want = d2d_cdiv(T, THREADS / 32 * ROWS_AT_ONCE), most = 4 * d2d_tc_sm_count();
    rc = launch_pdl(sort_rows_kernel, 1 + (want < most ? want : most), THREADS, s, st);
    if (rc != D2D_OK) return rc;
    d2d_gemm_args up = {};
    up.a = s.xs; up.b = L->w1; up.bias = L->b1; up.out = H;
    up.M = T; up.N = D.d_ff; up.K = D.d; up.epilogue = D2D_EPI_UP_MASKED; up.act = D.act;
    up.mask = s.smask; up.mask_words = 1; up.expert_size = D.expert_size; up.status = r->status;
    up.n_sel = n_sel; up.n_sel_max = n_sel_max;
    up.tile_counter = tile_counters;
    up.sorted = {true, s.up_items, s.n_items, nullptr, nullptr};
    rc = d2d_gemm_tc(up, st);
    if (rc != D2D_OK) return rc;
    d2d_gemm_args dn = {};
    dn.a = H; dn.b = L->w2; dn.bias = L->b2; dn.out = y;
    dn.M = T; dn.N = D.d; dn.K = D.d_ff; dn.epilogue = D2D_EPI_BIAS_BF16; dn.status = r->status; dn.expert_size = D.expert_size;
    dn.n_sel = n_sel; dn.n_sel_max = n_sel_max;
    dn.tile_counter = tile_counters + 1;
    dn.sorted = {true, nullptr, nullptr, s.down_items, s.order};
    return d2d_gemm_tc(dn, st);
}
