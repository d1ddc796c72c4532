// bf16 GEMM C[M,N] = epilogue(A[M,K] B[N,K]^T) on the 5th-generation tensor cores of sm_100a.
//
//   warp 0   TMA producer: cp.async.bulk.tensor tiles of A (128 x 64) and B (BN x 64), 128-byte
//            swizzled, into a ring of shared-memory stages guarded by full/empty mbarriers
//   warp 1   allocates TMEM and issues tcgen05.mma (one thread), fp32 accumulators in TMEM
//            (two buffers); tcgen05.commit releases a stage when the MMAs that read it have retired
//   warps 2-17 epilogue: tcgen05.ld the accumulator (one row per thread), bias / activation /
//            selection mask, vectorised stores; runs while the next tile's MMAs fill the other buffer
// The kernel is persistent: one CTA per SM walks over the output tiles.
//
// Every mbarrier wait is bounded: when the limit runs out the role records D2D_ERR_TIMEOUT in the
// status word and leaves its loop, all roles meet at the final barrier, TMEM is freed and the
// kernel returns (no trap, no endless spin).  Every load is a plain per-CTA load.
#include "gemm_tc.cuh"
#include "tc_common.cuh"

#include <stdlib.h>

namespace {

using namespace d2d_tc;

constexpr int BM = 128;          // rows of A per CTA = TMEM lanes
constexpr int BK = 64;           // 64 bf16 = one 128-byte swizzle row
constexpr int UMMA_K = 16;

struct EpiParams {
    const __nv_bfloat16 *bias;
    void *out;
    const uint32_t *mask;
    int mask_words;
    int expert_size;
    int32_t *status;
    // ceil(2^32 / expert_size), for sizes that are multiples of 8: column / expert_size = umulhi(column, inv) for columns that are,
    // too, up to columns x size = 2^35 (such a column is at least 8 below the next expert; 2^16 columns of any size)
    uint32_t inv_expert_size;
    int *tile_counter;               // device counter (zero at launch) for dynamic tile scheduling, NULL = static round-robin
    int late_wait;                   // 1: only the epilogue waits for the previous kernel of the stream (see below)
    int gate_cat;                    // 1 (gated): tm_b covers up and gate rows interleaved in blocks of BN, one load brings both
    int band_rows;                   // > 0: tiles are walked column-major inside bands of this many row tiles (L2 reuse)
    int batch;                       // >= 1 problems of one shape: A columns, B rows, bias entries and out advance per problem
    const int32_t *n_sel;            // density-adaptive dispatch: do nothing when *n_sel <= n_sel_max (NULL: always run)
    long long n_sel_max;
    float4 *zero;                    // optional: cleared by the epilogue warps before their first tile (see d2d_gemm_args)
    int zero_n;                      // 16-byte pieces
    int slices_per_sum;              // split-K: so many slices add to one float32 buffer (see pick_split)
    int test_skip_load;              // test aid: CTA 0 never requests the A tile of its first k-block (see d2d_gemm_args)
};

// Work lists of the kernels that run on tokens ordered by the experts they keep (see d2d_gemm_args::sorted).  Launches without any do
// without the code.
enum { SORTED_NONE = 0, SORTED_UP = 1, SORTED_DOWN = 2 };
struct NoItems {};
struct UpItems { const uint32_t *items; const int *n_items; };          // row tile << 8 | column tile
struct DownItems { const uint2 *items; const int *order; int kpe; };    // (row tile, union of its masks); k-blocks of an expert
template <int SORTED> struct ItemsOf { typedef NoItems type; };
template <> struct ItemsOf<SORTED_UP> { typedef UpItems type; };
template <> struct ItemsOf<SORTED_DOWN> { typedef DownItems type; };
inline void set_items(NoItems &, const d2d_gemm_args &) {}
inline void set_items(UpItems &s, const d2d_gemm_args &g) { s = {g.sorted.up_items, g.sorted.n_items}; }
inline void set_items(DownItems &s, const d2d_gemm_args &g) { s = {g.sorted.down_items, g.sorted.order, g.expert_size / 64}; }

// Number of items, and item `index`: row tile << 8 | column tile, and (down, cols of them per row tile) the union
__device__ __forceinline__ int n_items(const UpItems &s, int) { return __ldcg(s.n_items); }
__device__ __forceinline__ int n_items(const DownItems &, int tiles) { return tiles; }
__device__ __forceinline__ uint2 item_at(const UpItems &s, int index, int) { return make_uint2(__ldcg(s.items + index), 0u); }
__device__ __forceinline__ uint2 item_at(const DownItems &s, int index, int cols)
{
    const uint2 w = __ldcg(s.items + index / cols);
    return make_uint2(w.x << 8 | (uint32_t)(index % cols), w.y);
}
// k-blocks of an item of the down projection
__device__ __forceinline__ int kb_list(const DownItems &s, uint32_t uni) { return __popc(uni) * s.kpe; }
template <typename Items> __device__ __forceinline__ int kb_list(const Items &, uint32_t) { return 0; }

// Lists a down projection builds before its first tile.  Launches without any do without the code: carrying it cost a short layer
// call 1 us, whether it ran or not.
struct NoLists {};
template <int N> struct ListsOf { typedef d2d_list_jobs<N> type; };
template <> struct ListsOf<0> { typedef NoLists type; };
__device__ __forceinline__ void build_lists(const NoLists &, int, int, int, uint8_t *) {}
// by the epilogue warps, one mask word of one layer per CTA; scratch in the output buffers, which nothing uses yet
template <int N> __device__ __forceinline__ void build_lists(const d2d_list_jobs<N> &j, int T, int ew, int lane, uint8_t *scratch)
{
    for (int i = (int)blockIdx.x; i < j.n * j.W; i += (int)gridDim.x) {
        const auto sync = [] { asm volatile("bar.sync 1, 512;" ::: "memory"); };
        const int l = N == 1 ? 0 : i / j.W;
        d2d_lists::lists_of_word<16>(j.l[l], i - l * j.W, T, j.E, j.W, ew, lane, reinterpret_cast<uint16_t *>(scratch),
                                        reinterpret_cast<int *>(scratch + 2048), sync);
        sync();
    }
}
inline void set_lists(NoLists &, const d2d_gemm_args &) {}
template <int N> void set_lists(d2d_list_jobs<N> &j, const d2d_gemm_args &g)
{
    j.n = g.lists.n; j.T = g.lists.T; j.E = g.lists.E; j.W = g.lists.W;
    for (int l = 0; l < N; ++l) j.l[l] = g.lists.l[l];
}

// Tile index -> (row tile, column tile).  Plain order is row-major: CTAs that run together share a few rows of A and
// sweep all of B, so B is streamed from HBM once per wave when A and B together exceed L2.  With bands, the tiles of
// `band` consecutive row tiles are walked column by column: the band's rows of A stay in L2 while B is streamed once
// per band.
__device__ __forceinline__ void tile_coords(int tile, int rows, int cols, int band, int &r, int &c)
{
    if (band <= 0) { r = tile / cols; c = tile - r * cols; return; }
    const int per_band = band * cols;
    const int b = tile / per_band, idx = tile - b * per_band;
    const int h = rows - b * band < band ? rows - b * band : band;      // height of this band (the last may be short)
    c = idx / h;
    r = b * band + (idx - c * h);
}


// 16 accumulator columns -> 16 output values: bias (16 consecutive bf16 entries, zeros if there is none), activation.
template <int EPI, int ACT, bool GATED>
__device__ __forceinline__ void epilogue_16(const uint32_t (&r)[16], const uint32_t (&g)[16], float (&v)[16], const uint4 (&bias_w)[2])
{
    float bias[16];
    const uint32_t w[8] = {bias_w[0].x, bias_w[0].y, bias_w[0].z, bias_w[0].w, bias_w[1].x, bias_w[1].y, bias_w[1].z, bias_w[1].w};
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        bias[2 * j] = __uint_as_float(w[j] << 16);
        bias[2 * j + 1] = __uint_as_float(w[j] & 0xffff0000u);
    }
    if (EPI == D2D_EPI_UP_MASKED) {
        // math on pairs; the selection is applied by the caller on the packed bf16 words (each 8-column half belongs to one
        // expert)
#pragma unroll
        for (int j = 0; j < 16; j += 2) {
            // first accumulator = up projection (+ bias), second = gate
            const uint64_t z = add2(pack2(__uint_as_float(r[j]), __uint_as_float(r[j + 1])), pack2(bias[j], bias[j + 1]));
            const uint64_t h = GATED ? mul2(fast_act2<ACT>(pack2(__uint_as_float(g[j]), __uint_as_float(g[j + 1]))), z)
                                     : fast_act2<ACT>(z);
            unpack2(h, v[j], v[j + 1]);
        }
        return;
    }
#pragma unroll
    for (int j = 0; j < 16; ++j) {
        float z = __uint_as_float(r[j]) + bias[j];
        if (EPI == D2D_EPI_RELU_BF16) z = fmaxf(z, 0.0f);
        if (EPI == D2D_EPI_ABS_F32) z = fabsf(z);
        v[j] = z;
    }
}

// Same result with every bound checked (ragged last column tile, odd leading dimension, odd expert sizes).
// Statically indexed and inlined: an out-of-line version forced the accumulator registers onto the stack.
template <int EPI, int ACT, bool GATED>
__device__ __forceinline__ void epilogue_16_slow(const uint32_t (&r)[16], const uint32_t (&g)[16], const __nv_bfloat16 *bias,
                                                 void *out, int row, int M, int col0, int N, uint32_t keep)
{
    if (row >= M) return;
#pragma unroll
    for (int j = 0; j < 16; ++j) {
        if (col0 + j < N) {
            float z = __uint_as_float(r[j]) + (bias ? __bfloat162float(bias[col0 + j]) : 0.0f);
            if (EPI == D2D_EPI_RELU_BF16) z = fmaxf(z, 0.0f);
            if (EPI == D2D_EPI_ABS_F32) z = fabsf(z);
            if (EPI == D2D_EPI_UP_MASKED) {
                const float h = GATED ? fast_act<ACT>(__uint_as_float(g[j])) * z : fast_act<ACT>(z);
                z = ((keep >> j) & 1u) ? h : 0.0f;
            }
            if (EPI == D2D_EPI_PARTIAL_F32) atomicAdd((float *)out + (size_t)row * N + col0 + j, z);
            else if (EPI == D2D_EPI_ABS_F32) ((float *)out)[(size_t)row * N + col0 + j] = z;
            else ((__nv_bfloat16 *)out)[(size_t)row * N + col0 + j] = __float2bfloat16_rn(z);
        }
    }
}

constexpr int N_EPI_WARPS = 16;
constexpr int OUT_BUF_BYTES = BM * 128;          // 128 rows x 64 bf16 columns of output on their way to a TMA store, two buffers
constexpr int STAGE_BUDGET = 192 * 1024;         // shared memory for operand stages beside them
constexpr int NTHREADS_V2 = 64 + 32 * N_EPI_WARPS;

__host__ __device__ constexpr int pow2_at_least(int v) { return v <= 32 ? 32 : v <= 64 ? 64 : v <= 128 ? 128 : v <= 256 ? 256 : 512; }

// Persistent kernel: CTA c computes tiles c, c + gridDim.x, ... (128 x BN each, column tiles
// fastest).  PAIR: two CTAs of a cluster compute 256 x BN tiles with tcgen05.mma.cta_group::2: each stages its own 128 rows
// of A and HALF of the BN rows of B, the leader (rank 0) issues the MMAs, each CTA's tensor memory receives its own 128 rows.
// A k-block then brings 16 + BN / 16 KB into an SM instead of 16 + BN / 8: the fill from L2 (about 117 GB/s per SM), not
// the tensor pipe, bounds the single-CTA main loop.  Two accumulator buffers in TMEM let the epilogue of one tile overlap the MMAs of the
// next.  GATED: two B tiles (up, gate) share the A tile; the epilogue forms A(gate) * (up + bias).
template <int BN, int STAGES, int EPI, int ACT, bool GATED, bool PAIR, int LISTS, int SORTED>
__global__ void __launch_bounds__(NTHREADS_V2) __maxnreg__(GATED ? 96 : 80)
gemm_tc_kernel(const __grid_constant__ CUtensorMap tm_a, const __grid_constant__ CUtensorMap tm_b,
               const __grid_constant__ CUtensorMap tm_b2, const __grid_constant__ CUtensorMap tm_out, EpiParams ep, int M, int N, int K, int k_splits,
               const typename ListsOf<LISTS>::type lists, const typename ItemsOf<SORTED>::type items)
{
    static_assert(SORTED == SORTED_NONE || (!GATED && !PAIR && LISTS == 0), "lists of work: plain layers, single CTAs");
    constexpr int TM = PAIR ? 2 * BM : BM;                // rows of the tile a CTA (pair) computes
    // rows of B this CTA stages (of each matrix; a gated pair: the leader the up rows, its peer the gate rows, all BN of them)
    constexpr int B_ROWS = PAIR && !GATED ? BN / 2 : BN;
    constexpr int A_BYTES = BM * BK * 2;
    constexpr int B_BYTES = B_ROWS * BK * 2;
    constexpr int STAGE_BYTES = A_BYTES + (GATED && !PAIR ? 2 : 1) * B_BYTES;
    constexpr int BUF_COLS = pow2_at_least(GATED ? 2 * BN : BN);    // TMEM columns per accumulator buffer
    constexpr int TMEM_COLS = 2 * BUF_COLS;
    constexpr int COLS_PER_WARP = BN / 4;                            // four epilogue warps share a TMEM lane quadrant
    static_assert(TMEM_COLS <= 512 && BN % 64 == 0 && BN <= 256, "tile width");

    // Swizzle atoms are 1024-byte aligned.  224 KB at most, so that a small CTA of the list-building kernels, which run beside
    // this one, still finds 2 KB (and, with 80 registers per thread here, its registers) on the SM.
    extern __shared__ __align__(1024) uint8_t smem[];
    __shared__ uint64_t bar_full[STAGES], bar_empty[STAGES], bar_acc_full[2], bar_acc_empty[2];
    __shared__ uint32_t tmem_base_holder;
    // what the epilogue's leader publishes (per buffer parity): go on (or the work is done, or a wait ran out), tile coordinates
    __shared__ volatile int epi_go[2], epi_m0[2], epi_n0[2], epi_prob[2];
    // dynamic scheduling: the producer draws work items from a global counter and hands them to the MMA thread and
    // to the epilogue through a two-slot ring (a CTA that starts late, or gets slow tiles, simply draws fewer)
    __shared__ uint64_t sched_full[2], sched_empty[2];
    __shared__ volatile int sched_item[2];
    __shared__ volatile uint32_t sched_uni[2];                       // down projection by list: experts of the tile
    uint8_t *out_s = smem + (size_t)STAGES * STAGE_BYTES;            // two output buffers behind the operand stages
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;      // warp-uniform: roles, columns
    const int nkb = (K + BK - 1) / BK;
    const int n_tiles = (N + BN - 1) / BN;
    // work item = (output tile, K split); with k_splits > 1 every item accumulates a slice of K and the
    // epilogue adds its partial sums to a float32 buffer (small-M problems that would leave most SMs idle)
    const int tiles_pp = ((M + TM - 1) / TM) * n_tiles;            // output tiles per problem
    const int total_tiles = tiles_pp * ep.batch * k_splits;
    const int rank = PAIR ? (int)(blockIdx.x & 1) : 0;              // 0: the CTA that issues the MMAs
    const int worker = PAIR ? (int)(blockIdx.x >> 1) : (int)blockIdx.x;
    const int n_workers = PAIR ? (int)(gridDim.x >> 1) : (int)gridDim.x;

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(smem_u32(&bar_full[s]), 1);
            mbar_init(smem_u32(&bar_empty[s]), 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(smem_u32(&bar_acc_full[b]), 1);
            mbar_init(smem_u32(&bar_acc_empty[b]), PAIR ? 2 * N_EPI_WARPS : N_EPI_WARPS);
            mbar_init(smem_u32(&sched_full[b]), 1);
            // a slot's readers: the MMA thread and the epilogue's leader; of a pair also the peer's producer and epilogue leader
            mbar_init(smem_u32(&sched_empty[b]), PAIR ? 4 : 2);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        if (PAIR) {
            asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_holder)),
                         "r"((uint32_t)TMEM_COLS) : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
        } else {
            asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_holder)),
                         "r"((uint32_t)TMEM_COLS)
                         : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (PAIR) cluster_sync_all();          // the peer's barriers are initialised before anything signals them
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_base = tmem_base_holder;
    // Programmatic dependent launch: everything above (barriers, TMEM)
    // may run while the previous kernel of the stream drains; nothing below starts before that kernel has completed
    // and its writes are visible.  The next kernel of the stream may be scheduled onto SMs as this grid frees them.
    // With late_wait only the epilogue depends on that kernel (the selection mask written by the router): the
    // operand loads and the MMAs of the first tiles then overlap it, and only the epilogue warps wait.
    const bool dyn = SORTED != SORTED_NONE || ep.tile_counter != nullptr;
    // early_b: the B operand (weights) does not depend on the previous kernel either, so the producer requests the B
    // tiles of its first k-blocks BEFORE it waits for that kernel and only the A tiles after (static schedule only)
    const bool early_b = !PAIR && !dyn && !ep.late_wait && ep.n_sel == nullptr;
    if (warp >= 2 || (!ep.late_wait && !(early_b && warp == 0))) asm volatile("griddepcontrol.wait;" ::: "memory");
    // (router's hidden layer: only threads that have waited let the next kernel start, see router_scores_kernel)
    if (EPI != D2D_EPI_RELU_BF16 || !early_b || warp != 0) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    // density-adaptive dispatch: below the crossover the gathered kernel, launched next to this one, does the work
    // (every thread has passed the dependency wait here: the host never combines n_sel with late_wait)
    const bool run = ep.n_sel == nullptr || ((long long)__ldcg(ep.n_sel) > ep.n_sel_max) == (SORTED == SORTED_NONE);

    // Waits for barriers that threads of the pair's other CTA arrive at: the ring of work items (its slots are written and read
    // across the pair) and the accumulators handed back.  The operand and accumulator-full barriers are completed by the copy
    // engine and the tensor core.
    auto peer_wait = [&](uint64_t *bar, uint32_t parity) { return mbar_wait<64, 32, PAIR>(smem_u32(bar), parity, ep.status); };
    auto peer_wait_warp = [&](uint64_t *bar, uint32_t parity) { return mbar_wait_warp<PAIR>(smem_u32(bar), parity, ep.status); };

    if (!run) {
        // nothing to do
    } else if (SORTED != SORTED_NONE && warp == 0) {
        // ------------------------------------------------------------------ TMA producer, from a list of work
        if constexpr (SORTED != SORTED_NONE) {
            if (lane == 0) {
                const int total = n_items(items, total_tiles);
                // Items are drawn from the counter as in the dynamic schedule below, but two ahead: while one is worked on, the word
                // of the next is on its way and the number of the one behind that is being drawn.
                int index = worker, next = index < total ? n_workers + atomicAdd(ep.tile_counter, 1) : total;
                uint2 word = index < total ? item_at(items, index, n_tiles) : make_uint2(0u, 0u);
                uint32_t it = 0;
                bool ok = true;
                for (uint32_t local = 0; ok; ++local) {
                    const uint32_t sl = local & 1u;
                    ok = peer_wait(&sched_empty[sl], ((local >> 1) & 1u) ^ 1u);
                    if (!ok) break;
                    sched_item[sl] = index < total ? (int)word.x : -1;
                    sched_uni[sl] = word.y;
                    mbar_arrive(smem_u32(&sched_full[sl]));
                    if (index >= total) break;
                    const int m0 = (int)(word.x >> 8) * BM, n0 = (int)(word.x & 255u) * BN;
                    uint32_t uni = word.y;
                    index = next;
                    word = index < total ? item_at(items, index, n_tiles) : make_uint2(0u, 0u);
                    next = index < total ? n_workers + atomicAdd(ep.tile_counter, 1) : index;
                    const auto block = [&](int kb) {
                        const uint32_t s = it % STAGES, full = smem_u32(&bar_full[s]), dst = smem_u32(smem + (size_t)s * STAGE_BYTES);
                        ok = mbar_wait(smem_u32(&bar_empty[s]), ((it / STAGES) & 1u) ^ 1u, ep.status);
                        if (!ok) return;
                        mbar_expect_tx(full, (uint32_t)STAGE_BYTES);
                        tma_load_2d(dst, &tm_a, kb * BK, m0, full);
                        tma_load_2d(dst + A_BYTES, &tm_b, kb * BK, n0, full);
                        ++it;
                    };
                    if constexpr (SORTED == SORTED_UP) {
                        for (int kb = 0; kb < nkb && ok; ++kb) block(kb);
                    } else {
                        // the k-blocks of the experts that some token of the tile keeps
                        for (; uni && ok; uni &= uni - 1u) {
                            const int kb0 = (__ffs(uni) - 1) * items.kpe;
                            for (int k = 0; k < items.kpe && ok; ++k) block(kb0 + k);
                        }
                    }
                }
                // every worker that had an item draws one past the end, `total` values are drawn in all: the last leaves zero
                if (index == n_workers + total - 1) *ep.tile_counter = 0;
            }
        }
    } else if (warp == 0) {
        // ------------------------------------------------------------------ TMA producer
        if (lane == 0) {
            uint32_t it = 0, pre = 0;
            bool ok = true;
            // B tile(s) of k-block kb into the stage at dst (single-CTA form)
            auto load_b = [&](uint32_t dst, uint32_t full, int kb, int n0) {
                if (GATED && ep.gate_cat) {
                    // up rows [n0, n0+BN) and gate rows [n0, n0+BN) are adjacent in the interleaved copy: one
                    // 2*BN-row box (the producer thread's time per k-block is what bounds the gated main loop)
                    tma_load_2d(dst + A_BYTES, &tm_b, kb * BK, 2 * n0, full);
                } else {
                    tma_load_2d(dst + A_BYTES, &tm_b, kb * BK, n0, full);
                    if (GATED) tma_load_2d(dst + A_BYTES + B_BYTES, &tm_b2, kb * BK, n0, full);
                }
            };
            for (uint32_t local = 0; ok; ++local) {
                int item = worker + (int)local * n_workers;
                if (dyn) {
                    const uint32_t sl = local & 1u, use = local >> 1;
                    if (rank != 0) {
                        // the leader draws for the pair
                        ok = peer_wait(&sched_full[sl], use & 1u);
                        if (!ok) break;
                        item = sched_item[sl];
                        mbar_arrive_cluster(map_to_cta(smem_u32(&sched_empty[sl]), 0));
                        if (item < 0) break;
                    } else {
                        ok = peer_wait(&sched_empty[sl], (use & 1u) ^ 1u);
                        if (!ok) break;
                        // A worker's first item is its own index (no round trip to the counter before the first loads); the
                        // counter hands out the items from n_workers on.  Every worker draws exactly one value past the end,
                        // total_tiles draws in all: whoever gets the last one leaves the counter at zero for the next launch.
                        if (local > 0) {
                            const int c = atomicAdd(ep.tile_counter, 1);
                            if (c == total_tiles - 1) *ep.tile_counter = 0;
                            item = n_workers + c;
                        }
                        const int got = item < total_tiles ? item : -1;
                        sched_item[sl] = got;
                        if (PAIR) {
                            st_cluster_u32(map_to_cta(smem_u32((const void *)&sched_item[sl]), 1), (uint32_t)got);
                            mbar_arrive_cluster(map_to_cta(smem_u32(&sched_full[sl]), 1));
                        }
                        mbar_arrive(smem_u32(&sched_full[sl]));   // release: the slot's content is visible to whoever sees the phase
                    }
                }
                if (item >= total_tiles) break;
                int tile = (!GATED && k_splits == 1) ? item : item / k_splits;
                const int sp = item - tile * k_splits;
                // no split is the common case: skip the divisions (measured: faster for the plain kernels, slower for the
                // gated one, whose code layout is at its limit)
                const bool one = !GATED && k_splits == 1;
                const int kb0 = one ? 0 : (int)((long long)sp * nkb / k_splits), kb1 = one ? nkb : (int)((long long)(sp + 1) * nkb / k_splits);
                int prob = 0;
                if (ep.batch > 1) { prob = tile / tiles_pp; tile -= prob * tiles_pp; }
                int tr, tc;
                tile_coords(tile, (M + TM - 1) / TM, n_tiles, ep.band_rows, tr, tc);
                const int m0 = tr * TM + rank * BM, n0 = prob * N + tc * BN + (GATED ? 0 : rank * B_ROWS);
                const int ka = prob * K;                      // problem p reads columns [p*K, (p+1)*K) of A
                if (early_b && local == 0) {
                    // arm the first stages and request their B tiles, then wait for the previous kernel (A may be its output)
                    for (int kb = kb0; kb < kb1 && pre < (uint32_t)STAGES; ++kb, ++pre) {
                        const uint32_t full = smem_u32(&bar_full[pre]);
                        mbar_expect_tx(full, (uint32_t)STAGE_BYTES);
                        load_b(smem_u32(smem + (size_t)pre * STAGE_BYTES), full, kb, n0);
                    }
                    asm volatile("griddepcontrol.wait;" ::: "memory");
                }
                for (int kb = kb0; kb < kb1; ++kb, ++it) {
                    const uint32_t s = it % STAGES, round = it / STAGES;
                    if (it < pre) {                           // armed above, B already requested
                        // host-made fault for the failure-handling test: this stage's byte count is never reached, so the
                        // MMA warp's wait, then the epilogue's and this thread's own, run out and the CTA leaves in order
                        if (ep.test_skip_load && it == 0 && blockIdx.x == 0) continue;
                        tma_load_2d(smem_u32(smem + (size_t)s * STAGE_BYTES), &tm_a, ka + kb * BK, m0, smem_u32(&bar_full[s]));
                        continue;
                    }
                    ok = mbar_wait(smem_u32(&bar_empty[s]), (round & 1u) ^ 1u, ep.status);
                    if (!ok) break;
                    const uint32_t dst = smem_u32(smem + (size_t)s * STAGE_BYTES);
                    if (PAIR) {
                        // both CTAs' bytes are credited to the leader's barrier (where the MMAs are issued)
                        const uint32_t full = map_to_cta(smem_u32(&bar_full[s]), 0);
                        if (rank == 0) mbar_expect_tx(smem_u32(&bar_full[s]), 2u * (uint32_t)STAGE_BYTES);
                        tma_load_2d_pair(dst, &tm_a, ka + kb * BK, m0, full);
                        tma_load_2d_pair(dst + A_BYTES, GATED && rank ? &tm_b2 : &tm_b, kb * BK, n0, full);
                        continue;
                    }
                    const uint32_t full = smem_u32(&bar_full[s]);
                    mbar_expect_tx(full, (uint32_t)STAGE_BYTES);
                    tma_load_2d(dst, &tm_a, ka + kb * BK, m0, full);
                    load_b(dst, full, kb, n0);
                }
            }
        }
    } else if (warp == 1 && rank != 0) {
        // the leader's MMA warp works for both CTAs
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMA issuer
        // The whole warp walks the loop, so that waits, indices and descriptors are warp-uniform (the tensor-core
        // instructions take their operands from uniform registers); one elected lane issues the MMAs and commits.
        {
            // Gated: the up and gate tiles sit back to back in shared memory, so they are ONE K-major
            // B operand of 2*BN rows and one MMA fills both accumulators (columns [0,BN) up, [BN,2BN) gate).
            // Two N=BN instructions would each pay the full A-operand read and run at half the rate.
            const uint32_t idesc = instr_desc_bf16(TM, GATED ? 2 * BN : BN);
            uint32_t it = 0, local = 0;
            bool ok = true;
            // The tensor core accepts only a few instructions ahead, so whatever this thread executes between the last
            // MMA of one k-block and the first MMA of the next is a bubble in the MMA pipe.  The barrier of the NEXT
            // k-block is therefore tested between the MMAs of the current one (`have` carries the answer across
            // k-blocks and tiles), and nothing but the commit sits between two k-blocks whose data has landed.
            bool have = false;
            for (;; ++local) {
                int item = worker + (int)local * n_workers;
                uint32_t uni = 0u;
                if (dyn) {
                    const uint32_t sl = local & 1u, su = local >> 1;
                    ok = peer_wait_warp(&sched_full[sl], su & 1u);
                    if (!ok) break;
                    item = sched_item[sl];
                    if (SORTED == SORTED_DOWN) uni = sched_uni[sl];
                    __syncwarp();                              // every lane has read the slot before it is handed back
                    if (elect_one()) mbar_arrive(smem_u32(&sched_empty[sl]));
                    if (item < 0) break;
                }
                if (SORTED == SORTED_NONE && item >= total_tiles) break;
                const int sp = (!GATED && k_splits == 1) ? 0 : item % k_splits;
                // no split is the common case: skip the divisions (measured: faster for the plain kernels, slower for the
                // gated one, whose code layout is at its limit)
                const bool one = !GATED && k_splits == 1;
                const int kb0 = one ? 0 : (int)((long long)sp * nkb / k_splits),
                          kb1 = SORTED == SORTED_DOWN ? kb_list(items, uni) : one ? nkb : (int)((long long)(sp + 1) * nkb / k_splits);
                const uint32_t buf = local & 1u, use = local >> 1;
                ok = peer_wait_warp(&bar_acc_empty[buf], (use & 1u) ^ 1u);   // epilogue drained this buffer
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t acc = tmem_base + buf * BUF_COLS;
                for (int kb = kb0; kb < kb1; ++kb, ++it) {
                    const uint32_t s = it % STAGES, round = it / STAGES;
                    if (!have) {
                        ok = mbar_wait_warp(smem_u32(&bar_full[s]), round & 1u, ep.status);
                        if (!ok) break;
                    }
                    const uint32_t a_addr = smem_u32(smem + (size_t)s * STAGE_BYTES);
                    const uint64_t da = smem_desc_sw128(a_addr);
                    const uint64_t db = smem_desc_sw128(a_addr + A_BYTES);
                    const uint64_t db2 = smem_desc_sw128(a_addr + A_BYTES + B_BYTES);
                    const uint32_t s_next = (it + 1) % STAGES, round_next = (it + 1) / STAGES;
                    auto issue = [&](int k) {
                        const uint64_t koff = (uint64_t)((k * UMMA_K * 2) >> 4);    // 32 bytes per K step inside the swizzle row
                        const uint32_t accum = (kb > kb0 || k != 0) ? 1u : 0u;
                        if (PAIR) umma_bf16_pair(acc, da + koff, db + koff, idesc, accum);
                        else umma_bf16(acc, da + koff, db + koff, idesc, accum);
                    };
                    if (elect_one()) {
#pragma unroll
                        for (int k = 0; k < BK / UMMA_K - 1; ++k) issue(k);
                    }
                    // before the last MMA of this k-block: has the next k-block (of this or the next tile) landed?
                    have = __all_sync(0xffffffffu, mbar_test(smem_u32(&bar_full[s_next]), round_next & 1u));
                    if (elect_one()) {
                        issue(BK / UMMA_K - 1);
                        if (PAIR) umma_commit_pair(smem_u32(&bar_empty[s]));
                        else umma_commit(smem_u32(&bar_empty[s]));   // stage reusable once these MMAs have read it
                    }
                    __syncwarp();
                }
                if (!ok) break;
                if (elect_one()) {                           // accumulator of this tile complete
                    if (PAIR) umma_commit_pair(smem_u32(&bar_acc_full[buf]));
                    else umma_commit(smem_u32(&bar_acc_full[buf]));
                }
                __syncwarp();
            }
        }
    } else {
        // ------------------------------------------------------------------ epilogue (warps 2..17)
        // Sixteen warps (four per TMEM lane quadrant) so that the per-element math of one warp hides
        // the TMEM-load and MUFU latencies of another.  A warp walks its BN/4 columns in 16-column
        // units; the load of the next unit is in flight while the current one is processed, and the
        // rarely taken paths are out of line so that the unrolled body stays small (a 32-column,
        // everything-inline version of this epilogue was instruction-fetch bound).
        const int ew = warp - 2;
        const int quad = warp & 3;                          // TMEM lanes this warp may touch
        const int part = ew >> 2;                           // which 16 of every 64 columns of the tile
        constexpr int N_UNITS = COLS_PER_WARP / 16;
        auto acc_release = [&](uint32_t b) {                // to the MMA warp (the leader's)
            if (PAIR) mbar_arrive_cluster(map_to_cta(smem_u32(&bar_acc_empty[b]), 0));
            else mbar_arrive(smem_u32(&bar_acc_empty[b]));
        };
        uint32_t out_n = 0;                                 // output buffers used so far
        for (int i = (int)blockIdx.x * (N_EPI_WARPS * 32) + (int)threadIdx.x - 64; i < ep.zero_n; i += (int)gridDim.x * (N_EPI_WARPS * 32))
            ep.zero[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        build_lists(lists, M, ew, lane, out_s);
        for (uint32_t local = 0;; ++local) {
            const uint32_t buf = local & 1u, use = local >> 1;
            // ONE thread takes the item from the ring, works out its coordinates (integer divisions), waits for the accumulator
            // and publishes the outcome; the other epilogue warps sleep on a hardware barrier.  Sixteen pollers measurably slow
            // the producer and MMA threads, whose own barrier tests share the same unit.
            if (ew == 0 && lane == 0) {
                int item = worker + (int)local * n_workers;
                bool go = true;
                if (dyn) {
                    go = peer_wait(&sched_full[buf], use & 1u);
                    if (go) {
                        item = sched_item[buf];
                        // (problem number: none here; whether the tile's tokens keep nothing)
                        if (SORTED != SORTED_NONE) epi_prob[buf] = SORTED == SORTED_DOWN && sched_uni[buf] == 0u;
                        if (PAIR) mbar_arrive_cluster(map_to_cta(smem_u32(&sched_empty[buf]), 0));
                        else mbar_arrive(smem_u32(&sched_empty[buf]));
                    }
                }
                go = go && item >= 0 && (SORTED != SORTED_NONE || item < total_tiles);
                if (SORTED != SORTED_NONE) {
                    if (go) {
                        epi_m0[buf] = (item >> 8) * BM; epi_n0[buf] = (item & 255) * BN;
                        go = mbar_wait(smem_u32(&bar_acc_full[buf]), use & 1u, ep.status);
                    }
                } else if (go) {
                    int tile = (!GATED && k_splits == 1) ? item : item / k_splits;
                    int prob = 0, tr, tc;
                    const int sum = EPI == D2D_EPI_PARTIAL_F32 ? (item - tile * k_splits) / ep.slices_per_sum : 0;
                    if (ep.batch > 1) { prob = tile / tiles_pp; tile -= prob * tiles_pp; }
                    prob += sum * ep.batch;                    // the buffers' problems follow one another
                    tile_coords(tile, (M + TM - 1) / TM, n_tiles, ep.band_rows, tr, tc);
                    epi_m0[buf] = tr * TM + rank * BM; epi_n0[buf] = tc * BN; epi_prob[buf] = prob;
                    go = mbar_wait(smem_u32(&bar_acc_full[buf]), use & 1u, ep.status);
                }
                epi_go[buf] = go ? 1 : 0;
            }
            asm volatile("bar.sync 1, %0;" ::"r"(N_EPI_WARPS * 32) : "memory");
            if (!epi_go[buf]) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const int m0 = epi_m0[buf], n0 = epi_n0[buf], prob = SORTED == SORTED_NONE ? epi_prob[buf] : 0;
            const bool nothing = SORTED == SORTED_DOWN && epi_prob[buf] != 0;
            // down projection by list: the tokens of the two rows whose 16-byte pieces this thread stores
            int token[2] = {-1, -1};
            if constexpr (SORTED == SORTED_DOWN) {
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const int at = m0 + quad * 32 + 16 * i + 4 * part + (lane >> 3);
                    if (at < M) token[i] = __ldcg(items.order + at);
                }
            }
            // this problem's bias entries and output matrix
            const __nv_bfloat16 *bias_g = ep.bias ? ep.bias + prob * N : nullptr;
            void *out_p = (char *)ep.out + (size_t)prob * M * N * ((EPI == D2D_EPI_ABS_F32 || EPI == D2D_EPI_PARTIAL_F32) ? 4 : 2);
            const int row = m0 + quad * 32 + lane;
            // Selection of this row, for the 8-column groups of this warp's columns (expert sizes that are multiples of 8: a group
            // belongs to one expert): the experts of the range are consecutive bits of at most two mask words, loaded here and
            // looked at after the first unit's math; bit h of kbits = group h.  Which expert a group belongs to is the same for
            // all rows.  (Selecting among all words of the row in registers, group by group, was 3 of 18 instructions per
            // element.)
            const int colw = n0 + part * 16;                // unit u: columns colw + 64 u + 0..15
            const uint32_t *mrow = nullptr;
            uint32_t kbits = 0xffffffffu, mw0 = 0u, mw1 = 0u, e0 = 0u;
            if (EPI == D2D_EPI_UP_MASKED && ep.mask && row < M) {
                mrow = ep.mask + (size_t)row * ep.mask_words;
                if ((ep.expert_size & 7) == 0 && colw < N) {
                    e0 = __umulhi((uint32_t)colw, ep.inv_expert_size);
                    const int wi = (int)(e0 >> 5);
                    mw0 = __ldg(mrow + wi);
                    mw1 = wi + 1 < ep.mask_words ? __ldg(mrow + wi + 1) : 0u;
                }
            }
            const uint32_t tbase = tmem_base + buf * BUF_COLS + ((uint32_t)(quad * 32) << 16) + (uint32_t)(part * 16);

            const bool mask_on = EPI == D2D_EPI_UP_MASKED && ep.mask != nullptr;                         // CTA-uniform
            // The common case gets a loop of its own with nothing else in it (the epilogue is sensitive to its
            // instruction-cache footprint): a full-width tile, vector-aligned rows and expert sizes that are multiples of 8.
            // Everything else (ragged last column tile, odd sizes) goes through the compact generic loop below.
            // (lists of work come with whole column tiles only)
            const bool fast_tile = SORTED != SORTED_NONE || (N & 7) == 0 && n0 + BN <= N && (!mask_on || (ep.expert_size & 7) == 0);
            uint32_t ra[16], rb[GATED ? 1 : 16], ga[GATED ? 16 : 1];
            if (fast_tile) {
                // Non-gated: the next unit's accumulators are prefetched into a second register set.  Gated tiles need
                // two accumulators per column; a second set would spill, so each unit is loaded when it is needed and
                // the other epilogue warps of the SM sub-partition cover the latency.
                if (!GATED) tmem_ld16_issue(tbase, ra);
#pragma unroll
                for (int u = 0; u < N_UNITS; ++u) {             // at most 4 units
                    const int col0 = colw + u * 64;
                    uint4 bias_w[2] = {make_uint4(0, 0, 0, 0), make_uint4(0, 0, 0, 0)};       // the same for all lanes, out of L1
                    if (EPI != D2D_EPI_PARTIAL_F32 && ep.bias) {
                        bias_w[0] = __ldg(reinterpret_cast<const uint4 *>(bias_g + col0));
                        bias_w[1] = __ldg(reinterpret_cast<const uint4 *>(bias_g + col0 + 8));
                    }
                    uint32_t (&r)[16] = GATED ? ra : ((u & 1) ? reinterpret_cast<uint32_t (&)[16]>(rb) : ra);
                    uint32_t (&g)[16] = reinterpret_cast<uint32_t (&)[16]>(ga);
                    if (GATED) {
                        tmem_ld16_issue(tbase + u * 64, ra);
                        tmem_ld16_issue(tbase + u * 64 + BN, reinterpret_cast<uint32_t (&)[16]>(ga));
                    }
                    tmem_ld_wait();                                               // this unit's accumulators have landed
                    if (!GATED && u + 1 < N_UNITS)                                // the next unit's load overlaps the math below
                        tmem_ld16_issue(tbase + (u + 1) * 64, (u & 1) ? ra : reinterpret_cast<uint32_t (&)[16]>(rb));

                    if (SORTED == SORTED_DOWN && nothing) {
#pragma unroll
                        for (int j = 0; j < 16; ++j) r[j] = 0u;
                    }
                    float v[16];
                    epilogue_16<EPI, ACT, GATED>(r, g, v, bias_w);
                    if (EPI == D2D_EPI_UP_MASKED && u == 0 && mask_on) {
                        const uint32_t bits = __funnelshift_r(mw0, mw1, e0 & 31u);
                        kbits = 0u;
#pragma unroll
                        for (int h = 0; h < 2 * N_UNITS; ++h)
                            kbits |= ((bits >> (__umulhi((uint32_t)(colw + 64 * (h >> 1) + 8 * (h & 1)), ep.inv_expert_size) - e0)) & 1u) << h;
                    }
                    // all ones where the token keeps the expert of the unit's first / second eight columns
                    const uint32_t keep2[2] = {(uint32_t)((int)(kbits << (31 - 2 * u)) >> 31), (uint32_t)((int)(kbits << (30 - 2 * u)) >> 31)};
                    if (u == N_UNITS - 1) {
                        // all of this warp's TMEM reads of the buffer are complete: hand it back to the MMA warp
                        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                        __syncwarp();
                        if (lane == 0) acc_release(buf);
                    }
                    if (EPI == D2D_EPI_PARTIAL_F32) {
                        if (row < M) {
                            float *o = (float *)out_p + (size_t)row * N + col0;
#pragma unroll
                            for (int j = 0; j < 16; j += 4)
                                asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(o + j), "f"(v[j]), "f"(v[j + 1]),
                                             "f"(v[j + 2]), "f"(v[j + 3]) : "memory");
                        }
                    } else if (EPI == D2D_EPI_ABS_F32) {
                        if (row < M) {
                            float *o = (float *)out_p + (size_t)row * N + col0;
#pragma unroll
                            for (int j = 0; j < 16; j += 4) *reinterpret_cast<float4 *>(o + j) = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
                        }
                    } else {
                        uint32_t pk[8];
#pragma unroll
                        for (int j = 0; j < 8; ++j) {
                            __nv_bfloat162 t = __floats2bfloat162_rn(v[2 * j], v[2 * j + 1]);
                            pk[j] = *reinterpret_cast<uint32_t *>(&t);
                            // selection: an expert the token did not keep contributes zeros (also when its
                            // pre-activations are not finite)
                            if (EPI == D2D_EPI_UP_MASKED) pk[j] &= keep2[j >> 2];
                        }
                        // The sixteen warps put 128 rows x 64 columns into a buffer (128-byte rows, swizzled as the TMA expects) and one
                        // thread stores it: whole 128-byte lines.  (Every thread storing 32 bytes of its own row took 15 % of the
                        // kernel: 112 us against 96 us without stores on the ViT-shaped up projection.)
                        uint8_t *o = out_s + (out_n & 1u) * OUT_BUF_BYTES + (quad * 32 + lane) * 128;
                        *reinterpret_cast<uint4 *>(o + (((2 * part) ^ (lane & 7)) << 4)) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
                        *reinterpret_cast<uint4 *>(o + (((2 * part + 1) ^ (lane & 7)) << 4)) = make_uint4(pk[4], pk[5], pk[6], pk[7]);
                        if constexpr (SORTED == SORTED_DOWN) {
                            // rows go to their tokens: eight threads store 128 bytes of a row (the buffer is written again two units
                            // on, behind the barrier of the next)
                            asm volatile("bar.sync %0, 128;" ::"r"(2 + quad) : "memory");
#pragma unroll
                            for (int i = 0; i < 2; ++i) {
                                const int rr = 16 * i + 4 * part + (lane >> 3), ch = lane & 7;
                                const uint4 w = *reinterpret_cast<const uint4 *>(out_s + (out_n & 1u) * OUT_BUF_BYTES + (quad * 32 + rr) * 128 +
                                                                                 ((ch ^ (rr & 7)) << 4));
                                if (token[i] >= 0)
                                    *reinterpret_cast<uint4 *>((__nv_bfloat16 *)out_p + (size_t)token[i] * N + n0 + u * 64 + ch * 8) = w;
                            }
                            ++out_n;
                            continue;
                        }
                        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                        // the store before this one has read the other buffer: free for everybody behind the barrier
                        if (part == 0 && lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
                        asm volatile("bar.sync %0, 128;" ::"r"(2 + quad) : "memory");
                        if (part == 0 && lane == 0) {
                            asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.bulk_group [%0, {%1, %2, %3}], [%4];"
                                         ::"l"(&tm_out), "r"(n0 + u * 64), "r"(m0 + quad * 32), "r"(prob),
                                         "r"(smem_u32(out_s + (out_n & 1u) * OUT_BUF_BYTES + quad * 32 * 128)) : "memory");
                            asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                        }
                        ++out_n;
                    }
                }
            } else {
                // generic loop: one unit at a time, every bound checked, any expert size
                // expert that owns the first column of this warp's range (one division per tile; advanced incrementally)
                int e = 0, lo = 0, widx = -1;
                uint32_t word = 0u;
                if (EPI == D2D_EPI_UP_MASKED && mrow) {
                    e = colw / ep.expert_size;
                    lo = e * ep.expert_size - colw;         // first column of expert e relative to the current unit (<= 0)
                }
                uint32_t (&g)[16] = reinterpret_cast<uint32_t (&)[16]>(ga);
#pragma unroll 1
                for (int u = 0; u < N_UNITS; ++u) {
                    const int col0 = colw + u * 64;
                    if (col0 >= N) break;                       // warp-uniform (ragged last column tile)
                    tmem_ld16_issue(tbase + u * 64, ra);
                    if (GATED) tmem_ld16_issue(tbase + u * 64 + BN, g);
                    uint32_t keep = 0xffffu;
                    if (mask_on && mrow) {
                        keep = 0u;
                        const int s = ep.expert_size;
                        int ee = e, l = lo;
                        while (l < 16) {
                            if ((ee >> 5) != widx) {
                                widx = ee >> 5;
                                word = __ldg(mrow + widx);
                            }
                            const int hi = l + s;
                            if ((word >> (ee & 31)) & 1u) {
                                const int a = l < 0 ? 0 : l, b2 = hi > 16 ? 16 : hi;
                                keep |= ((1u << b2) - 1u) & ~((1u << a) - 1u);
                            }
                            l = hi;
                            ++ee;
                        }
                        // advance to the expert that owns the first column of the next unit
                        lo -= 64;
                        while (lo + s <= 0) { lo += s; ++e; }
                    }
                    tmem_ld_wait();
                    epilogue_16_slow<EPI, ACT, GATED>(ra, g, bias_g, out_p, row, M, col0, N, keep);
                }
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                __syncwarp();
                if (lane == 0) acc_release(buf);
            }
        }
        // the buffers may not go away, nor the kernel count as finished, before the last stores are done
        if (part == 0 && lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    }

    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (PAIR) cluster_sync_all();          // neither CTA releases shared memory or TMEM while the other may still use it
    if (PAIR && warp == 1)
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)TMEM_COLS) : "memory");
    if (!PAIR && warp == 1)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)TMEM_COLS) : "memory");
}

// ------------------------------------------------------------------------------------------ host side

// Band height (in row tiles) for the tile walk, 0 = plain row-major.  Row-major order re-reads B once per wave of
// CTAs, which is free while B stays in L2 (126 MB) beside the streaming A; only a large B (Llama-sized weights) needs
// bands.  The band is sized so that its rows of A take about 32 MB (measured best on the Llama-shaped layer: 32 row
// tiles of 1 MB, 1050 us against 1427 us for the up projection).
int band_rows_for(int M, int N, int K, int tile_m, bool gated)
{
    (void)M;
    const double b_bytes = 2.0 * N * K * (gated ? 2 : 1);
    if (b_bytes < 48e6) return 0;
    const char *e = getenv("D2D_GEMM_BAND");
    if (e) return atoi(e);
    int band = (int)(32e6 / (2.0 * tile_m * K) + 0.5);
    return band < 16 ? 16 : band;                           // shorter bands stream B too often (16 .. 32 measured alike)
}

// cudaFuncAttributeMaxDynamicSharedMemorySize is a per-device attribute: set it once per (kernel, device).
template <typename K> bool ensure_smem_attr(K kern, size_t smem, bool (&done)[64])
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return false;
    if (!__atomic_load_n(&done[dev], __ATOMIC_ACQUIRE)) {
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) return false;
        __atomic_store_n(&done[dev], true, __ATOMIC_RELEASE);
    }
    return true;
}

template <int BN, int EPI, int ACT, bool GATED, bool PAIR = false, int LISTS = 0, int SORTED = SORTED_NONE>
d2d_status launch(const d2d_gemm_args &g, cudaStream_t st, int slices_per_sum = 1)
{
    if constexpr ((EPI == D2D_EPI_BIAS_BF16 || EPI == D2D_EPI_PARTIAL_F32) && LISTS == 0 && SORTED == SORTED_NONE) {
        if (g.lists.n == 1) return launch<BN, EPI, ACT, GATED, PAIR, 1>(g, st, slices_per_sum);
        if (g.lists.n > 1) return launch<BN, EPI, ACT, GATED, PAIR, D2D_MAX_GROUP>(g, st, slices_per_sum);
    }
    constexpr int B_ROWS = PAIR && !GATED ? BN / 2 : BN, TM = PAIR ? 2 * BM : BM;
    constexpr int STAGE_BYTES = BM * BK * 2 + (GATED && !PAIR ? 2 : 1) * B_ROWS * BK * 2;
    constexpr int STAGES = STAGE_BUDGET / STAGE_BYTES > 8 ? 8 : STAGE_BUDGET / STAGE_BYTES;
    constexpr size_t SMEM = (size_t)STAGES * STAGE_BYTES + 2 * (size_t)OUT_BUF_BYTES;
    static_assert(SMEM <= 224 * 1024, "shared memory per CTA");
    CUtensorMap ta, tb, tb2, to = {};
    const bool gate_cat = GATED && !PAIR && g.b_cat != nullptr && g.b_cat_block == BN;
    const int batch = g.batch > 1 ? g.batch : 1;
    if (batch > 1 && (GATED || g.K % BK != 0)) return D2D_ERR_UNSUPPORTED;
    if (!d2d_tc_make_map(&ta, g.a, g.M, g.K * batch, BM)) return D2D_ERR_CUDA;
    if (gate_cat) {
        if (!d2d_tc_make_map(&tb, g.b_cat, 2 * BN * d2d_cdiv(g.N, BN), g.K, 2 * BN)) return D2D_ERR_CUDA;
        tb2 = tb;
    } else {
        if (!d2d_tc_make_map(&tb, g.b, g.N * batch, g.K, B_ROWS)) return D2D_ERR_CUDA;
        if (GATED) {
            if (!d2d_tc_make_map(&tb2, g.b_gate, g.N, g.K, B_ROWS)) return D2D_ERR_CUDA;
        } else {
            tb2 = tb;
        }
    }
    if (EPI != D2D_EPI_PARTIAL_F32 && EPI != D2D_EPI_ABS_F32 && g.N % 8 == 0) {       // (other widths: every tile takes the generic loop)
        const cuuint64_t dims[3] = {(cuuint64_t)g.N, (cuuint64_t)g.M, (cuuint64_t)batch};
        const cuuint64_t strides[2] = {(cuuint64_t)g.N * 2, (cuuint64_t)g.N * g.M * 2};
        const cuuint32_t box[3] = {64, 32, 1};
        if (!d2d_tc_encode_map(&to, false, 3, g.out, dims, strides, box)) return D2D_ERR_CUDA;
    }
    auto kern = gemm_tc_kernel<BN, STAGES, EPI, ACT, GATED, PAIR, LISTS, SORTED>;
    static bool attr_set[64] = {};
    if (!ensure_smem_attr(kern, SMEM, attr_set)) return D2D_ERR_CUDA;
    const int es = g.expert_size > 0 ? g.expert_size : 1;
    EpiParams ep{(const __nv_bfloat16 *)g.bias, g.out, g.mask, g.mask_words, es, g.status,
                 (uint32_t)((0x100000000ull + (unsigned long long)es - 1) / (unsigned long long)es),
                 g.tile_counter, (g.pdl_late_wait && !g.n_sel && d2d_tc_pdl_enabled()) ? 1 : 0, gate_cat ? 1 : 0,
                 band_rows_for(g.M, g.N, g.K, TM, GATED), batch, g.n_sel, g.n_sel_max, (float4 *)g.zero, g.zero ? (int)(g.zero_floats / 4) : 0, slices_per_sum,
                 (g.test_skip_load && !g.tile_counter && !g.pdl_late_wait && !g.n_sel) ? 1 : 0};
    typename ListsOf<LISTS>::type lists = {};
    set_lists(lists, g);
    typename ItemsOf<SORTED>::type items = {};
    set_items(items, g);
    const int k_splits = g.k_splits > 1 ? g.k_splits : 1;
    const int tiles = d2d_cdiv(g.N, BN) * d2d_cdiv(g.M, TM) * k_splits * batch;
    const int workers = PAIR ? d2d_tc_sm_count() / 2 : d2d_tc_sm_count();
    const int grid = (tiles < workers ? tiles : workers) * (PAIR ? 2 : 1);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid, 1, 1);
    cfg.blockDim = dim3(NTHREADS_V2, 1, 1);
    cfg.dynamicSmemBytes = SMEM;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = PAIR ? 2 : 1; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    // the kernel's prologue may overlap the tail of the previous kernel in the stream (see griddepcontrol.wait in the kernel)
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = d2d_tc_pdl_enabled() ? 2 : 1;
    const cudaError_t err = cudaLaunchKernelEx(&cfg, kern, ta, tb, tb2, to, ep, g.M, g.N, g.K, k_splits, lists, items);
    D2D_LAUNCHED(1);
    return err == cudaSuccess && cudaGetLastError() == cudaSuccess ? D2D_OK : D2D_ERR_CUDA;
}

// Tile with the least modelled time: rounds over the SMs (pairs of SMs) x the time of one 64-deep k-block.  That time is not
// proportional to the width bn: every k-block brings 16 KB of A and bn / 8 KB of B (a pair's CTA: half of them) into an SM,
// and the fill from L2 is what bounds it.  Measured on B200 under sustained load (us per k-block, K = 3072 .. 11008):
// single CTAs 0.457 / 0.40 / 0.345 at bn = 256 / 192 / 128, pairs 0.42 / 0.345 / 0.29.  Wider tiles win ties.
// Pairs: not for one row tile, nor for K below 2048, where their coarser tiles and set-up cost more than the fill saves
// (BERT-shaped layer with pairs in both projections / in the down projection / none: 55.6 / 51.7 / 52.4 us; ViT-shaped
// 252 / 248.5 / 249; Llama-shaped down projection 505-533 us with pairs under sustained load, 550 without).
struct tile_choice { int bn; bool pair; };
tile_choice pick_tile(int M, int N, int K, int batch, bool pairs_ok, bool gated)
{
    // A ragged last column tile takes the epilogue's generic loop, about 15 us that nothing hides in short problems (N = 8192,
    // 300 tokens: 34 us with 192-column tiles against 18 us with 256-column ones).  Gated tiles always have 128 columns.
    const auto ragged = [&](int bn) { return !gated && N % bn ? 15.0 / d2d_cdiv(K, BK) : 0.0; };
    const int sms = d2d_tc_sm_count();
    const int bns[4] = {256, 192, 128, 64};
    const double t1[4] = {0.457, 0.40, 0.345, 0.28}, t2[3] = {0.42, 0.345, 0.29};
    tile_choice best = {256, false};
    double best_cost = 1e300;
    for (int i = 0; i < 4; ++i) {
        const long tiles = (long)d2d_cdiv(N, bns[i]) * d2d_cdiv(M, BM) * batch;
        const double cost = (double)((tiles + sms - 1) / sms) * t1[i] + ragged(bns[i]);
        if (cost < best_cost - 1e-9) { best_cost = cost; best = {bns[i], false}; }
    }
    if (!pairs_ok || M <= BM || K < 2048) return best;
    const int pairs = sms / 2;
    for (int i = 0; i < 3; ++i) {
        const long tiles = (long)d2d_cdiv(N, bns[i]) * d2d_cdiv(M, 2 * BM) * batch;
        const double cost = (double)((tiles + pairs - 1) / pairs) * t2[i] + ragged(bns[i]);
        if (cost < best_cost - 1e-9) { best_cost = cost; best = {bns[i], true}; }
    }
    return best;
}

template <int EPI, int ACT, bool GATED>
d2d_status launch_bn(const d2d_gemm_args &g, cudaStream_t st)
{
    if constexpr (EPI == D2D_EPI_UP_MASKED && !GATED) {
        if (g.sorted.on) return launch<256, EPI, ACT, false, false, 0, SORTED_UP>(g, st);
    }
    const bool pairs_ok = !g.test_skip_load && EPI != D2D_EPI_ABS_F32;
    if (GATED) {
        if (pairs_ok && g.M > BM) return launch<128, EPI, ACT, GATED, true>(g, st);
        return launch<128, EPI, ACT, GATED>(g, st);
    }
    const tile_choice c = pick_tile(g.M, g.N, g.K, g.batch > 1 ? g.batch : 1, pairs_ok, GATED);
    if (c.pair) {
        if (c.bn == 256) return launch<GATED ? 128 : 256, EPI, ACT, GATED, EPI != D2D_EPI_ABS_F32>(g, st);
        if (c.bn == 192) return launch<GATED ? 128 : 192, EPI, ACT, GATED, EPI != D2D_EPI_ABS_F32>(g, st);
        return launch<128, EPI, ACT, GATED, EPI != D2D_EPI_ABS_F32>(g, st);
    }
    switch (c.bn) {
    case 256: return launch<GATED ? 128 : 256, EPI, ACT, GATED>(g, st);
    case 192: return launch<GATED ? 128 : 192, EPI, ACT, GATED>(g, st);
    case 128: return launch<128, EPI, ACT, GATED>(g, st);
    default: return launch<GATED ? 128 : 64, EPI, ACT, GATED>(g, st);
    }
}

template <bool GATED>
d2d_status launch_up(const d2d_gemm_args &g, cudaStream_t st)
{
    switch (g.act) {
    case D2D_ACT_RELU: return launch_bn<D2D_EPI_UP_MASKED, D2D_ACT_RELU, GATED>(g, st);
    case D2D_ACT_GELU_ERF: return launch_bn<D2D_EPI_UP_MASKED, D2D_ACT_GELU_ERF, GATED>(g, st);
    case D2D_ACT_GELU_TANH: return launch_bn<D2D_EPI_UP_MASKED, D2D_ACT_GELU_TANH, GATED>(g, st);
    case D2D_ACT_SILU: return launch_bn<D2D_EPI_UP_MASKED, D2D_ACT_SILU, GATED>(g, st);
    }
    return D2D_ERR_INVALID_ARG;
}

}  // namespace

// y = bf16(sum of the buffers + bias) after a split-K GEMM; `batch` problems back to back ([sums, batch, M, N], [batch, N] bias)
__global__ void __launch_bounds__(256)
splitk_finalize_kernel(const float *__restrict__ partial, const __nv_bfloat16 *__restrict__ bias, __nv_bfloat16 *__restrict__ out,
                       int M, int N, int batch, int sums)
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const size_t per = (size_t)M * N, total = per * batch;
    for (size_t i = ((size_t)blockIdx.x * 256 + threadIdx.x) * 4; i < total; i += (size_t)gridDim.x * 1024) {
        float4 v = __ldcg(reinterpret_cast<const float4 *>(partial + i));
        for (int s = 1; s < sums; ++s) {
            const float4 w = __ldcg(reinterpret_cast<const float4 *>(partial + (size_t)s * total + i));
            v.x += w.x; v.y += w.y; v.z += w.z; v.w += w.w;
        }
        const int c = (int)(i / per) * N + (int)(i % N);
        const float o[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) out[i + q] = __float2bfloat16_rn(o[q] + (bias ? __bfloat162float(bias[c + q]) : 0.0f));
    }
}

namespace {

typedef CUresult (*encode_tiled_fn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                    const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                    CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

encode_tiled_fn get_encode()
{
    static encode_tiled_fn fn = [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            p = nullptr;
        return (encode_tiled_fn)p;
    }();
    return fn;
}

}  // namespace

bool d2d_tc_make_map(CUtensorMap *map, const void *base, int rows, int cols, int box_rows)
{
    encode_tiled_fn enc = get_encode();
    if (!enc) return false;
    cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)cols * 2};
    cuuint32_t box[2] = {64u, (cuuint32_t)box_rows};
    cuuint32_t estr[2] = {1, 1};
    return enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(base), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool d2d_tc_encode_map(CUtensorMap *map, bool bytes, int rank, const void *base, const cuuint64_t *dims, const cuuint64_t *strides,
                       const cuuint32_t *box)
{
    encode_tiled_fn enc = get_encode();
    const cuuint32_t estr[5] = {1, 1, 1, 1, 1};
    return enc && enc(map, bytes ? CU_TENSOR_MAP_DATA_TYPE_UINT8 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, (cuuint32_t)rank, const_cast<void *>(base),
                      dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                      CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

int d2d_tc_sm_count()
{
    static int cached = 0;
    if (cached == 0) {
        int dev = 0, n = 0;
        if (cudaGetDevice(&dev) == cudaSuccess &&
            cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && n > 0)
            cached = n;
        else
            return 148;
    }
    return cached;
}

// D2D_GEMM_PDL=0 launches every GEMM fully serialised (no programmatic dependent launch)
bool d2d_tc_pdl_enabled()
{
    static const bool on = [] {
        const char *e = getenv("D2D_GEMM_PDL");
        return !(e && e[0] == '0');
    }();
    return on;
}

bool d2d_gemm_tc_available() { return get_encode() != nullptr; }

// Slices of K and tile width.  Split are only problems whose output tiles would occupy less than half of the SMs (a few hundred
// tokens at most).  With tiles of 64 columns a slice is at least two k-blocks; tiles of 128 columns need more slices for the same
// number of CTAs, hence more partial sums, and bring more weight bytes in flight (16 KB a stage instead of 8: the narrow ones reached
// 3.1 TB/s on 90 MB of weights): they are taken where a slice is 40 k-blocks or more (14 us of main loop, against about 4 for the
// sums).  Llama-shaped layer (d_ff = 11008), back to back: 74.7 -> 69.4 us at 40 tokens, 82.5 -> 80.5 at 128, and 113.5 -> 102.5 at 200,
// where narrow tiles leave nothing to split.
// A slice adds its partial sums to a float32 buffer.  Wide tiles have a buffer for every two slices: the sum of two does not depend on
// which comes first, and the buffers are added in order, so these batches (Llama-shaped layer, 9 to 256 tokens) give the same bits on
// every call.  Narrow tiles, mostly in more slices, share one buffer and do not (a buffer a slice: 23.8 instead of 22.1 us for the
// BERT-shaped layer of 128 tokens, 29.3 instead of 27.5 for the GPT-2-medium-shaped one of 200).
struct split_choice { int n, bn, per_sum; };
static split_choice pick_split(int M, int N, int K, int batch)
{
    if (N & 3) return {1, 64, 1};
    const int nkb = d2d_cdiv(K, BK), sms = d2d_tc_sm_count();
    const long rows = (long)d2d_cdiv(M, BM) * (batch > 1 ? batch : 1);
    const int wide = (int)(sms / (rows * d2d_cdiv(N, 128)));
    if (wide >= 2 && N % 128 == 0 && nkb / wide >= 40) return {wide, 128, 2};
    int splits = (int)(sms / (rows * d2d_cdiv(N, 64)));
    if (splits > nkb / 2) splits = nkb / 2;
    if (splits < 2) splits = 1;
    return {splits, 64, splits};
}

int d2d_gemm_tc_splits(int M, int N, int K, int batch) { return M > 0 ? pick_split(M, N, K, batch).n : 1; }

size_t d2d_gemm_tc_partial_floats(int M, int N, int K, int batch)
{
    if (M <= 0) return 0;
    const split_choice c = pick_split(M, N, K, batch);
    return c.n > 1 ? (size_t)d2d_cdiv(c.n, c.per_sum) * (batch > 1 ? batch : 1) * M * N : 0;
}

d2d_status d2d_gemm_tc(const d2d_gemm_args &g, cudaStream_t st)
{
    if (g.M <= 0 || g.N <= 0 || g.K <= 0) return D2D_OK;
    if (g.K % 8) return D2D_ERR_UNSUPPORTED;
    switch (g.epilogue) {
    case D2D_EPI_RELU_BF16: return launch_bn<D2D_EPI_RELU_BF16, 0, false>(g, st);
    case D2D_EPI_ABS_F32: return launch_bn<D2D_EPI_ABS_F32, 0, false>(g, st);
    case D2D_EPI_BIAS_BF16:
        if (g.sorted.on) return launch<256, D2D_EPI_BIAS_BF16, 0, false, false, 0, SORTED_DOWN>(g, st);
        if (g.k_splits > 1 && g.partial) {
            const int batch = g.batch > 1 ? g.batch : 1;
            const split_choice c = pick_split(g.M, g.N, g.K, batch);
            const int sums = d2d_cdiv(c.n, c.per_sum);
            if (c.n != g.k_splits) return D2D_ERR_INVALID_ARG;
            if (!g.partial_zero && cudaMemsetAsync(g.partial, 0, (size_t)sums * batch * g.M * g.N * sizeof(float), st) != cudaSuccess) return D2D_ERR_CUDA;
            d2d_gemm_args p = g;
            p.epilogue = D2D_EPI_PARTIAL_F32;
            p.bias = nullptr;
            p.out = g.partial;
            const d2d_status rc = c.bn == 128 ? launch<128, D2D_EPI_PARTIAL_F32, 0, false>(p, st, c.per_sum)
                                              : launch<64, D2D_EPI_PARTIAL_F32, 0, false>(p, st, c.per_sum);
            if (rc != D2D_OK) return rc;
            const int blocks = d2d_cdiv(batch * g.M * g.N, 1024);
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(blocks < 148 ? blocks : 148, 1, 1);
            cfg.blockDim = dim3(256, 1, 1);
            cfg.stream = st;
            cudaLaunchAttribute attr[1];
            attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
            attr[0].val.programmaticStreamSerializationAllowed = 1;
            cfg.attrs = attr;
            cfg.numAttrs = d2d_tc_pdl_enabled() ? 1 : 0;
            const cudaError_t err = cudaLaunchKernelEx(&cfg, splitk_finalize_kernel, (const float *)g.partial, (const __nv_bfloat16 *)g.bias,
                                                       (__nv_bfloat16 *)g.out, g.M, g.N, batch, sums);
            D2D_LAUNCHED(1);
            return err == cudaSuccess ? D2D_OK : D2D_ERR_CUDA;
        }
        return launch_bn<D2D_EPI_BIAS_BF16, 0, false>(g, st);
    case D2D_EPI_UP_MASKED: return g.b_gate ? launch_up<true>(g, st) : launch_up<false>(g, st);
    }
    return D2D_ERR_INVALID_ARG;
}
