// The whole layer of a float32 problem whose weights fit one SM's shared memory, in one launch (Sec. 3.2-3.4).
//
// At this size the time is a chain of latencies.  Every CTA brings ALL weights into its shared memory with a few bulk
// copies, requested before the dependency wait (138 KB for the 64 x 256 layer: about 2 us, once, where fetching the kept
// experts' rows when they are known costs a round trip through L2 per step of the chain: router, scores, up, down), then
// runs its tokens (one while there are SMs left) from there: a sub-warp per output with 16-byte reads, free of bank
// conflicts; the down projection with the hidden neurons split over thread groups in a fixed order.  The CTA that finishes
// last (ticket) builds the per-expert lists and writes the status word.  Exact float32 FMA throughout.
// More tokens than SMs: a CTA's threads form two teams with a token each, because a token keeps few threads busy between its
// barriers (64 x 256 layer, one team / two / four: 17.8 / 15.6 / 21.5 us at 149 tokens, 47.4 / 40.7 / 39.0 at 1000).
#include "d2d_common.cuh"
#include "lists.cuh"
#include "small_select.cuh"
#include "tc_common.cuh"

namespace {

constexpr int NT = 512, NWARP = NT / 32;
constexpr int MAX_COLS = 2;                         // output columns per thread: d <= NT * MAX_COLS
constexpr size_t kSmemLimit = 216 * 1024;

struct SmallF32Args {
    const float *x, *w_r1, *b_r1, *w_r2, *b_r2, *w1, *b1, *w_gate, *w2t, *b2;
    float *y, *R_out;               // R_out: [T, E] or NULL
    d2d_routing r;                  // mask, k, status required; lists optional as a set
    unsigned int *ticket;           // [0] exit ticket, [1] largest condition: zero at launch, left at zero
    int T, d, d_h, d_ff, E, s, W, lists, per;       // per: tokens per CTA
    float tau;
};

__device__ __forceinline__ void bulk_copy(void *dst, const void *src, uint32_t bytes, uint32_t bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(d2d_tc::smem_u32(dst)), "l"(src), "r"(bytes), "r"(bar) : "memory");
}

// Lanes that share one weight row (four elements per lane and step): a power of two, at most a warp
__device__ __forceinline__ int lanes_per_row(int len) { int l = 1; while (l < 32 && l * 4 < len) l <<= 1; return l; }

// What a team keeps of its token: x, u, hidden values, partial sums, scores, kept experts, mask words (a multiple of 16 bytes)
__host__ __device__ __forceinline__ size_t team_floats(int d, int d_h, int d_ff, int E, int W, int threads)
{
    return ((size_t)d + d_h + d_ff + threads * MAX_COLS + 2 * E + W + 3) / 4 * 4;
}

// dot(row, vec) for the sub-warp of `lpr` lanes this lane belongs to (every lane of the warp must call it)
__device__ __forceinline__ float subwarp_dot(const float *row, const float *vec, int len, int lpr, int sl)
{
    float v = 0.0f;
    for (int c = sl * 4; c < len; c += lpr * 4) {
        const float4 a = *reinterpret_cast<const float4 *>(row + c), b = *reinterpret_cast<const float4 *>(vec + c);
        v = fmaf(a.x, b.x, v); v = fmaf(a.y, b.y, v); v = fmaf(a.z, b.z, v); v = fmaf(a.w, b.w, v);
    }
    for (int o = lpr >> 1; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

template <int ACT, bool GATED, int TEAMS>
__global__ void __launch_bounds__(NT, 1)
layer_f32_small_kernel(const SmallF32Args a)
{
    constexpr int TN = NT / TEAMS, TW = TN / 32;        // threads and warps of a team
    extern __shared__ __align__(16) float smem[];
    const int d = a.d, d_h = a.d_h, E = a.E, d_ff = a.d_ff, s = a.s;
    float *w_r1 = smem, *w_r2 = w_r1 + d * d_h, *w1 = w_r2 + E * d_h, *wg = w1 + d_ff * d, *w2t = wg + (GATED ? d_ff * d : 0);
    const int cta_warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), team = cta_warp / TW;
    float *xs = w2t + d_ff * d + (size_t)team * team_floats(d, d_h, d_ff, E, a.W, TN);      // [d], and what follows: one per team
    float *us = xs + d;                                 // [d_h]
    float *hs = us + d_h;                               // [d_ff] hidden values of the kept experts
    float *red = hs + d_ff;                             // [TN * MAX_COLS] partial sums
    float *Rs = red + TN * MAX_COLS;                    // [E]
    int *kept = reinterpret_cast<int *>(Rs + E);        // [E] kept experts of this token, ascending
    uint32_t *words = reinterpret_cast<uint32_t *>(kept + E);                 // [W]
    // [T * W] all tokens' words, [T] their k (last CTA, lists only)
    uint32_t *smask = reinterpret_cast<uint32_t *>(w2t + d_ff * d + (size_t)TEAMS * team_floats(d, d_h, d_ff, E, a.W, TN));
    __shared__ uint64_t bar[2];
    __shared__ int n_kept_s[TEAMS], is_last;
    int &n_kept = n_kept_s[team];
    const int tid = (int)threadIdx.x - team * TN, lane = tid & 31, warp = cta_warp - team * TW;      // inside the team
    auto team_sync = [&]() {
        if (TEAMS == 1) __syncthreads();
        else asm volatile("bar.sync %0, %1;" ::"r"(1 + team), "n"(TN) : "memory");
    };
    if (threadIdx.x == 0) {
        d2d_tc::mbar_init(d2d_tc::smem_u32(&bar[0]), 1);
        d2d_tc::mbar_init(d2d_tc::smem_u32(&bar[1]), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        const uint32_t b0 = d2d_tc::smem_u32(&bar[0]), b1 = d2d_tc::smem_u32(&bar[1]);
        const uint32_t n1 = (uint32_t)(d * d_h) * 4u, n2 = (uint32_t)(E * d_h) * 4u, nw = (uint32_t)(d_ff * d) * 4u;
        d2d_tc::mbar_expect_tx(b0, n1 + n2);
        bulk_copy(w_r1, a.w_r1, n1, b0);
        bulk_copy(w_r2, a.w_r2, n2, b0);
        d2d_tc::mbar_expect_tx(b1, (GATED ? 3u : 2u) * nw);
        bulk_copy(w1, a.w1, nw, b1);
        if (GATED) bulk_copy(wg, a.w_gate, nw, b1);
        bulk_copy(w2t, a.w2t, nw, b1);
    }
    __syncthreads();
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    int32_t *cond = reinterpret_cast<int32_t *>(a.ticket + 1);
    const int t_begin = (int)blockIdx.x * a.per, t_end = min(a.T, t_begin + a.per);
    bool ok = true;
    for (int t = t_begin + team; t < t_end; t += TEAMS) {
        for (int c = tid; c < d; c += TN) xs[c] = a.x[(size_t)t * d + c];
        if (t == t_begin + team) ok = d2d_tc::mbar_wait_warp(d2d_tc::smem_u32(&bar[0]), 0, cond);
        team_sync();
        // ---- router: u = ReLU(W_r1 x + b_r1), R = |W_r2 u + b_r2|
        {
            const int lpr = lanes_per_row(d), rpw = 32 / lpr, sub = lane / lpr, sl = lane % lpr;
            for (int j0 = warp * rpw; j0 < d_h; j0 += TW * rpw) {
                const int j = min(j0 + sub, d_h - 1);
                const float v = subwarp_dot(w_r1 + j * d, xs, d, lpr, sl);
                if (sl == 0) us[j] = fmaxf(v + (a.b_r1 ? __ldg(a.b_r1 + j) : 0.0f), 0.0f);
            }
        }
        team_sync();
        {
            const int lpr = lanes_per_row(d_h), rpw = 32 / lpr, sub = lane / lpr, sl = lane % lpr;
            for (int e0 = warp * rpw; e0 < E; e0 += TW * rpw) {
                const int e = min(e0 + sub, E - 1);
                const float v = subwarp_dot(w_r2 + e * d_h, us, d_h, lpr, sl);
                if (sl == 0) Rs[e] = fabsf(v + (a.b_r2 ? __ldg(a.b_r2 + e) : 0.0f));
            }
        }
        team_sync();
        // ---- dynamic-k rule (Eq. 4): keep expert i iff R_i >= tau * max_j R_j, the product rounded once to float32
        if (warp == 0) {
            float m = -INFINITY;
            bool bad = !ok;
            for (int i = lane; i < E; i += 32) {
                const float v = Rs[i];
                bad |= !d2d_small::finite_f32(v);
                m = v > m ? v : m;
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
            bad = __any_sync(0xffffffffu, bad);
            const float thr = __fmul_rn(a.tau, m);
            int kt = 0;
            for (int w = 0; w < a.W; ++w) {
                const int i = w * 32 + lane;
                const uint32_t word = __ballot_sync(0xffffffffu, i < E && (bad || Rs[i] >= thr));
                if (lane == 0) { words[w] = word; a.r.mask[(size_t)t * a.W + w] = word; }
                if ((word >> lane) & 1u) kept[kt + __popc(word & ((1u << lane) - 1u))] = i;      // ascending
                kt += __popc(word);
            }
            if (lane == 0) {
                a.r.k[t] = kt;
                n_kept = kt;
                if (bad) atomicMax(cond, (int32_t)D2D_ERR_NONFINITE);
            }
        } else if (a.R_out) {
            for (int i = tid - 32; i < E; i += TN - 32) a.R_out[(size_t)t * E + i] = Rs[i];
        }
        if (t == t_begin + team) ok = d2d_tc::mbar_wait_warp(d2d_tc::smem_u32(&bar[1]), 0, cond) && ok;
        team_sync();
        // ---- kept experts, up projection + activation: all their hidden neurons, a sub-warp each
        const int n_hidden = n_kept * s;
        {
            const int lpr = lanes_per_row(d), rpw = 32 / lpr, sub = lane / lpr, sl = lane % lpr;
            for (int i0 = warp * rpw; i0 < n_hidden; i0 += TW * rpw) {
                const int idx = min(i0 + sub, n_hidden - 1);
                const int q = idx / s, n = kept[q] * s + idx - q * s;
                float up = subwarp_dot(w1 + n * d, xs, d, lpr, sl);
                const float gate = GATED ? subwarp_dot(wg + n * d, xs, d, lpr, sl) : 0.0f;
                if (sl == 0) {
                    if (a.b1) up += __ldg(a.b1 + n);
                    hs[idx] = GATED ? d2d_activate<ACT>(gate) * up : d2d_activate<ACT>(up);
                }
            }
        }
        team_sync();
        // ---- down projection: a thread owns output columns; the kept experts' neurons are split over TN / d thread groups
        const int groups = d < TN ? TN / d : 1;
        const int grp = d < TN ? tid / d : 0, col0 = d < TN ? tid % d : tid;
        float acc[MAX_COLS] = {0.0f, 0.0f};
        if (grp < groups) {
            for (int q = 0; q < n_kept; ++q) {
                const float *base = w2t + kept[q] * s * d;
#pragma unroll 4
                for (int n = grp; n < s; n += groups) {
                    const float hv = hs[q * s + n];
#pragma unroll
                    for (int i = 0; i < MAX_COLS; ++i) {
                        const int c = col0 + TN * i;
                        if (i == 0 || c < d) acc[i] = fmaf(hv, base[n * d + (c < d ? c : 0)], acc[i]);
                    }
                }
            }
        }
        if (groups > 1) {
            if (grp < groups) red[grp * d + col0] = acc[0];
            team_sync();
            if (tid < d) {
                float v = a.b2 ? __ldg(a.b2 + tid) : 0.0f;
                for (int q = 0; q < groups; ++q) v += red[q * d + tid];
                a.y[(size_t)t * d + tid] = v;
            }
        } else {
#pragma unroll
            for (int i = 0; i < MAX_COLS; ++i) {
                const int c = tid + TN * i;
                if (c < d) a.y[(size_t)t * d + c] = acc[i] + (a.b2 ? __ldg(a.b2 + c) : 0.0f);
            }
        }
    }
    // ---- the CTA that finishes last builds the lists from everybody's mask words and writes the status
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned int done;                                         // releases the whole CTA's results (the barrier before it), acquires all
        asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;" : "=r"(done) : "l"(a.ticket) : "memory");
        is_last = done == gridDim.x - 1;
        if (is_last) *a.ticket = 0u;
        if (is_last) *a.r.status = atomicExch(cond, 0);
    }
    __syncthreads();
    if (!is_last || !a.lists) return;
    if (!a.r.tok_off && a.T > 32) {
        // A warp that fetches one token's words after the other, as select_cta does, waits for L2 every time: 14.6 us for the layer at
        // 128 tokens, 12.3 this way; 61.8 and 40.7 at 1000; up to two tokens a warp it is the shorter way (10.2 and 11.2 at
        // 16).  Scratch where the first team kept its token, at least 1088 bytes.
        const d2d_list_io io = {a.r.mask, nullptr, a.r.counts, a.r.offsets, a.r.perm, a.r.n_sel, a.r.status, (long long)a.r.perm_capacity};
        uint16_t *cnt = reinterpret_cast<uint16_t *>(w2t + d_ff * d);
        for (int w = 0; w < a.W; ++w) {
            d2d_lists::lists_of_word<NWARP, true>(io, w, a.T, E, a.W, cta_warp, lane, cnt, reinterpret_cast<int *>(cnt + NT), [] { __syncthreads(); });
            __syncthreads();
        }
        return;
    }
    d2d_small::select_cta(nullptr, a.T, E, a.W, a.tau, a.r.mask, a.r.k, a.r.counts, a.r.offsets, a.r.perm, a.r.tok_off, a.r.tok_exp,
                          a.r.n_sel, a.r.status, a.r.perm_capacity, 1, smask, reinterpret_cast<int *>(smask + a.T * a.W));
}

size_t smem_bytes(const d2d_layer_desc &D, int T, bool lists, int teams)
{
    const size_t W = (size_t)(D.n_experts + 31) / 32;
    return ((size_t)D.d * D.d_h + (size_t)D.n_experts * D.d_h + (size_t)(D.gated ? 3 : 2) * D.d_ff * D.d +
            teams * team_floats(D.d, D.d_h, D.d_ff, D.n_experts, (int)W, NT / teams) + (lists ? T * (W + 1) : 0)) * 4;
}

// Teams of a CTA: two where it has several tokens and a team has threads for all output columns
constexpr int MANY = 2;
int teams_for(const d2d_layer_desc &D, int T, bool lists)
{
    return d2d_cdiv(T, d2d_tc_sm_count()) >= 2 && D.d <= NT / MANY * MAX_COLS && smem_bytes(D, T, lists, MANY) <= kSmemLimit ? MANY : 1;
}

template <int ACT, bool GATED, int TEAMS> d2d_status launch(const SmallF32Args &a, int grid, size_t smem, cudaStream_t st)
{
    auto kern = layer_f32_small_kernel<ACT, GATED, TEAMS>;
    static bool attr_set[64] = {};                          // the attribute is per device
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return D2D_ERR_CUDA;
    if (!__atomic_load_n(&attr_set[dev], __ATOMIC_ACQUIRE)) {
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemLimit) != cudaSuccess) return D2D_ERR_CUDA;
        __atomic_store_n(&attr_set[dev], true, __ATOMIC_RELEASE);
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid, 1, 1);
    cfg.blockDim = dim3(NT, 1, 1);
    cfg.dynamicSmemBytes = smem;
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

template <int ACT> d2d_status launch_gated(const SmallF32Args &a, bool gated, int teams, int grid, size_t smem, cudaStream_t st)
{
    if (teams > 1) return gated ? launch<ACT, true, MANY>(a, grid, smem, st) : launch<ACT, false, MANY>(a, grid, smem, st);
    return gated ? launch<ACT, true, 1>(a, grid, smem, st) : launch<ACT, false, 1>(a, grid, smem, st);
}

}  // namespace

// All weights of the layer in one SM's shared memory; lists by one CTA
bool d2d_layer_f32_small_supports(const d2d_layer_desc &D, int T, bool lists)
{
    if (D.dtype != D2D_F32 || T < 1 || D.d > NT * MAX_COLS || D.d % 8 || D.d_h % 8) return false;
    if (lists && T > 4096) return false;                   // (the lists are the work of one CTA)
    return smem_bytes(D, T, lists, 1) <= kSmemLimit;
}

d2d_status d2d_layer_f32_small(const d2d_layer *L, const void *x, int T, float tau, void *y, float *R_out, const d2d_routing *r,
                               bool lists, unsigned int *ticket, cudaStream_t st)
{
    const d2d_layer_desc &D = L->desc;
    SmallF32Args a = {};
    a.x = (const float *)x; a.w_r1 = (const float *)L->w_r1; a.b_r1 = (const float *)L->b_r1; a.w_r2 = (const float *)L->w_r2;
    a.b_r2 = (const float *)L->b_r2; a.w1 = (const float *)L->w1; a.b1 = (const float *)L->b1; a.w_gate = (const float *)L->w_gate;
    a.w2t = (const float *)L->w2t; a.b2 = (const float *)L->b2;
    a.y = (float *)y; a.R_out = R_out; a.r = *r; a.ticket = ticket;
    a.T = T; a.d = D.d; a.d_h = D.d_h; a.d_ff = D.d_ff; a.E = D.n_experts; a.s = D.expert_size; a.W = (D.n_experts + 31) / 32;
    a.lists = lists ? 1 : 0; a.tau = tau;
    a.per = d2d_cdiv(T, d2d_tc_sm_count());
    const int grid = d2d_cdiv(T, a.per);
    const int teams = teams_for(D, T, lists);
    const size_t smem = smem_bytes(D, T, lists, teams);
    switch (D.act) {
    case D2D_ACT_RELU: return launch_gated<D2D_ACT_RELU>(a, D.gated != 0, teams, grid, smem, st);
    case D2D_ACT_GELU_ERF: return launch_gated<D2D_ACT_GELU_ERF>(a, D.gated != 0, teams, grid, smem, st);
    case D2D_ACT_GELU_TANH: return launch_gated<D2D_ACT_GELU_TANH>(a, D.gated != 0, teams, grid, smem, st);
    case D2D_ACT_SILU: return launch_gated<D2D_ACT_SILU>(a, D.gated != 0, teams, grid, smem, st);
    }
    return D2D_ERR_INVALID_ARG;
}
