// Router, dynamic-k selection and per-expert lists of a decode batch (Sec. 3.3, Eq. 4, Listing 1) in one launch: one
// thread-block cluster per layer, one CTA per 16 hidden units.
//
// What bounds it is a chain of dependent latencies, not bytes: read x -> u -> scores -> row maximum -> lists.  The CTAs
// of a cluster hand u (and, for large W_r2, the scores) on through distributed shared memory with asynchronous stores
// that signal the receiver's barrier, where a grid would need tickets and round trips through L2 at every step; the
// selection and the lists are then the work of CTA 0 alone, whose steps are 50 ns apart (a cluster barrier costs 0.7 us:
// an exchange of row maxima and counts between all CTAs measured 1.4 us more).  Everything that does not depend on the
// previous kernel of the stream (both weight matrices and biases) is requested before the dependency wait: the first
// layer's rows go straight into registers as matrix-instruction operands (a warp takes every 16th block of 32 k values,
// the partial sums of the 16 warps meet in shared memory), the second layer's into shared memory.
#include "decode.cuh"
#include "tc_common.cuh"

namespace {

using namespace d2d_decode;

constexpr int NT = 512, NWARP = NT / 32;
constexpr int MAX_W = 16;              // mask words per token: E <= 512
constexpr unsigned FULL = 0xffffffffu;

__device__ __forceinline__ uint32_t cluster_rank_addr(uint32_t addr, uint32_t rank)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
// 4 bytes into the shared memory of another CTA of the cluster; counted by that CTA's barrier
__device__ __forceinline__ void st_async_u32(uint32_t addr, uint32_t v, uint32_t bar)
{
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(addr), "r"(v), "r"(bar) : "memory");
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

__device__ __forceinline__ bool finite_f32(float v) { return (__float_as_uint(v) & 0x7f800000u) != 0x7f800000u; }

__device__ __forceinline__ int warp_iscan(int v, int lane)
{
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int n = __shfl_up_sync(FULL, v, o);
        if (lane >= o) v += n;
    }
    return v;
}

// rows of 16-byte pieces that eight lanes read as 64 bytes of two adjacent rows: a pitch of 64 (mod 128) bytes is free
// of bank conflicts
__host__ __device__ constexpr int frag_pitch(int bytes) { return (bytes + 127) / 128 * 128 + 64; }

// KB: 32-wide k blocks per warp held in registers at a time; NT8: tokens / 8.  planes: 1 = u rounded to bf16 (batches
// that continue on bf16 hidden activations), 3 = u kept to float32 precision (see split3).
// ONE: CTA 0 computes all scores, 16 experts per warp, their rows of W_r2 in registers (at most 256 experts, d_h <= 128; from
// shared memory the reads alone, 64 KB and the token rows per warp, took 1 us); otherwise mask word w belongs to CTA
// w % CS, which keeps its rows in shared memory.
template <int KB, int NT8, bool ONE>
__global__ void __launch_bounds__(NT, 1)
decode_router_kernel(const __nv_bfloat16 *__restrict__ x, int T, int d, int d_h, int E, float tau, int do_mask, int planes,
                     int zero_words, const __grid_constant__ d2d_decode_router_args args)
{
    constexpr int T8 = 8 * NT8;
    const d2d_decode_router_layer &P = args.l[blockIdx.y];
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ uint64_t bar_u, bar_s;            // u has arrived; the scores have arrived (CTA 0)
    __shared__ uint32_t smask[MAX_W][T8];
    __shared__ int stot[MAX_W];                  // selected pairs per mask word
    __shared__ uint32_t skept[MAX_W];            // experts some token keeps
    __shared__ int sbad;
    const int tid = threadIdx.x, lane = tid & 31, g = lane >> 2, c = lane & 3;
    const int warp = __shfl_sync(FULL, tid >> 5, 0);                           // warp-uniform for the compiler: see mma16816
    const uint32_t rank = blockIdx.x, CS = gridDim.x;
    const int n_sc = ONE ? 1 : (int)CS;                                        // CTAs that compute scores
    const int W = (E + 31) / 32, WPC = (W + n_sc - 1) / n_sc, EP = W * 32 + 1;
    const int n_recv = ONE ? 1 : ((int)CS < W ? (int)CS : W);            // CTAs that need u
    const int pitch = frag_pitch(d_h * 2);
    float *red = reinterpret_cast<float *>(smem);                              // [16 warps][16 units][T8]
    unsigned char *us = smem + (size_t)NWARP * 16 * T8 * 4;                    // [planes][T8] rows of d_h bf16
    unsigned char *w2s = us + (size_t)planes * T8 * pitch;                     // [WPC * 32] rows of d_h bf16
    float *b2s = reinterpret_cast<float *>(w2s + (ONE ? 0 : (size_t)WPC * 32 * pitch));    // [WPC * 32]
    float *Rs = b2s + WPC * 32;                                                // [T8][EP] scores (CTA 0)

    // ---- parameters: requested before anything else
    const int unit0 = (int)rank * 16;
    uint4 wa[KB][2];
    auto load_w1 = [&](int b0) {
#pragma unroll
        for (int b = 0; b < KB; ++b) {
            const int k = ((b0 + b) * NWARP + warp) * 32 + c * 8;
#pragma unroll
            for (int h = 0; h < 2; ++h)
                wa[b][h] = k < d ? __ldg(reinterpret_cast<const uint4 *>(P.w_r1 + (size_t)(unit0 + g + 8 * h) * d + k)) : make_uint4(0, 0, 0, 0);
        }
    };
    load_w1(0);
    uint4 wr[ONE ? 4 : 1][2];                                                  // rows warp * 16 + g, + 8 of W_r2
    if ((int)rank < n_recv) {
        if (ONE) {
#pragma unroll
            for (int kb = 0; kb < 4; ++kb)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int e = warp * 16 + g + 8 * h, k = kb * 32 + c * 8;
                    wr[ONE ? kb : 0][h] = e < E && k < d_h ? __ldg(reinterpret_cast<const uint4 *>(P.w_r2 + (size_t)e * d_h + k)) : make_uint4(0, 0, 0, 0);
                }
        } else {
            const int cpr = d_h / 8;                                           // 16-byte pieces per row
            for (int i = tid; i < WPC * 32 * cpr; i += NT) {
                const int r = i / cpr, p = i - r * cpr;
                const int e = ((int)rank + (r >> 5) * n_sc) * 32 + (r & 31);
                if (e < E) cp_async16(smem_addr(w2s + (size_t)r * pitch + p * 16), P.w_r2 + (size_t)e * d_h + p * 8);
            }
        }
        for (int i = tid; i < WPC * 32; i += NT) {
            const int e = ((int)rank + (i >> 5) * n_sc) * 32 + (i & 31);
            b2s[i] = P.b_r2 && e < E ? __bfloat162float(P.b_r2[e]) : 0.0f;
        }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    const int out_unit = tid / T8 * 2, out_tok = tid % T8;                     // this thread's two hidden values (tid < 8 * T8)
    float b1v[2] = {0.0f, 0.0f};
    if (P.b_r1 && tid < 8 * T8) {
        b1v[0] = __bfloat162float(P.b_r1[unit0 + out_unit]);
        b1v[1] = __bfloat162float(P.b_r1[unit0 + out_unit + 1]);
    }
    if (tid == 0) {
        sbad = 0;
        d2d_tc::mbar_init(smem_addr(&bar_u), 1);
        d2d_tc::mbar_init(smem_addr(&bar_s), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        if ((int)rank < n_recv) d2d_tc::mbar_expect_tx(smem_addr(&bar_u), CS * 8u * (uint32_t)T * 4u * (uint32_t)planes);
        if (rank == 0 && !ONE && do_mask) d2d_tc::mbar_expect_tx(smem_addr(&bar_s), (uint32_t)(T * E) * 4u);
    }
    cluster_arrive();                                                          // barriers are set up: see the wait below

    pdl_wait();
    pdl_trigger();
    for (int i = (int)rank * NT + tid; i < zero_words / 4; i += (int)CS * NT) reinterpret_cast<float4 *>(P.zero)[i] = make_float4(0.f, 0.f, 0.f, 0.f);

    // ---- hidden layer: u = relu(W_r1 x + b_r1)
    float acc[NT8][4];
#pragma unroll
    for (int n = 0; n < NT8; ++n) acc[n][0] = acc[n][1] = acc[n][2] = acc[n][3] = 0.0f;
    const int nkb = (d + NWARP * 32 - 1) / (NWARP * 32);
    for (int b0 = 0; b0 < nkb; b0 += KB) {
        if (b0 > 0) load_w1(b0);
        uint4 xb[KB][NT8];
#pragma unroll
        for (int b = 0; b < KB; ++b) {
            const int k = ((b0 + b) * NWARP + warp) * 32 + c * 8;
#pragma unroll
            for (int n = 0; n < NT8; ++n)
                xb[b][n] = k < d && n * 8 + g < T ? *reinterpret_cast<const uint4 *>(x + (size_t)(n * 8 + g) * d + k) : make_uint4(0, 0, 0, 0);
        }
#pragma unroll
        for (int b = 0; b < KB; ++b)
#pragma unroll
            for (int n = 0; n < NT8; ++n) {
                mma16816(acc[n], wa[b][0].x, wa[b][1].x, wa[b][0].y, wa[b][1].y, xb[b][n].x, xb[b][n].y);
                mma16816(acc[n], wa[b][0].z, wa[b][1].z, wa[b][0].w, wa[b][1].w, xb[b][n].z, xb[b][n].w);
            }
    }
#pragma unroll
    for (int n = 0; n < NT8; ++n) {
        float *r = red + (size_t)(warp * 16 + g) * T8 + n * 8 + 2 * c;
        *reinterpret_cast<float2 *>(r) = make_float2(acc[n][0], acc[n][1]);
        *reinterpret_cast<float2 *>(r + 8 * T8) = make_float2(acc[n][2], acc[n][3]);
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    cluster_wait();                                                            // remote shared memory may be written from here on
    if (tid < 8 * T8 && out_tok < T) {
        float v0 = 0.0f, v1 = 0.0f;
        const float *r = red + out_unit * T8 + out_tok;
#pragma unroll
        for (int w = 0; w < NWARP; ++w) { v0 += r[w * 16 * T8]; v1 += r[w * 16 * T8 + T8]; }
        __nv_bfloat16 t0[3], t1[3];
        split3(fmaxf(v0 + b1v[0], 0.0f), t0);
        split3(fmaxf(v1 + b1v[1], 0.0f), t1);
        const uint32_t bar = smem_addr(&bar_u);
#pragma unroll
        for (int p = 0; p < 3; ++p) {
            if (p == planes) break;
            const uint32_t at = smem_addr(us + (size_t)(p * T8 + out_tok) * pitch + (unit0 + out_unit) * 2);
            const uint32_t bits = (uint32_t)__bfloat16_as_ushort(t0[p]) | (uint32_t)__bfloat16_as_ushort(t1[p]) << 16;
            for (int q = 0; q < n_recv; ++q) st_async_u32(cluster_rank_addr(at, q), bits, cluster_rank_addr(bar, q));
        }
    }
    if ((int)rank >= n_recv) return;                                           // nobody writes to this CTA
    bool ok = mbar_wait_cluster(smem_addr(&bar_u), 0, P.status);

    // ---- scores: R = |W_r2 u + b_r2|; a warp takes 16 experts x 8 tokens
    const uint32_t rs0 = cluster_rank_addr(smem_addr(Rs), 0), bar0 = cluster_rank_addr(smem_addr(&bar_s), 0);
    auto put = [&](int e, int row, int t, float v) {
        v = fabsf(v + b2s[row]);
        if (e < E && t < T) {
            if (P.R) P.R[(size_t)t * E + e] = v;
            if (ONE) Rs[t * EP + e] = v;
            else if (do_mask) st_async_u32(rs0 + (uint32_t)(t * EP + e) * 4u, __float_as_uint(v), bar0);
        }
    };
    // rows of u of tokens beyond the batch are not read: fewer shared-memory wavefronts
    auto load_u = [&](int p, int t, int k) {
        return t < T && k < d_h ? *reinterpret_cast<const uint4 *>(us + (size_t)(p * T8 + t) * pitch + k * 2) : make_uint4(0, 0, 0, 0);
    };
    for (int task = warp; task < WPC * 2; task += NWARP) {
        const int w = (int)rank + (task >> 1) * n_sc;
        if (w >= W) continue;
        float sc[NT8][2][4];
#pragma unroll
        for (int n = 0; n < NT8; ++n)
#pragma unroll
            for (int i = 0; i < 2; ++i) sc[n][i][0] = sc[n][i][1] = sc[n][i][2] = sc[n][i][3] = 0.0f;
        const unsigned char *ar = w2s + (size_t)(task * 16 + g) * pitch;
        auto step = [&](int kb, const uint4 &a0, const uint4 &a1) {
            const int k = kb * 32 + c * 8;
#pragma unroll
            for (int n = 0; n < NT8; ++n) {
                const uint4 b = load_u(0, n * 8 + g, k);
                mma16816(sc[n][0], a0.x, a1.x, a0.y, a1.y, b.x, b.y);
                mma16816(sc[n][1], a0.z, a1.z, a0.w, a1.w, b.z, b.w);
            }
            if (NT8 == 1 && planes == 3) {
#pragma unroll
                for (int p = 1; p < 3; ++p) {
                    const uint4 b = load_u(p, g, k);
                    mma16816(sc[0][0], a0.x, a1.x, a0.y, a1.y, b.x, b.y);
                    mma16816(sc[0][1], a0.z, a1.z, a0.w, a1.w, b.z, b.w);
                }
            }
        };
        if (ONE) {
#pragma unroll
            for (int kb = 0; kb < 4; ++kb)
                if (kb * 32 < d_h) step(kb, wr[ONE ? kb : 0][0], wr[ONE ? kb : 0][1]);
        } else {
#pragma unroll 2
            for (int kb = 0; kb * 32 < d_h; ++kb) {
                const int k = kb * 32 + c * 8;
                uint4 a0 = make_uint4(0, 0, 0, 0), a1 = a0;
                if (k < d_h) {
                    a0 = *reinterpret_cast<const uint4 *>(ar + k * 2);
                    a1 = *reinterpret_cast<const uint4 *>(ar + 8 * pitch + k * 2);
                }
                step(kb, a0, a1);
            }
        }
#pragma unroll
        for (int n = 0; n < NT8; ++n)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int row = task * 16 + g + 8 * h, e = w * 32 + (row & 31), t = n * 8 + 2 * c;
                put(e, row, t, sc[n][0][2 * h] + sc[n][1][2 * h]);
                put(e, row, t + 1, sc[n][0][2 * h + 1] + sc[n][1][2 * h + 1]);
            }
    }
    if (!do_mask || rank != 0) return;                                         // nobody writes to this CTA any more
    if (!ONE) ok = ok && mbar_wait_cluster(smem_addr(&bar_s), 0, P.status);
    __syncthreads();

    // ---- CTA 0: the rule (Eq. 4), a warp per token
    for (int t = warp; t < T; t += NWARP) {
        const float *row = Rs + t * EP;
        float m = -INFINITY;
        bool bad = !ok;
        for (int e = lane; e < E; e += 32) {
            const float v = row[e];
            bad |= !finite_f32(v);
            m = v > m ? v : m;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(FULL, m, o));
        bad = __any_sync(FULL, bad);
        const float thr = __fmul_rn(tau, m);                                   // the one rounding the rule is defined with
        int kt = 0;
        for (int w = 0; w < W; ++w) {
            const int e = w * 32 + lane;
            const uint32_t word = __ballot_sync(FULL, e < E && (bad || row[e] >= thr));
            if (lane == 0) { P.mask[(size_t)t * W + w] = word; smask[w][t] = word; }
            kt += __popc(word);
        }
        if (lane == 0) {
            P.k[t] = kt;
            if (bad) sbad = 1;
        }
    }
    __syncthreads();

    // ---- lists: a warp per mask word, lane = expert; the tokens that keep it are one 32-bit word (T <= 32)
    uint32_t bm = 0u, kept = 0u;
    int incl = 0;
    if (warp < W) {
        for (int t = 0; t < T; ++t) bm |= ((smask[warp][t] >> lane) & 1u) << t;
        kept = __ballot_sync(FULL, bm != 0u);
        incl = warp_iscan(__popc(bm), lane);
        if (lane == 31) { stot[warp] = incl; skept[warp] = kept; }
    }
    __syncthreads();
    const bool lists = P.counts != nullptr;
    if (warp < W) {
        int base = 0;
        for (int w = 0; w < warp; ++w) base += stot[w];
        const int e = warp * 32 + lane;
        if (P.units) {
            // the kept experts' 16-neuron units in ascending order, from unit u0 on (a multiple of the units per expert): what
            // the expert kernel shares out once the selection is known
            const int e0 = P.u0 / P.upe;
            int at = 0, total = 0;
            for (int w = 0; w < W; ++w) {
                const int lo = e0 - w * 32;
                const uint32_t kw = lo >= 32 ? 0u : lo > 0 ? skept[w] & ~((1u << lo) - 1u) : skept[w];
                total += __popc(kw);
                at += w < warp ? __popc(kw) : w == warp ? __popc(kw & ((1u << lane) - 1u)) : 0;
            }
            if (bm && e >= e0)
                for (int i = 0; i < P.upe; ++i) P.units[1 + at * P.upe + i] = e * P.upe + i;
            if (warp == 0 && lane == 0) P.units[0] = total * P.upe;
        }
        if (lists && e < E) {
            long long at = base + incl - __popc(bm);
            P.counts[e] = __popc(bm);
            P.offsets[e] = (int)at;
            for (uint32_t m = bm; m; m &= m - 1, ++at)
                if (at < P.capacity) P.perm[at] = __ffs(m) - 1;
        }
    }
    if (warp == NWARP - 1) {
        int n = 0;
        for (int w = 0; w < W; ++w) n += stot[w];
        if (lane == 0) {
            if (lists) { P.offsets[E] = n; *P.n_sel = n; }
            *P.status = !ok ? (int32_t)D2D_ERR_TIMEOUT : lists && (long long)n > P.capacity ? (int32_t)D2D_ERR_CAPACITY : sbad ? (int32_t)D2D_ERR_NONFINITE : 0;
        }
        if (P.tok_off) {                                                       // lane = token
            int kt = 0;
            if (lane < T)
                for (int w = 0; w < W; ++w) kt += __popc(smask[w][lane]);
            const int inc = warp_iscan(kt, lane);
            if (lane < T) {
                P.tok_off[lane + 1] = inc;
                long long at = inc - kt;
                for (int w = 0; w < W; ++w)
                    for (uint32_t m = smask[w][lane]; m; m &= m - 1, ++at)
                        if (at < P.capacity) P.tok_exp[at] = w * 32 + __ffs(m) - 1;
            }
            if (lane == 0) P.tok_off[0] = 0;
        }
    }
}

// CTA 0 computes all scores (see ONE)
bool one_scorer(const d2d_layer_desc &D) { return D.n_experts <= 256 && D.d_h <= 128 && D.d <= 2048; }

size_t router_smem(const d2d_layer_desc &D, int nt8, int planes)
{
    const bool one = one_scorer(D);
    const int w = (D.n_experts + 31) / 32, n_sc = one ? 1 : D.d_h / 16, wpc = (w + n_sc - 1) / n_sc, t8 = 8 * nt8, pitch = frag_pitch(D.d_h * 2);
    return (size_t)NWARP * 16 * t8 * 4 + (size_t)planes * t8 * pitch + (one ? 0 : (size_t)wpc * 32 * pitch) + (size_t)wpc * 32 * 4 +
           (size_t)t8 * (w * 32 + 1) * 4;
}
constexpr size_t kSmemLimit = 200 * 1024;

int token_blocks(int T) { return T <= 8 ? 1 : T <= 16 ? 2 : 4; }
int planes_for(const d2d_layer_desc &D, int T) { return T <= d2d_decode_max_tokens(D) ? 3 : 1; }

template <int KB, int NT8, bool ONE>
d2d_status launch(const d2d_layer_desc &D, int n_layers, const d2d_decode_router_args &a, const void *x, int T, float tau, int do_mask,
                  int zero_words, cudaStream_t st)
{
    auto kern = decode_router_kernel<KB, NT8, ONE>;
    static bool attr_set[64] = {};                          // the attributes are per device
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return D2D_ERR_CUDA;
    if (!__atomic_load_n(&attr_set[dev], __ATOMIC_ACQUIRE)) {
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemLimit) != cudaSuccess ||
            cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
            return D2D_ERR_CUDA;
        __atomic_store_n(&attr_set[dev], true, __ATOMIC_RELEASE);
    }
    const int planes = planes_for(D, T);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(D.d_h / 16, n_layers, 1);
    cfg.blockDim = dim3(NT, 1, 1);
    cfg.dynamicSmemBytes = router_smem(D, NT8, planes);
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = D.d_h / 16; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = d2d_tc_pdl_enabled() ? 2 : 1;
    const cudaError_t err = cudaLaunchKernelEx(&cfg, kern, (const __nv_bfloat16 *)x, T, D.d, D.d_h, D.n_experts, tau, do_mask, planes, zero_words, a);
    D2D_LAUNCHED(1);
    return err == cudaSuccess ? D2D_OK : D2D_ERR_CUDA;
}

}  // namespace

// d_h is 16 hidden units per CTA of the cluster (a power of two of them, at most 16), a warp per mask word
bool d2d_decode_router_supports(const d2d_layer_desc &D, int T)
{
    const int cs = D.d_h / 16, w = (D.n_experts + 31) / 32;
    if (D.dtype != D2D_BF16 || T < 1 || T > 32 || D.d_h % 16 || cs < 1 || cs > 16 || (cs & (cs - 1)) || D.d % 8) return false;
    return w <= MAX_W && router_smem(D, token_blocks(T), planes_for(D, T)) <= kSmemLimit;
}

d2d_status d2d_decode_router(const d2d_layer_desc &D, int n_layers, const d2d_decode_router_args &a, const void *x, int T, float tau,
                             int do_mask, int zero_words, cudaStream_t st)
{
    if (n_layers < 1 || n_layers > D2D_MAX_GROUP || !d2d_decode_router_supports(D, T)) return D2D_ERR_UNSUPPORTED;
    const int nb = token_blocks(T);
    // blocks of 32 k values per warp kept in registers: all of a row up to d = 4096 for eight tokens
    if (one_scorer(D)) {
        if (nb == 1) return launch<4, 1, true>(D, n_layers, a, x, T, tau, do_mask, zero_words, st);
        if (nb == 2) return launch<2, 2, true>(D, n_layers, a, x, T, tau, do_mask, zero_words, st);
        return launch<2, 4, true>(D, n_layers, a, x, T, tau, do_mask, zero_words, st);
    }
    if (nb == 1) return launch<8, 1, false>(D, n_layers, a, x, T, tau, do_mask, zero_words, st);
    if (nb == 2) return launch<2, 2, false>(D, n_layers, a, x, T, tau, do_mask, zero_words, st);
    return launch<2, 4, false>(D, n_layers, a, x, T, tau, do_mask, zero_words, st);
}
