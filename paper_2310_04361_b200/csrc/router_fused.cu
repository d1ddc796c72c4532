// Fused router + dynamic-k mask for bf16 layers (Sec. 3.3 and Eq. 4): one kernel computes
//   u = relu(x W_r1^T + b_r1)            tcgen05 GEMM, 128 tokens x d_h, accumulator in TMEM
//   R = | u W_r2^T + b_r2 |              second tcgen05 GEMM whose A operand is u, written by the first
//                                        epilogue straight into shared memory in the swizzled K-major layout
//   m = max_i R[t,i], thr = tau * m (one fp32 RN multiply), mask words, k[t]     per-row epilogue on TMEM
// so the hidden activations never touch HBM, R is written once (the caller may want it) and the
// mask kernel's extra pass over R disappears.  One CTA per 128 tokens; 18 warps: TMA producer,
// MMA issuer, 16 epilogue warps (four per TMEM lane quadrant, each a quarter of the columns).
// All mbarrier waits are bounded (status D2D_ERR_TIMEOUT); every load is a plain per-CTA load.
#include <cuda.h>

#include "d2d_common.cuh"
#include "gemm_tc.cuh"
#include "tc_common.cuh"

namespace {

using d2d_tc::smem_u32; using d2d_tc::mbar_init; using d2d_tc::mbar_expect_tx; using d2d_tc::mbar_arrive;
using d2d_tc::tma_load_2d; using d2d_tc::smem_desc_sw128; using d2d_tc::instr_desc_bf16; using d2d_tc::umma_bf16;
using d2d_tc::umma_commit; using d2d_tc::tmem_ld16_issue; using d2d_tc::tmem_ld_wait;

constexpr int BM = 128, BK = 64, UMMA_K = 16;
// 5 x 32 KB of operands in flight: the first GEMM's main loop is bound by load latency; 3 where two CTAs share an SM
__host__ __device__ constexpr int stages_for(bool two) { return two ? 3 : 5; }
constexpr int NTHREADS = 64 + 512;       // TMA warp, MMA warp, 16 epilogue warps

// every barrier wait of this kernel: 4096 back-to-back polls, then one poll every 128 ns
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, int32_t *status)
{
    return d2d_tc::mbar_wait<4096, 128>(bar, parity, status);
}
// 16 accumulator columns of this thread's TMEM lane, complete on return
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16])
{
    tmem_ld16_issue(taddr, r);
    tmem_ld_wait();
}

struct RouterLayerIO {
    float *R;              // [T, E] scores or NULL
    uint32_t *mask;        // [T, ceil(E/32)]
    int32_t *k;            // [T]
    int32_t *status;
};
struct RouterGroupIO {
    RouterLayerIO l[D2D_MAX_GROUP];
    uint32_t *mask_cat;    // merged mask [T, cat_words] or NULL
    int cat_words;
    int32_t *ksum[D2D_MAX_GROUP];      // all or none NULL, per layer: [0..1] running sum of k and exit count (64 bits), [2] largest condition
                           // (all zero at launch and left at zero), [4] receives the total = number of selected (token,
                           // expert) pairs; the last CTA then writes *status
};

// Number of selected pairs of the whole batch, for the density-adaptive dispatch of the expert step, and the status word: one
// 64-bit addition per CTA carries its sum (36 bits), its exit (14 bits) and whether it saw a condition (14 bits); whoever
// completes the count publishes and resets.  Called by four warps (one per TMEM lane quadrant) with their sums of k.
__device__ __forceinline__ void publish_batch(int32_t *ksum, int32_t *status_out, int quad, int lane, int k_warp, bool cond_warp,
                                              int *warp_k, int *warp_bad)
{
    if (lane == 0) { warp_k[quad] = k_warp; warp_bad[quad] = cond_warp; }
    asm volatile("bar.sync 2, 128;" ::: "memory");
    if (quad != 0 || lane != 0) return;
    const int cond = warp_bad[0] | warp_bad[1] | warp_bad[2] | warp_bad[3];
    if (cond) __threadfence();                       // its entry in the condition word comes first
    const unsigned long long add = (unsigned long long)(warp_k[0] + warp_k[1] + warp_k[2] + warp_k[3]) + (1ull << 36) +
                                   (cond ? 1ull << 50 : 0ull);
    unsigned long long *acc64 = reinterpret_cast<unsigned long long *>(ksum);
    const unsigned long long tot = atomicAdd(acc64, add) + add;
    if (((tot >> 36) & 0x3fffu) != (unsigned long long)gridDim.x) return;
    *acc64 = 0ull;
    ksum[4] = (int32_t)(tot & 0xfffffffffull);
    int32_t st = 0;
    if (tot >> 50) {
        __threadfence();
        st = atomicExch(ksum + 2, 0);
    }
    *status_out = st;
}

// 16 consecutive scores of one row, from column c0
__device__ __forceinline__ void store_scores16(float *__restrict__ R, int row, int E, int c0, const float *v)
{
    float *o = R + (size_t)row * E + c0;
    if (c0 + 16 <= E && (E & 7) == 0 && (reinterpret_cast<uintptr_t>(R) & 31) == 0) {
        // 32-byte stores: a whole sector per lane and instruction
#pragma unroll
        for (int j = 0; j < 16; j += 8)
            asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(o + j), "f"(v[j]), "f"(v[j + 1]),
                         "f"(v[j + 2]), "f"(v[j + 3]), "f"(v[j + 4]), "f"(v[j + 5]), "f"(v[j + 6]), "f"(v[j + 7]) : "memory");
    } else if (c0 + 16 <= E && (E & 3) == 0) {
#pragma unroll
        for (int j = 0; j < 16; j += 4) *reinterpret_cast<float4 *>(o + j) = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
    } else {
#pragma unroll
        for (int j = 0; j < 16; ++j)
            if (c0 + j < E) o[j] = v[j];
    }
}

// Shared memory (dynamic, 1024-byte aligned):
//   [ STAGES x (x tile 128x64 | W_r1 tile DH x 64) ]        first GEMM operand ring
//   [ u: DH/64 k-blocks x (128 rows x 128 B) ]              A operand of the second GEMM (written by epilogue 1)
//   W_r2 (DH/64 k-blocks x 256 rows x 128 B, the B operand of the second GEMM) reuses the first stages of the ring:
//   it is loaded as soon as the last k-blocks that used those stages have been consumed, under epilogue 1.
// TMEM: columns [0, DH) accumulator of u, columns [256, 256 + E_pad) accumulator of R (E <= 256).
// Several routers that read the same tokens (the Q, K and V projections of one attention layer) run as ONE grid:
// blockIdx.y picks the router.  Their weights are stacked (W_r1 [n*DH, d], b_r1 [n*DH], W_r2 [n*E, DH], b_r2 [n*E]);
// every router writes its own outputs and, when mask_cat is given, its mask words once more into a merged mask
// [T, cat_words] at word offset l * ceil(E/32) (the selection mask of the merged up projection).
// TWO: two CTAs per SM, for batches of more row tiles than SMs (see launch_for): three stages, u in the ring's last one, the scores in
// the columns of u's accumulator (both are used up by then), scores read from TMEM twice instead of kept in registers.
template <int DH, bool TWO>
__global__ void __launch_bounds__(NTHREADS, TWO ? 2 : 1)
router_fused_kernel(const __grid_constant__ CUtensorMap tm_x, const __grid_constant__ CUtensorMap tm_w1,
                    const __grid_constant__ CUtensorMap tm_w2, const __nv_bfloat16 *__restrict__ b_r1_all,
                    const __nv_bfloat16 *__restrict__ b_r2_all, int T, int d, int E, int EN /* E rounded up to 16 */,
                    float tau, int do_mask, const __grid_constant__ RouterGroupIO io)
{
    const int layer = blockIdx.y;
    const __nv_bfloat16 *b_r1 = b_r1_all ? b_r1_all + layer * DH : nullptr;
    const __nv_bfloat16 *b_r2 = b_r2_all ? b_r2_all + layer * E : nullptr;
    float *__restrict__ R = io.l[layer].R;
    uint32_t *__restrict__ mask = io.l[layer].mask;
    int32_t *__restrict__ k = io.l[layer].k;
    // conditions are collected in a word of the layer and published once (no memset in front of the kernel)
    int32_t *const ksum = io.ksum[layer];
    int32_t *__restrict__ status = ksum ? ksum + 2 : io.l[layer].status;
    constexpr int STAGES = stages_for(TWO);
    constexpr int KB2 = DH / BK;                          // k-blocks of the second GEMM
    constexpr int A_BYTES = BM * BK * 2, B1_BYTES = DH * BK * 2;
    constexpr int STAGE_BYTES = A_BYTES + B1_BYTES;
    constexpr int U_BYTES = KB2 * BM * 128;
    constexpr int W2_KB_BYTES = 256 * 128;                // one k-block of W_r2 rows (box of 256 rows, zero filled past E)

    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t *u_s = smem + (size_t)(TWO ? STAGES - 1 : STAGES) * STAGE_BYTES;
    uint8_t *w2_s = smem;                                  // aliases the first stages (see above)
    static_assert((size_t)KB2 * W2_KB_BYTES <= (size_t)(TWO ? STAGES - 1 : STAGES) * STAGE_BYTES, "W_r2 must fit in the operand ring");
    static_assert(!TWO || U_BYTES <= STAGE_BYTES, "u must fit in a stage");
    constexpr uint32_t TMEM_COLS = TWO ? 256 : 512;
    constexpr int W2_STAGES = (KB2 * W2_KB_BYTES + STAGE_BYTES - 1) / STAGE_BYTES;      // stages W_r2 overwrites
    __shared__ uint64_t bar_full[STAGES], bar_empty[STAGES], bar_w2, bar_acc1, bar_u_ready, bar_acc2;
    __shared__ uint32_t tmem_base_holder;
    __shared__ __align__(16) float b1_s[DH], b2_s[256];    // biases as float32
    __shared__ uint32_t pmax_s[4 * BM];                    // per column-part row maxima (bit patterns of non-negative floats)
    __shared__ int pk_s[4 * BM];
    __shared__ int warp_k[4], warp_bad[4];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int m0 = blockIdx.x * BM;
    const int nkb = (d + BK - 1) / BK;

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(smem_u32(&bar_full[s]), 1);
            mbar_init(smem_u32(&bar_empty[s]), 1);
        }
        mbar_init(smem_u32(&bar_w2), 1);
        mbar_init(smem_u32(&bar_acc1), 1);
        mbar_init(smem_u32(&bar_u_ready), 16);            // one arrival per epilogue warp
        mbar_init(smem_u32(&bar_acc2), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_holder)),
                     "r"(TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_base = tmem_base_holder;
    const uint32_t tmem_r = TWO ? tmem_base : tmem_base + 256;
    // The set-up above may overlap the tail of the previous kernel of the stream, and so may the weights' part of the first stages.
    const int early = nkb < STAGES ? nkb : STAGES;
    if (warp == 0 && lane == 0)
        for (int kb = 0; kb < early; ++kb) {
            mbar_expect_tx(smem_u32(&bar_full[kb]), (uint32_t)STAGE_BYTES);
            tma_load_2d(smem_u32(smem + (size_t)kb * STAGE_BYTES) + A_BYTES, &tm_w1, kb * BK, layer * DH, smem_u32(&bar_full[kb]));
        }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    // the expert up projection that follows on the stream may start its operand loads and MMAs on the SMs this
    // grid leaves idle (T / 128 CTAs); its epilogue waits for this kernel to complete before it reads the mask
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    if (warp == 0) {
        // ------------------------------------------------------------------ TMA producer
        if (lane == 0) {
            bool ok = true;
            for (int kb = 0; kb < nkb && ok; ++kb) {
                const uint32_t s = kb % STAGES, round = kb / STAGES;
                const uint32_t full = smem_u32(&bar_full[s]);
                const uint32_t dst = smem_u32(smem + (size_t)s * STAGE_BYTES);
                if (kb >= early) {
                    ok = mbar_wait(smem_u32(&bar_empty[s]), (round & 1u) ^ 1u, status);
                    if (!ok) break;
                    mbar_expect_tx(full, (uint32_t)STAGE_BYTES);
                    tma_load_2d(dst + A_BYTES, &tm_w1, kb * BK, layer * DH, full);
                }
                tma_load_2d(dst, &tm_x, kb * BK, m0, full);
            }
            // W_r2 goes into stages 0 .. W2_STAGES-1 once the MMAs of the last k-block that used each of them have retired
            for (int s = 0; s < W2_STAGES && ok; ++s) {
                if (s < nkb) {
                    const int last = s + ((nkb - 1 - s) / STAGES) * STAGES;      // last k-block held by stage s
                    ok = mbar_wait(smem_u32(&bar_empty[s]), (uint32_t)(last / STAGES) & 1u, status);
                }
            }
            if (ok) {
                mbar_expect_tx(smem_u32(&bar_w2), (uint32_t)(KB2 * W2_KB_BYTES));
                for (int kb = 0; kb < KB2; ++kb)
                    tma_load_2d(smem_u32(w2_s + (size_t)kb * W2_KB_BYTES), &tm_w2, kb * BK, layer * E, smem_u32(&bar_w2));
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMA issuer
        if (lane == 0) {
            bool ok = true;
            const uint32_t idesc1 = instr_desc_bf16(BM, DH);
            for (int kb = 0; kb < nkb && ok; ++kb) {
                const uint32_t s = kb % STAGES, round = kb / STAGES;
                ok = mbar_wait(smem_u32(&bar_full[s]), round & 1u, status);
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t a_addr = smem_u32(smem + (size_t)s * STAGE_BYTES);
                const uint64_t da = smem_desc_sw128(a_addr), db = smem_desc_sw128(a_addr + A_BYTES);
#pragma unroll
                for (int q = 0; q < BK / UMMA_K; ++q) {
                    const uint64_t koff = (uint64_t)((q * UMMA_K * 2) >> 4);
                    umma_bf16(tmem_base, da + koff, db + koff, idesc1, (kb | q) != 0 ? 1u : 0u);
                }
                umma_commit(smem_u32(&bar_empty[s]));
            }
            umma_commit(smem_u32(&bar_acc1));              // u accumulator complete
            // second GEMM: wait for u (written to shared memory by the epilogue warps) and for W_r2
            ok = ok && mbar_wait(smem_u32(&bar_u_ready), 0, status) && mbar_wait(smem_u32(&bar_w2), 0, status);
            if (ok) {
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t idesc2 = instr_desc_bf16(BM, EN);
                for (int kb = 0; kb < KB2; ++kb) {
                    const uint64_t da = smem_desc_sw128(smem_u32(u_s + (size_t)kb * BM * 128));
                    const uint64_t db = smem_desc_sw128(smem_u32(w2_s + (size_t)kb * W2_KB_BYTES));
#pragma unroll
                    for (int q = 0; q < BK / UMMA_K; ++q) {
                        const uint64_t koff = (uint64_t)((q * UMMA_K * 2) >> 4);
                        umma_bf16(tmem_r, da + koff, db + koff, idesc2, (kb | q) != 0 ? 1u : 0u);
                    }
                }
            }
            umma_commit(smem_u32(&bar_acc2));
        }
    } else {
        // ------------------------------------------------------------------ 16 epilogue warps
        // warp -> TMEM lane quadrant (warp & 3) and one of four column parts; a thread owns one token row
        const int quad = warp & 3, part = (warp - 2) >> 2;
        const int r_local = quad * 32 + lane;
        const int row = m0 + r_local;
        const uint32_t lane_base = (uint32_t)(quad * 32) << 16;
        auto publish = [&](int k_warp, bool cond_warp) { publish_batch(ksum, io.l[layer].status, quad, lane, k_warp, cond_warp, warp_k, warp_bad); };
        // biases, while the first GEMM runs (in front of the first barrier they held up its loads)
        for (int i = (int)threadIdx.x - 64; i < DH; i += NTHREADS - 64) b1_s[i] = b_r1 ? __bfloat162float(b_r1[i]) : 0.0f;
        for (int i = (int)threadIdx.x - 64; i < 256; i += NTHREADS - 64) b2_s[i] = (b_r2 && i < E) ? __bfloat162float(b_r2[i]) : 0.0f;
        asm volatile("bar.sync 1, %0;" ::"n"(NTHREADS - 64) : "memory");
        int okw = 1;
        if (lane == 0) okw = mbar_wait(smem_u32(&bar_acc1), 0, status) ? 1 : 0;
        bool ok = __shfl_sync(0xffffffffu, okw, 0) != 0;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (ok) {
            // ---- epilogue 1: u = relu(acc + b_r1) -> bf16 -> swizzled K-major tile in shared memory
            constexpr int C1 = DH / 4;                     // columns of u per part
#pragma unroll
            for (int cc = 0; cc < C1; cc += 16) {
                const int c0 = part * C1 + cc;
                uint32_t acc[16];
                tmem_ld16(tmem_base + lane_base + (uint32_t)c0, acc);
                uint32_t pk[8];
#pragma unroll
                for (int j = 0; j < 16; j += 2) {
                    const __nv_bfloat162 v = __floats2bfloat162_rn(fmaxf(__uint_as_float(acc[j]) + b1_s[c0 + j], 0.0f),
                                                                   fmaxf(__uint_as_float(acc[j + 1]) + b1_s[c0 + j + 1], 0.0f));
                    pk[j >> 1] = *reinterpret_cast<const uint32_t *>(&v);
                }
                // 16 columns = two 16-byte chunks of this row inside k-block c0/64; chunk index XOR (row % 8)
                const int kb = c0 >> 6, chunk = (c0 & 63) >> 3;
                uint8_t *rowp = u_s + (size_t)kb * BM * 128 + (size_t)r_local * 128;
                *reinterpret_cast<uint4 *>(rowp + (((chunk) ^ (r_local & 7)) << 4)) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
                *reinterpret_cast<uint4 *>(rowp + (((chunk + 1) ^ (r_local & 7)) << 4)) = make_uint4(pk[4], pk[5], pk[6], pk[7]);
            }
            // make the generic-proxy writes visible to the tensor-core (async) proxy, then signal the MMA warp
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&bar_u_ready));

            // ---- epilogue 2: R = |acc + b_r2|; part p owns mask words p and p + 4 (columns 32w .. 32w+31)
            if (lane == 0) okw = mbar_wait(smem_u32(&bar_acc2), 0, status) ? 1 : 0;
            ok = __shfl_sync(0xffffffffu, okw, 0) != 0;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const int W = (E + 31) / 32;
            float v[TWO ? 1 : 2][TWO ? 16 : 32];
            // 16 scores of this thread's row, from column c0 on
            auto scores16 = [&](int c0, float *o) {
                uint32_t acc[16];
                tmem_ld16(tmem_r + lane_base + (uint32_t)c0, acc);
#pragma unroll
                for (int j = 0; j < 16; j += 4) {
                    const float4 b = *reinterpret_cast<const float4 *>(b2_s + c0 + j);
                    o[j] = fabsf(__uint_as_float(acc[j]) + b.x);
                    o[j + 1] = fabsf(__uint_as_float(acc[j + 1]) + b.y);
                    o[j + 2] = fabsf(__uint_as_float(acc[j + 2]) + b.z);
                    o[j + 3] = fabsf(__uint_as_float(acc[j + 3]) + b.w);
                }
            };
            // Scores are non-negative, so their bit patterns order like the values, with infinities and NaNs on top: ONE integer
            // maximum per element yields the row maximum and whether a score is not finite.
            uint32_t mb = 0u;
            if (ok) {
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    const int w = part + 4 * q;
                    if (w < W) {
                        const bool whole = w * 32 + 32 <= E;
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const int c0 = w * 32 + h * 16;
                            float *const o = TWO ? v[0] : &v[TWO ? 0 : q][TWO ? 0 : h * 16];
                            if (c0 < EN) {
                                scores16(c0, o);
                                if (whole) {
#pragma unroll
                                    for (int j = 0; j < 16; ++j) mb = max(mb, __float_as_uint(o[j]));
                                } else {
#pragma unroll
                                    for (int j = 0; j < 16; ++j)
                                        if (c0 + j < E) mb = max(mb, __float_as_uint(o[j]));
                                }
                                if (R && row < T) store_scores16(R, row, E, c0, o);
                            } else {
#pragma unroll
                                for (int j = 0; j < 16; ++j) o[j] = 0.0f;
                            }
                        }
                    }
                }
            }
            if (do_mask) {
                // row maximum across the four column parts, through shared memory
                pmax_s[part * BM + r_local] = mb;
                asm volatile("bar.sync 1, 512;" ::: "memory");           // the 16 epilogue warps only
                uint32_t mm = pmax_s[r_local];
#pragma unroll
                for (int p = 1; p < 4; ++p) mm = max(mm, pmax_s[p * BM + r_local]);
                const bool bad = mm >= 0x7f800000u;
                // a row with a score that is not finite keeps every expert: no score is below a negative threshold
                const float thr = bad ? -1.0f : __fmul_rn(tau, __uint_as_float(mm));
                int kt = 0;
                if (ok) {
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        const int w = part + 4 * q;
                        if (w < W) {
                            uint32_t word = 0u;
                            if constexpr (TWO) {
#pragma unroll
                                for (int h = 0; h < 2; ++h) {
                                    if (w * 32 + h * 16 >= EN) continue;
                                    scores16(w * 32 + h * 16, v[0]);
#pragma unroll
                                    for (int j = 0; j < 16; ++j) word |= !(v[0][j] < thr) ? 1u << (h * 16 + j) : 0u;
                                }
                            } else {
#pragma unroll
                                for (int j = 0; j < 32; ++j) word |= !(v[q][j] < thr) ? 1u << j : 0u;
                            }
                            if (w * 32 + 32 > E) word &= (1u << (E - w * 32)) - 1u;
                            if (row < T) {
                                mask[(size_t)row * W + w] = word;
                                if (io.mask_cat) io.mask_cat[(size_t)row * io.cat_words + layer * W + w] = word;
                            }
                            kt += __popc(word);
                        }
                    }
                }
                pk_s[part * BM + r_local] = kt;
                asm volatile("bar.sync 1, 512;" ::: "memory");
                if (part == 0) {
                    int k_row = 0;
                    if (row < T) {
                        k_row = pk_s[r_local] + pk_s[BM + r_local] + pk_s[2 * BM + r_local] + pk_s[3 * BM + r_local];
                        k[row] = k_row;
                        if (bad) atomicMax(status, (int32_t)D2D_ERR_NONFINITE);
                    }
                    if (ksum) {
                        const bool any = __any_sync(0xffffffffu, bad && row < T);
#pragma unroll
                        for (int o = 16; o > 0; o >>= 1) k_row += __shfl_xor_sync(0xffffffffu, k_row, o);
                        publish(k_row, any || !ok);
                    }
                }
            }
        } else if (do_mask) {
            // keep the named barrier balanced when a bounded wait ran out
            asm volatile("bar.sync 1, 512;" ::: "memory");
            asm volatile("bar.sync 1, 512;" ::: "memory");
            if (ksum && part == 0) publish(0, true);
        }
    }

    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 1) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(TMEM_COLS) : "memory");
    }
}

// Second router layer and selection for the shapes the kernel above has no room for (d_h up to 256, E up to 384): u comes from
// a GEMM of its own, and this kernel reads it once, keeps the scores in TMEM and writes mask and k (and R when wanted).
// One CTA per 128 tokens.  All of u's tile (d_h / 64 k-blocks of 16 KB) and three k-blocks of W_r2 (128-row boxes, up to
// 48 KB each) are in flight at once; a fourth k-block takes the first one's place.  The scores fill up to 384 TMEM columns, too
// many for registers, so the epilogue reads them twice: once for the row maxima, once for the mask words.
// Bound by latency (one CTA per SM at most, one tile each): loads, 4 k-blocks of MMAs, two passes over TMEM.  Measured at
// d = 4096, d_h = 256, E = 344, against a GEMM that wrote R and a kernel that read it twice (11 MB each way): hidden layer and
// scores 38 us against 57 us at 8192 tokens (launches on their own, cold L2); the whole layer 110.7 -> 104.6 us at 128 tokens,
// at 8192 in three runs of each side 1688 to 1716 -> 1629 to 1692.
constexpr int S_MAX_KB = 4, S_STAGES = 3, S_STAGE_BYTES = 384 * 128, S_WORDS = 3;      // a part owns mask words p, p + 4, p + 8
__global__ void __launch_bounds__(NTHREADS, 1)
router_scores_kernel(const __grid_constant__ CUtensorMap tm_u, const __grid_constant__ CUtensorMap tm_w2,
                     const __nv_bfloat16 *__restrict__ b_r2, int T, int kb2, int E, int EN /* E rounded up to 16 */, float tau,
                     const __grid_constant__ RouterGroupIO io)
{
    float *__restrict__ R = io.l[0].R;
    int32_t *__restrict__ status = io.ksum[0] + 2;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *u_s = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t *w2_s = u_s + (size_t)S_MAX_KB * BM * 128;
    __shared__ uint64_t bar_u, bar_w[S_MAX_KB], bar_free, bar_acc;
    __shared__ uint32_t tmem_base_holder;
    __shared__ __align__(16) float b2_s[384];
    __shared__ uint32_t pmax_s[4 * BM];
    __shared__ int pk_s[4 * BM];
    __shared__ int warp_k[4], warp_bad[4];
    for (int i = threadIdx.x; i < 384; i += NTHREADS) b2_s[i] = (b_r2 && i < E) ? __bfloat162float(b_r2[i]) : 0.0f;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int m0 = blockIdx.x * BM;
    const int boxes = (E + 127) / 128;
    auto load_w2 = [&](int kb) {
        mbar_expect_tx(smem_u32(&bar_w[kb]), (uint32_t)boxes * 128 * 128);
        for (int i = 0; i < boxes; ++i)
            tma_load_2d(smem_u32(w2_s + (size_t)(kb % S_STAGES) * S_STAGE_BYTES + (size_t)i * 128 * 128), &tm_w2, kb * BK, i * 128,
                        smem_u32(&bar_w[kb]));
    };
    if (threadIdx.x == 0) {
        for (int kb = 0; kb < S_MAX_KB; ++kb) mbar_init(smem_u32(&bar_w[kb]), 1);
        mbar_init(smem_u32(&bar_u), 1);
        mbar_init(smem_u32(&bar_free), 1);
        mbar_init(smem_u32(&bar_acc), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        // the weights do not depend on the previous kernel of the stream
        for (int kb = 0; kb < kb2 && kb < S_STAGES; ++kb) load_w2(kb);
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_holder)), "r"(512u)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_base = tmem_base_holder;
    // The up projection behind this kernel may start at once, beside the hidden layer: this kernel runs since every CTA of that one
    // has waited for what came before, so x and the workspace are the layer's own; what depends on the mask waits for this kernel.
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");

    if (warp == 0) {
        if (lane == 0) {
            mbar_expect_tx(smem_u32(&bar_u), (uint32_t)kb2 * BM * 128);
            for (int kb = 0; kb < kb2; ++kb) tma_load_2d(smem_u32(u_s + (size_t)kb * BM * 128), &tm_u, kb * BK, m0, smem_u32(&bar_u));
            if (kb2 > S_STAGES && mbar_wait(smem_u32(&bar_free), 0, status)) load_w2(S_STAGES);
        }
    } else if (warp == 1) {
        if (lane == 0) {
            bool ok = mbar_wait(smem_u32(&bar_u), 0, status);
            for (int kb = 0; kb < kb2 && ok; ++kb) {
                ok = mbar_wait(smem_u32(&bar_w[kb]), 0, status);
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint64_t da = smem_desc_sw128(smem_u32(u_s + (size_t)kb * BM * 128));
                const uint32_t w_addr = smem_u32(w2_s + (size_t)(kb % S_STAGES) * S_STAGE_BYTES);
                for (int n0 = 0; n0 < EN; n0 += 256) {       // one instruction takes at most 256 columns
                    const uint64_t db = smem_desc_sw128(w_addr + (uint32_t)n0 * 128);
                    const uint32_t idesc = instr_desc_bf16(BM, min(EN - n0, 256));
#pragma unroll
                    for (int q = 0; q < BK / UMMA_K; ++q) {
                        const uint64_t koff = (uint64_t)((q * UMMA_K * 2) >> 4);
                        umma_bf16(tmem_base + (uint32_t)n0, da + koff, db + koff, idesc, (kb | q) != 0 ? 1u : 0u);
                    }
                }
                if (kb == 0) umma_commit(smem_u32(&bar_free));
            }
            umma_commit(smem_u32(&bar_acc));
        }
    } else {
        const int quad = warp & 3, part = (warp - 2) >> 2;
        const int r_local = quad * 32 + lane, row = m0 + r_local;
        const uint32_t lane_base = (uint32_t)(quad * 32) << 16;
        const int W = (E + 31) / 32;
        int okw = 1;
        if (lane == 0) okw = mbar_wait(smem_u32(&bar_acc), 0, status) ? 1 : 0;
        const bool ok = __shfl_sync(0xffffffffu, okw, 0) != 0;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        auto scores16 = [&](int c0, float (&v)[16]) {
            uint32_t acc[16];
            tmem_ld16(tmem_base + lane_base + (uint32_t)c0, acc);
#pragma unroll
            for (int j = 0; j < 16; j += 4) {
                const float4 b = *reinterpret_cast<const float4 *>(b2_s + c0 + j);
                v[j] = fabsf(__uint_as_float(acc[j]) + b.x);
                v[j + 1] = fabsf(__uint_as_float(acc[j + 1]) + b.y);
                v[j + 2] = fabsf(__uint_as_float(acc[j + 2]) + b.z);
                v[j + 3] = fabsf(__uint_as_float(acc[j + 3]) + b.w);
            }
        };
        uint32_t mb = 0u;                                    // integer maximum of the bit patterns, as above
        for (int q = 0; q < S_WORDS && ok; ++q) {
            const int w = part + 4 * q;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int c0 = w * 32 + h * 16;
                if (c0 >= EN) break;
                float v[16];
                scores16(c0, v);
#pragma unroll
                for (int j = 0; j < 16; ++j) mb = max(mb, c0 + j < E ? __float_as_uint(v[j]) : 0u);
                if (R && row < T) store_scores16(R, row, E, c0, v);
            }
        }
        pmax_s[part * BM + r_local] = mb;
        asm volatile("bar.sync 1, 512;" ::: "memory");
        uint32_t mm = pmax_s[r_local];
#pragma unroll
        for (int p = 1; p < 4; ++p) mm = max(mm, pmax_s[p * BM + r_local]);
        const bool bad = mm >= 0x7f800000u;
        const float thr = bad ? -1.0f : __fmul_rn(tau, __uint_as_float(mm));
        int kt = 0;
        for (int q = 0; q < S_WORDS && ok; ++q) {
            const int w = part + 4 * q;
            if (w >= W) break;
            uint32_t word = 0u;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int c0 = w * 32 + h * 16;
                if (c0 >= EN) break;
                float v[16];
                scores16(c0, v);
#pragma unroll
                for (int j = 0; j < 16; ++j) word |= !(v[j] < thr) ? 1u << (h * 16 + j) : 0u;
            }
            if (w * 32 + 32 > E) word &= (1u << (E - w * 32)) - 1u;
            if (row < T) io.l[0].mask[(size_t)row * W + w] = word;
            kt += __popc(word);
        }
        pk_s[part * BM + r_local] = kt;
        asm volatile("bar.sync 1, 512;" ::: "memory");
        if (part == 0) {
            int k_row = 0;
            if (row < T) {
                k_row = pk_s[r_local] + pk_s[BM + r_local] + pk_s[2 * BM + r_local] + pk_s[3 * BM + r_local];
                io.l[0].k[row] = k_row;
                if (bad) atomicMax(status, (int32_t)D2D_ERR_NONFINITE);
            }
            const bool any = __any_sync(0xffffffffu, bad && row < T);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) k_row += __shfl_xor_sync(0xffffffffu, k_row, o);
            publish_batch(io.ksum[0], io.l[0].status, quad, lane, k_row, any || !ok, warp_k, warp_bad);
        }
    }

    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 1)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
}

// Launch with programmatic dependent launch; `done` remembers per device that the kernel's shared memory limit is set.
template <typename K, typename... A>
d2d_status launch_kernel(K kern, bool (&done)[64], dim3 grid, size_t smem, cudaStream_t st, A... args)
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return D2D_ERR_CUDA;
    if (!__atomic_load_n(&done[dev], __ATOMIC_ACQUIRE)) {
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) return D2D_ERR_CUDA;
        __atomic_store_n(&done[dev], true, __ATOMIC_RELEASE);
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(NTHREADS, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = d2d_tc_pdl_enabled() ? 1 : 0;
    const cudaError_t err = cudaLaunchKernelEx(&cfg, kern, args...);
    D2D_LAUNCHED(1);
    return err == cudaSuccess ? D2D_OK : D2D_ERR_CUDA;
}

template <int DH, bool TWO>
d2d_status launch_for(const d2d_layer_desc &D, const d2d_router_weights &w, int n_layers, const void *x, int T, float tau, int do_mask,
                  const RouterGroupIO &io, cudaStream_t st)
{
    constexpr int STAGE_BYTES = BM * BK * 2 + DH * BK * 2;
    constexpr int KB2 = DH / BK;
    constexpr size_t SMEM = (size_t)stages_for(TWO) * STAGE_BYTES + (TWO ? 0 : (size_t)KB2 * BM * 128) + 1024;
    CUtensorMap tx, tw1, tw2;
    if (!d2d_tc_make_map(&tx, x, T, D.d, BM) || !d2d_tc_make_map(&tw1, w.w_r1, D.d_h * n_layers, D.d, DH) ||
        !d2d_tc_make_map(&tw2, w.w_r2, D.n_experts * n_layers, D.d_h, 256))
        return D2D_ERR_CUDA;
    static bool attr_set[64] = {};                         // the attribute is per device
    return launch_kernel(router_fused_kernel<DH, TWO>, attr_set, dim3(d2d_cdiv(T, BM), n_layers, 1), SMEM, st, tx, tw1, tw2,
                         (const __nv_bfloat16 *)w.b_r1, (const __nv_bfloat16 *)w.b_r2, T, D.d, D.n_experts,
                         (D.n_experts + 15) / 16 * 16, tau, do_mask, io);
}

template <int DH>
d2d_status launch(const d2d_layer_desc &D, const d2d_router_weights &w, int n_layers, const void *x, int T, float tau, int do_mask,
                  const RouterGroupIO &io, cudaStream_t st)
{
    // More row tiles than SMs: two CTAs per SM, so that the last round is not a nearly empty one of its own and the up projection
    // starts behind the first.  Bound by the latency of a CTA's chain (loads, two GEMMs, epilogues), which two CTAs overlap.  ViT-shaped
    // layer, 25216 tokens (197 tiles on 148 SMs): 248.4 us with one CTA per SM, 245.0 with two.  Up to one tile per SM the
    // five stages of the other form are in nobody's way and hide more of the latency.
    return d2d_cdiv(T, BM) * n_layers > d2d_tc_sm_count() ? launch_for<DH, true>(D, w, n_layers, x, T, tau, do_mask, io, st)
                                                          : launch_for<DH, false>(D, w, n_layers, x, T, tau, do_mask, io, st);
}

}  // namespace

bool d2d_router_fused_supports(const d2d_layer_desc &D, int T)
{
    // d_h = 128 (the paper's router width) and E <= 256: operand ring, u and W_r2 then fit in shared memory together
    return D.dtype == D2D_BF16 && T > d2d_decode_max_tokens(D) && D.d_h == 128 && D.n_experts <= 256 && D.d % 8 == 0 &&
           T <= 16000 * BM && d2d_gemm_tc_available();          // (the exit count has 14 bits)
}

// R may be NULL when only the mask is wanted; mask / k / status are used when do_mask != 0.
d2d_status d2d_router_fused(const d2d_layer *L, const void *x, int T, float tau, int do_mask, float *R, uint32_t *mask,
                            int32_t *k, int32_t *status, cudaStream_t st, int32_t *ksum)
{
    RouterGroupIO io = {};
    io.l[0] = {R, mask, k, status};
    io.ksum[0] = do_mask ? ksum : nullptr;
    const d2d_router_weights w = {L->w_r1, L->b_r1, L->w_r2, L->b_r2};
    return launch<128>(L->desc, w, 1, x, T, tau, do_mask, io, st);
}

// n routers of one shape with stacked weights, one grid; routing[l] receives mask, k and status of router l.
d2d_status d2d_router_fused_group(const d2d_layer *const *layers, int n_layers, const d2d_router_weights &w, const void *x, int T,
                                  float tau, const d2d_routing *routing, uint32_t *mask_cat, int cat_words, cudaStream_t st)
{
    if (n_layers < 1 || n_layers > D2D_MAX_GROUP) return D2D_ERR_INVALID_ARG;
    RouterGroupIO io = {};
    for (int l = 0; l < n_layers; ++l) {
        io.l[l] = {nullptr, routing[l].mask, routing[l].k, routing[l].status};
        io.ksum[l] = (int32_t *)(layers[l]->tickets + 40);
    }
    io.mask_cat = mask_cat;
    io.cat_words = cat_words;
    return launch<128>(layers[0]->desc, w, n_layers, x, T, tau, 1, io, st);
}

bool d2d_router_scores_supports(const d2d_layer_desc &D, int T)
{
    // u's tile and three k-blocks of W_r2 fill the shared memory at d_h = 256 and E = 384
    return D.dtype == D2D_BF16 && T > d2d_decode_max_tokens(D) && D.d_h <= S_MAX_KB * BK && D.d_h % 8 == 0 && D.n_experts <= S_STAGE_BYTES / 128 &&
           D.d % 8 == 0 && T <= 16000 * BM && d2d_gemm_tc_available();
}

d2d_status d2d_router_scores(const d2d_layer *L, const void *x, void *u, int T, float tau, float *R, uint32_t *mask,
                             int32_t *k, int32_t *status, cudaStream_t st, int32_t *ksum)
{
    const d2d_layer_desc &D = L->desc;
    d2d_gemm_args l1 = {};
    l1.a = x; l1.b = L->w_r1; l1.bias = L->b_r1; l1.out = u;
    l1.M = T; l1.N = D.d_h; l1.K = D.d; l1.epilogue = D2D_EPI_RELU_BF16;
    const d2d_status rc = d2d_gemm_tc(l1, st);
    if (rc != D2D_OK) return rc;
    RouterGroupIO io = {};
    io.l[0] = {R, mask, k, status};
    io.ksum[0] = ksum;
    CUtensorMap tu, tw2;
    if (!d2d_tc_make_map(&tu, u, T, D.d_h, BM) || !d2d_tc_make_map(&tw2, L->w_r2, D.n_experts, D.d_h, 128)) return D2D_ERR_CUDA;
    static bool attr_set[64] = {};
    return launch_kernel(router_scores_kernel, attr_set, dim3(d2d_cdiv(T, BM), 1, 1),
                         (size_t)S_MAX_KB * BM * 128 + (size_t)S_STAGES * S_STAGE_BYTES + 1024, st, tu, tw2, (const __nv_bfloat16 *)L->b_r2, T,
                         d2d_cdiv(D.d_h, BK), D.n_experts, (D.n_experts + 15) / 16 * 16, tau, io);
}
