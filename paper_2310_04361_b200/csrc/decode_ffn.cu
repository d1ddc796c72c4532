// Expert step of a decode batch (Sec. 3.2, 3.4; gated form App. G): y = b2 + sum over kept experts, for a few tokens.
//
// Bound by the bytes of the kept experts' weights.  The unit of work is 16 adjacent neurons: their rows of W1 (and
// W_gate) and of the transposed W2.  A cluster of CL CTAs takes CL units per round: CTA r forms the 16 hidden values of unit
// r for all tokens, hands them (a few hundred bytes) to the other CTAs through distributed shared memory, and all CTAs
// then add all CL units' contributions to their own d / CL output columns.  The output accumulators of those columns stay
// in registers from the first round to the last, so a CTA adds T d / CL floats to the result, once (CTAs that kept all
// columns added CL times as much: 6 us of reductions, fences and conversion behind 13 tokens of a d = 1024 layer).
//
// A producer warp streams the weights into a ring of 32 KB stages of [16 rows x 128 bytes] blocks, brought by TMA requests
// for up to 16 blocks each (a 3-D box; one request per row piece measured 50 ns a piece, a third of the memory rate); 16
// consumer warps compute.  The matrix instructions are the warp-level ones: at 8 to 32 tokens the tensor pipe is idle
// either way, and these read weights as their 16-row operand with no padding to 128 rows.
//
// Which units: a cluster starts on `n_static` rounds fixed by its index before the selection is known (their copies and
// up projections run beside the router), and takes its share of the others once the router's list of kept units is
// there.  The up projection of the next round precedes the down projection of the current one, which hides the exchange.
// The last CTA to add to its columns (a ticket per rank) adds b2 and writes y.
//
// Measured, whole layer calls back to back (small_batch_ffn.cu or the tensor-core path -> these two kernels): d = 1024,
// 256 experts of 16: 18.1 -> 12.1 us at 1 token, 38 -> 14.7 us at 13; d = 4096, 344 gated experts of 32: 114 -> 56.8 us at 7
// tokens, 64 -> 37 us at 1 with 8-bit weights; three d = 1024 layers of 128 experts on 8 shared tokens: 43 -> 15.8 us.
//
// How many tokens fit is a matter of shared memory: the token rows, the partial sums and the hidden values grow with them, and
// the ring beside them needs three stages.  One layer of bf16 weights: 32 tokens with d = 512 or 640, 16 with 768, 1024 or 2048, 8
// with 4096.  Beyond that the tensor-core path takes over with a step in time (d = 1024: 15.1 us at 16 tokens, 24.5 at 17; d = 4096:
// 63 us at 8 tokens, 73 at 9).
#include <cuda_fp8.h>

#include "decode.cuh"
#include "tc_common.cuh"

namespace {

using namespace d2d_decode;

constexpr int NCW = 16, NC = NCW * 32, NT = NC + 64;      // consumer warps / threads, all threads (a producer warp, one that talks to the cluster)
constexpr int SUB_BYTES = 16 * 128;                       // a block: 16 rows x 128 bytes, 128-byte swizzle
constexpr int STAGE_BLOCKS = 16, STAGE_BYTES = STAGE_BLOCKS * SUB_BYTES;
constexpr int MAX_STAGES = 6;
constexpr int MAX_UNITS = 4096, MAX_LIST = 128;          // units of a layer; entries of a cluster's list (see plan)
constexpr int H_ROW = 48;                                 // bytes between tokens' rows of 16 hidden values: free of bank conflicts
constexpr unsigned FULL = 0xffffffffu;

template <typename WT> __host__ __device__ constexpr int sub_cols() { return 128 / (int)sizeof(WT); }       // columns per warp and stage
template <typename WT> __host__ __device__ constexpr int seg_cols() { return NCW * sub_cols<WT>(); }        // columns per stage
// Token rows in shared memory: 16 bytes beyond a multiple of 128, so that eight rows' 16-byte pieces do not meet in a bank
__host__ __device__ constexpr int x_pitch(int d) { return (d * 2 + 127) / 128 * 128 + 16; }

// One stage: 16 rows from `row` on, the 128-byte column blocks from `block` on (3-D map: column in block, row, block)
// `policy`: weights that do not stay in L2 from one call to the next anyway leave it first, so that what both decode kernels
// keep coming back to (their instructions above all) stays: with 270 MB of weights passing through L2 in a call, every piece of
// code that an SM ran for the first time in a launch came from a busy memory, 1 to 2 us a time (Llama-shaped layer, 7 tokens:
// 68.5 -> 65.5 us, 8-bit weights at 1 token: 55.7 -> 53).  Layers whose weights L2 holds lose by it (d = 1024, 13 tokens, 16 MB:
// 15.4 -> 15.7 us, three layers of 8 MB: 17.3 -> 17.9).
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap *map, int row, int block, uint32_t bar, uint64_t policy)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%2, %3, %4}], [%5], %6;"
        ::"r"(dst), "l"(map), "r"(0), "r"(row), "r"(block), "r"(bar), "l"(policy) : "memory");
}
__device__ __forceinline__ uint64_t weight_policy(bool pass)
{
    uint64_t p;
    if (pass) asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    else asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(p));
    return p;
}
__device__ __forceinline__ void red_add4(float *p, float4 v)
{
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}
__device__ __forceinline__ uint32_t cluster_addr(uint32_t addr, uint32_t rank)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
// 16 bytes into the shared memory of another CTA of the cluster; counted by that CTA's barrier
__device__ __forceinline__ void st_async4(uint32_t addr, uint4 v, uint32_t bar)
{
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];"
                 ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w), "r"(bar) : "memory");
}
__device__ __forceinline__ void arrive_cluster(uint32_t bar)
{
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
// ... announcing `bytes` bytes of asynchronous stores (which order themselves, and may have been counted before: relaxed)
__device__ __forceinline__ void arrive_cluster(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.relaxed.cluster.shared::cluster.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void consumer_bar() { asm volatile("bar.sync 1, %0;" ::"n"(NC) : "memory"); }

// Two e4m3 codes as a bf16 pair.  t holds them in the upper bytes of its halves (lower bytes: anything).  Sign and the
// seven exponent and mantissa bits are moved to where bf16 has them; the exponent's bias differs by 127 - 7, which one
// exact multiplication by 2^120 makes up (also for the codes below the normal range).
__device__ __forceinline__ uint32_t e4m3_to_bf16x2(uint32_t t)
{
    const uint32_t v = ((t >> 4) & 0x07f007f0u) | (t & 0x80008000u);
    const uint32_t scale = 0x7b807b80u;                   // 2^120 twice
    uint32_t r;
    asm("mul.rn.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(v), "r"(scale));
    return r;
}

// Shared-memory offset of byte `col` of row `row` inside a warp's sub-tile (16-byte pieces XORed with the row)
__device__ __forceinline__ uint32_t swz(int row, int col) { return (uint32_t)(row * 128 + (col ^ ((row & 7) << 4))); }

// Four 8 x 8 matrices of bf16; lane i gives the row address of row i % 8 of matrix i / 8.  TRANS: each is transposed.
template <bool TRANS> __device__ __forceinline__ void ldmatrix4(uint32_t (&o)[4], uint32_t addr)
{
    if (TRANS)
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];" : "=r"(o[0]), "=r"(o[1]), "=r"(o[2]), "=r"(o[3]) : "r"(addr) : "memory");
    else
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];" : "=r"(o[0]), "=r"(o[1]), "=r"(o[2]), "=r"(o[3]) : "r"(addr) : "memory");
}
// Column j of four of two rows of codes (four adjacent columns each) as a bf16 pair, lower half = first row
template <int J> __device__ __forceinline__ uint32_t pair_of(uint32_t r0, uint32_t r1)
{
    return e4m3_to_bf16x2(__byte_perm(r0, r1, ((4 + J) << 12) | (J << 4)));
}
// Sixteen codes -> eight float16 pairs, in order
__device__ __forceinline__ void widen16(const uint4 &r, uint32_t (&o)[8])
{
    const uint32_t w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        asm("{\n\t.reg .b16 lo, hi;\n\tmov.b32 {lo, hi}, %2;\n\tcvt.rn.f16x2.e4m3x2 %0, lo;\n\tcvt.rn.f16x2.e4m3x2 %1, hi;\n\t}"
            : "=r"(o[2 * i]), "=r"(o[2 * i + 1]) : "r"(w[i]));
    }
}
// Place of columns 4 q .. 4 q + 3 (8 bytes) of a token row beside codes: every 32 columns, two 16-column pieces a and b, become
// a[0..3] b[0..3] a[4..7] b[4..7] ..., so that a lane of a matrix instruction finds its four columns of both pieces in 16 bytes.
__device__ __forceinline__ uint32_t x_place(int q) { return (uint32_t)((q & ~7) | ((q & 3) << 1) | ((q >> 2) & 1)) * 8u; }
__device__ __forceinline__ uint2 lds8(uint32_t addr)
{
    uint2 v;
    asm volatile("ld.shared.v2.b32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ uint4 lds16(uint32_t addr)
{
    uint4 v;
    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
    return v;
}
// Eight codes -> four bfloat16 pairs, in order (by way of float16: a code's value is exact in either)
__device__ __forceinline__ void widen8(const uint2 &r, uint32_t (&o)[4])
{
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const __half2_raw h = __nv_cvt_fp8x2_to_halfraw2((__nv_fp8x2_storage_t)((i < 2 ? r.x : r.y) >> (16 * (i & 1))), __NV_E4M3);
        const float2 f = __half22float2(__half2(h));
        const __nv_bfloat162 b = __floats2bfloat162_rn(f.x, f.y);
        o[i] = *reinterpret_cast<const uint32_t *>(&b);
    }
}
// mma16816 on float16 operands
__device__ __forceinline__ void mma16816_f16(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1)
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// The up projection of a unit from codes and bfloat16 rows, for rows that float16 would not hold.  Rare, but what it does to the code
// around it is paid by every call: a function of its own where accumulators leave registers for one, in line where they do not
// (Llama-shaped layer, us, function / in line / no such rows: 38.3 / 39.5 / 37.9 at 1 token, 55.4 / 57.1 / 54.9 at 2; with 8 tiles a
// warp 68.0 / 61.9 / 60.8 at 6, 62.0 / 59.0 / 58.3 at 8).
struct up_rows {
    uint32_t bar_full, bar_empty, ring, xs;
    int xp, T, d, nq, n_mat, stages, warp, slot;
    uint32_t phase;
    int32_t *status;                                          // NULL: a wait has run out before, there is nothing to wait for
};
template <int NT8, int CH> struct up_sums {
    float v[2][NT8 * CH][4];
    int slot;
    uint32_t phase;
    bool ok;
};
template <int NT8, int CH> __device__ __forceinline__ up_sums<NT8, CH> up_spread_rows(up_rows a)
{
    const int lane = threadIdx.x & 31, g = lane >> 2, c = lane & 3;
    up_sums<NT8, CH> o;
#pragma unroll
    for (int m = 0; m < 2; ++m)
#pragma unroll
        for (int t = 0; t < NT8 * CH; ++t) o.v[m][t][0] = o.v[m][t][1] = o.v[m][t][2] = o.v[m][t][3] = 0.0f;
    o.ok = a.status != nullptr;
#pragma unroll 1
    for (int q = 0; q < a.nq; ++q) {
        const int k0 = q * seg_cols<uint8_t>() + a.warp * sub_cols<uint8_t>();
#pragma unroll
        for (int m = 0; m < 2; ++m) {
            if (m == 1 && a.n_mat == 1) break;
            if (o.ok) o.ok = d2d_tc::mbar_wait_warp(a.bar_full + 8 * a.slot, a.phase, a.status);
            const uint32_t st = a.ring + a.slot * STAGE_BYTES + a.warp * SUB_BYTES;
#pragma unroll 1
            for (int hp = 0; hp < 4 && k0 < a.d; ++hp) {      // half of the columns, 8-byte part of a 16-byte piece
                const int h = hp >> 1, p = hp & 1;
                uint32_t wa[2][4];
#pragma unroll
                for (int i = 0; i < 2; ++i) widen8(lds8(st + swz(g + 8 * i, c * 16 + h * 64) + p * 8), wa[i]);
#pragma unroll
                for (int t = 0; t < NT8; ++t) {
                    const uint4 xb = lds16(a.xs + min(t * 8 + g, a.T - 1) * a.xp + (k0 + h * 64) * 2 + c * 32 + p * 16);
                    mma16816(o.v[m][t * CH], wa[0][0], wa[1][0], wa[0][1], wa[1][1], xb.x, xb.y);
                    mma16816(o.v[m][t * CH + CH - 1], wa[0][2], wa[1][2], wa[0][3], wa[1][3], xb.z, xb.w);
                }
            }
            __syncwarp();
            if (lane == 0) d2d_tc::mbar_arrive(a.bar_empty + 8 * a.slot);
            if (++a.slot == a.stages) { a.slot = 0; a.phase ^= 1u; }
        }
    }
    o.slot = a.slot; o.phase = a.phase;
    return o;
}
template <int NT8, int CH> __device__ __noinline__ up_sums<NT8, CH> up_spread_rows_call(up_rows a) { return up_spread_rows<NT8, CH>(a); }

__device__ __forceinline__ float act_accurate(int act, float z)
{
    return act == D2D_ACT_RELU ? d2d_activate<D2D_ACT_RELU>(z) : act == D2D_ACT_GELU_ERF ? d2d_activate<D2D_ACT_GELU_ERF>(z)
         : act == D2D_ACT_GELU_TANH ? d2d_activate<D2D_ACT_GELU_TANH>(z) : d2d_activate<D2D_ACT_SILU>(z);
}
__device__ __forceinline__ float act_fast(int act, float z)
{
    return act == D2D_ACT_RELU ? d2d_tc::fast_act<D2D_ACT_RELU>(z) : act == D2D_ACT_GELU_ERF ? d2d_tc::fast_act<D2D_ACT_GELU_ERF>(z)
         : act == D2D_ACT_GELU_TANH ? d2d_tc::fast_act<D2D_ACT_GELU_TANH>(z) : d2d_tc::fast_act<D2D_ACT_SILU>(z);
}

// v 2^k, rounded once
__device__ __forceinline__ float times_pow2(float v, int k)
{
    return (unsigned)(k + 126) <= 252u ? v * __uint_as_float((uint32_t)(k + 127) << 23) : ldexpf(v, k);
}

struct FfnShape {
    int T, d, d_ff, E, s, W, act, gated;
    uint32_t inv_s;          // ceil(2^32 / s) for s > 1, see expert_of
    int planes;              // 3: hidden values kept to float32 precision and exact activations; 1: bf16 and the fast ones
    int cl, clusters;        // CTAs per cluster, clusters per layer
    int n_static, stages;    // rounds fixed by the cluster's index; stages of the ring
    int pass;                // the weights only pass through L2
    int up_blocks;           // blocks one request of the up matrices brings
    int nb, sps;             // blocks of a unit's rows of W2T one CTA reads (its d / cl columns); units per stage of those
};

// neuron / s.  The rounded-up reciprocal is exact for neurons below 2^16 (its error, less than s, times the neuron stays
// below 2^32); that of s = 1 does not fit 32 bits.
__device__ __forceinline__ int expert_of(const FfnShape &S, int neuron)
{
    return S.s == 1 ? neuron : (int)__umulhi((uint32_t)neuron, S.inv_s);
}

// TPW: 16-column output tiles per warp (d / cl <= 256 TPW); NT8: tokens / 8.
template <typename WT, int TPW, int NT8>
__global__ void __launch_bounds__(NT, 1)
decode_ffn_kernel(const __nv_bfloat16 *__restrict__ x, const FfnShape S, const __grid_constant__ d2d_decode_ffn_args args)
{
    constexpr int T8 = 8 * NT8;
    constexpr bool Q8 = sizeof(WT) == 1;
    constexpr int SUB = sub_cols<WT>(), SEG = seg_cols<WT>();
    constexpr int TPS = SUB / 16, PARTS = TPW > TPS ? TPW / TPS : 1, TPP = TPW > TPS ? TPS : TPW;      // tiles per warp: of a full stage; stages per unit; per stage
    constexpr int ACC = Q8 && TPW == 1 ? 2 : TPW;              // codes: tiles come in pairs (32 columns)
    const d2d_decode_ffn_layer &P = args.l[blockIdx.y];
    extern __shared__ unsigned char smem_raw[];
    unsigned char *smem = (unsigned char *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);       // swizzle atoms are 1024 bytes
    __shared__ uint64_t bar_full[MAX_STAGES], bar_empty[MAX_STAGES], h_full[3], h_empty[2], h_read[2], h_done[2], bar_go;
    __shared__ int unit_list[MAX_LIST], unit_list_p[MAX_LIST], n_units;
    __shared__ uint32_t keep_bits[MAX_UNITS / 32];
    __shared__ int keep_pre[MAX_UNITS / 32];
    __shared__ unsigned int my_ticket;
    __shared__ volatile int rounds_s, n_s;                     // all rounds of this cluster and the list's length, for the talking warp
    __shared__ uint32_t x_max[Q8 ? T8 * 16 : 1];               // codes: largest magnitude of the pieces of the token rows ...
    __shared__ float x_inv[T8];                                // ... what takes the scaling of a row back ...
    __shared__ int x_spread;                                   // ... and whether some row does not fit float16
    const int tid = threadIdx.x, lane = tid & 31, g = lane >> 2, c = lane & 3;
    const int warp = __shfl_sync(FULL, tid >> 5, 0);           // warp-uniform for the compiler: see mma16816
    const int d = S.d, T = S.T, U = S.d_ff / 16, CL = S.cl, NCL = S.clusters;
    const int rank = (int)blockIdx.x % CL, cid = (int)blockIdx.x / CL;
    const int n_mat = S.gated ? 2 : 1, nq = (d + SEG - 1) / SEG;
    const int xp = x_pitch(d);
    unsigned char *ring = smem;
    unsigned char *xs = ring + (size_t)S.stages * STAGE_BYTES;
    float *red = reinterpret_cast<float *>(xs + (size_t)T * xp);               // [n_mat][16 warps][16][T8]
    float *zs = red + (size_t)n_mat * NCW * 16 * T8;                           // [n_static + 1][3][16 * T8] up, gate, scale of a round
    unsigned char *hs = reinterpret_cast<unsigned char *>(zs + (size_t)(S.n_static + 1) * 3 * 16 * T8);     // [n_static + 2][CL][planes][T8] rows
    uint32_t *smask = reinterpret_cast<uint32_t *>(hs + (size_t)(S.n_static + 2) * CL * S.planes * T8 * H_ROW);     // [T][W], then the union [W]

    if (tid == 0) {
        for (int i = 0; i < S.stages; ++i) {
            d2d_tc::mbar_init(smem_addr(&bar_full[i]), 1);
            d2d_tc::mbar_init(smem_addr(&bar_empty[i]), NCW);
        }
        for (int i = 0; i < 3; ++i) d2d_tc::mbar_init(smem_addr(&h_full[i]), CL);
        for (int i = 0; i < 2; ++i) {
            d2d_tc::mbar_init(smem_addr(&h_empty[i]), CL);
            d2d_tc::mbar_init(smem_addr(&h_read[i]), NCW);
            d2d_tc::mbar_init(smem_addr(&h_done[i]), NCW);
        }
        d2d_tc::mbar_init(smem_addr(&bar_go), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncwarp();
    cluster_arrive();
    cluster_wait();                                            // the barriers of every CTA of the cluster exist
    pdl_trigger();

    // Rounds: the first `my_static` take units (cid + r * NCL) * CL + slot, the others the list's entries in the same order.
    // `n`: entries of the list.  Slots are filled from 0 on: `slots` of a round hold a unit.
    const int my_static = min(S.n_static, cid * CL < U ? (U - cid * CL + NCL * CL - 1) / (NCL * CL) : 0);
    auto rounds_for = [&](int n) { return my_static + (n > cid * CL ? (n - cid * CL + NCL * CL - 1) / (NCL * CL) : 0); };
    auto slots = [&](int r, int n) { return min(CL, r < my_static ? U - (cid + r * NCL) * CL : n - (cid + (r - my_static) * NCL) * CL); };
    auto unit_of = [&](int r, int k, const int *list) { return r < my_static ? (cid + r * NCL) * CL + k : list[(r - my_static) * CL + k]; };
    // whether, after the static rounds' up projections, round ru's comes before round rd's down projection
    auto up_next = [&](int ru, int rd, int R) { return ru < R && ru <= rd + 1 && !(ru == my_static && rd < my_static); };
    // this cluster's entries of the router's list
    auto load_list = [&](int *list, int i0, int step) {
        for (int i = i0; i < MAX_LIST; i += step) {
            const int j = (cid + i / CL * NCL) * CL + i % CL;
            if (j >= U) break;
            list[i] = __ldcg(P.units + 1 + j);
        }
    };

    // Hidden values live in buffers [static round, or n_static + the parity of a shared round][slot]; the static rounds' are
    // exchanged together, once.
    auto buffer = [&](int r) { return hs + (size_t)(r < my_static ? r : S.n_static + ((r - my_static) & 1)) * CL * S.planes * T8 * H_ROW; };

    if (warp == NCW) {
        // ------------------------------------------------------------------ producer
        uint32_t it = 0, phase = 1;                                            // stages requested; parity of "free" at `slot`
        int slot = -1;
        bool ok = true;
        const uint64_t policy = weight_policy(S.pass);
        // waits for the next stage, announces `blocks` blocks for it and returns its address
        auto next_stage = [&](int blocks) -> uint32_t {
            if (++slot == S.stages) slot = 0;
            if (slot == 0) phase ^= 1u;
            if (it >= (uint32_t)S.stages) ok = ok && d2d_tc::mbar_wait_warp(smem_addr(&bar_empty[slot]), phase ^ 1u, P.status);
            if (ok && lane == 0) d2d_tc::mbar_expect_tx(smem_addr(&bar_full[slot]), (uint32_t)(blocks * SUB_BYTES));
            ++it;
            return smem_addr(ring + (size_t)slot * STAGE_BYTES);
        };
        auto full_bar = [&]() { return smem_addr(&bar_full[slot]); };
        auto up = [&](int r, int n) {
            if (rank >= slots(r, n)) return;
            const int u = unit_of(r, rank, unit_list_p);
            for (int q = 0; q < nq && ok; ++q)
                for (int m = 0; m < n_mat && ok; ++m) {
                    const uint32_t dst = next_stage(S.up_blocks);
                    if (ok && lane == 0) tma_load_3d(dst, m ? &P.tm_wg : &P.tm_w1, u * 16, q * STAGE_BLOCKS, full_bar(), policy);
                    __syncwarp();
                }
        };
        // the down stages of round r from number `from` on, while fewer than `limit` stages have been requested (0: all)
        auto down = [&](int r, int from, uint32_t limit, int n) -> int {
            int st = 0;
            const int nv = slots(r, n);
            for (int k0 = 0; k0 < nv; k0 += S.sps)
                for (int part = 0; part < PARTS; ++part, ++st) {
                    if (st < from) continue;
                    if ((limit > 0 && it >= limit) || !ok) return st;
                    const int k1 = min(nv, k0 + S.sps);
                    const uint32_t dst = next_stage((k1 - k0) * (PARTS > 1 ? STAGE_BLOCKS : S.nb));
                    if (ok && lane == 0)
                        for (int k = k0; k < k1; ++k)
                            tma_load_3d(dst + (k - k0) * S.nb * SUB_BYTES, &P.tm_w2t, unit_of(r, k, unit_list_p) * 16, rank * S.nb + part * STAGE_BLOCKS, full_bar(), policy);
                    __syncwarp();
                }
            return -1;
        };
        // Before anything is known about the selection: the up stages of the static rounds, which the consumers use up
        // before they wait for it, and of the down stages what the ring holds.
        for (int r = 0; r < my_static; ++r) up(r, 0);
        int r = 0, from = 0;
        const uint32_t early = it + (uint32_t)S.stages;
        for (; r < my_static; ++r) {
            from = down(r, 0, early, 0);
            if (from >= 0) break;
            from = 0;
        }
        int n = 0;
        if (P.units) {
            pdl_wait();
            n = __ldcg(P.units);
            load_list(unit_list_p, lane, 32);
            __syncwarp();
        } else {
            asm volatile("bar.sync 2, %0;" ::"n"(NC + 32) : "memory");           // the consumers have built unit_list
            n = n_units;
            for (int i = lane; i < MAX_LIST; i += 32) unit_list_p[i] = unit_list[i];
            __syncwarp();
        }
        const int R = rounds_for(n);
        for (int ru = my_static; r < R && ok; ) {
            if (up_next(ru, r, R)) {
                up(ru, n);
                ++ru;
            } else {
                down(r, from, 0, n);
                ++r;
                from = 0;
            }
        }
        // nothing may be in flight when the CTA exits: the consumers wait for every stage they use, so only a run that
        // gave up needs this
        if (!ok)
            for (uint32_t k = it > (uint32_t)S.stages ? it - S.stages : 0; k + 1 < it; ++k)
                d2d_tc::mbar_wait_warp(smem_addr(&bar_full[k % S.stages]), (k / S.stages) & 1u, P.status);
        cluster_arrive();
    } else if (warp > NCW) {
        // ------------------------------------------------------------------ talks to the cluster: sends the hidden values, and tells
        // the others that a round's have been read.  A release at cluster scope takes 0.6 us, sending as much: a consumer warp would
        // hold up all others with it (Llama-shaped layer, tau = 0.2, us, with the sends by consumer warps / here: 37.7 / 35.4 at 1 token (163
        // experts kept) and 52.9 / 50.6 at 6, 8-bit weights; 59.4 / 56.7 at 7 tokens.  A warp for each other CTA: the same with clusters of two, and 43.7
        // instead of 40.9 at 1 token, where they are of four.)
        bool ok = d2d_tc::mbar_wait_warp(smem_addr(&bar_go), 0, P.status);
        __syncwarp();
        const uint32_t hs_addr = smem_addr(hs);
        const int nj = ok ? rounds_s - my_static : 0, n = n_s, q0 = my_static > 0 ? 1 : 0;
        for (int q = 0; ok && q < nj + q0; ++q) {
            const int j = q - q0;                              // number of the shared round, or -1: the static ones
            if (j >= 2) {                                      // the consumers have read the buffer's last contents: others may write it
                ok = d2d_tc::mbar_wait_warp(smem_addr(&h_read[j & 1]), ((j >> 1) & 1u) ^ 1u, P.status);
                __syncwarp();
                if (ok && lane < CL) arrive_cluster(cluster_addr(smem_addr(&h_empty[j & 1]), lane));
            }
            // two barriers in turn: the consumers are at most one round ahead, since a round's down projection waits for what is sent here
            ok = ok && d2d_tc::mbar_wait_warp(smem_addr(&h_done[q & 1]), (q >> 1) & 1u, P.status);
            __syncwarp();
            if (ok && j >= 2) ok = mbar_wait_cluster(smem_addr(&h_empty[j & 1]), ((j >> 1) & 1u) ^ 1u, P.status);
            __syncwarp();
            const uint32_t full = smem_addr(&h_full[j < 0 ? 2 : j & 1]);
            // 16-byte asynchronous stores, counted by the receiver's barrier (4-byte ones by the threads that have the values took 2.6
            // us, plain stores and an arrival that releases them 1.4); a piece goes to all others at once
            uint32_t to[3], bar[3], bytes = 0;
#pragma unroll
            for (int p = 0; p < 3; ++p) {
                to[p] = cluster_addr(hs_addr, (rank + 1 + p) % CL);
                bar[p] = cluster_addr(full, (rank + 1 + p) % CL);
            }
            for (int r = j < 0 ? 0 : my_static + j; r < (j < 0 ? my_static : my_static + j + 1); ++r) {
                if (rank >= slots(r, n)) break;
                bytes += 32u * (uint32_t)(NT8 == 1 ? T8 * S.planes : T);
                const uint32_t own = (uint32_t)(buffer(r) - hs) + (uint32_t)rank * S.planes * T8 * H_ROW;
                for (int i = lane; i < 2 * T8 * S.planes; i += 32) {
                    const uint32_t off = own + (i >> 1) * H_ROW + (i & 1) * 16;
                    if (NT8 > 1 && (i >> 1) >= T) break;
                    const uint4 v = lds16(hs_addr + off);
#pragma unroll
                    for (int p = 0; p < 3; ++p)
                        if (p + 1 < CL) st_async4(to[p] + off, v, bar[p]);
                }
            }
#pragma unroll
            for (int p = 0; p < 3; ++p)
                if (p + 1 < CL && lane == 0) arrive_cluster(bar[p], bytes);
            // only now the CTA's own consumers: what they wait for here lets them write this slot again, two rounds on
            __syncwarp();
            if (lane == 0) d2d_tc::mbar_arrive(full);
        }
        cluster_arrive();
    } else {
        // ------------------------------------------------------------------ consumers
        // x does not depend on the router (the kernel behind which this one may start early waits for its own
        // predecessor before it lets this one start)
        if (!Q8) {
            for (int i = tid, t = 0; t < T; ) {
                if (i >= d / 8) { i -= d / 8; ++t; continue; }
                cp_async16(smem_addr(xs + (size_t)t * xp + i * 16), x + (size_t)t * d + i * 8);
                i += NC;
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
            asm volatile("cp.async.wait_group 0;" ::: "memory");
            consumer_bar();
        } else {
            // Codes widen to float16 in one instruction, to bfloat16 in four, so beside codes the rows become float16 where that loses
            // nothing: scaled so that a row's largest value lies in [2^14, 2^15), float16 has all eight bits of a value down to 2^-17,
            // that is of one whose exponent is at most 31 below the largest.  A batch with a non-zero value further below stays
            // bfloat16: its rows are fetched again.
            // wpt warps a token, a piece of the row each; a lane looks at what it fetched itself
            const int wpt = T <= 1 ? 16 : T <= 2 ? 8 : T <= 4 ? 4 : T <= 8 ? 2 : 1, part = warp % wpt, np = d / 8;
            const int i0 = np * part / wpt, i1 = np * (part + 1) / wpt;
            auto fetch = [&](bool placed) {
                for (int t = warp / wpt; t < T; t += NCW / wpt)
                    for (int i = i0 + lane; i < i1; i += 32) {
                        const __nv_bfloat16 *src = x + (size_t)t * d + i * 8;
                        const uint32_t row = smem_addr(xs + (size_t)t * xp);
                        if (placed) {
                            cp_async8(row + x_place(2 * i), src);
                            cp_async8(row + x_place(2 * i + 1), src + 4);
                        } else {
                            cp_async16(row + i * 16, src);
                        }
                    }
                asm volatile("cp.async.commit_group;" ::: "memory");
                asm volatile("cp.async.wait_group 0;" ::: "memory");
            };
            // a lane's own eight columns, as they lie after a placed fetch
            auto own = [&](int t, int i, int h) { return reinterpret_cast<uint2 *>(xs + (size_t)t * xp + x_place(2 * i + h)); };
            if (tid == 0) x_spread = 0;
            fetch(true);
            for (int t = warp / wpt; t < T; t += NCW / wpt) {
                uint32_t m = 0u;
                for (int i = i0 + lane; i < i1; i += 32) {
                    const uint2 a = *own(t, i, 0), b = *own(t, i, 1);
                    const uint32_t w[4] = {a.x, a.y, b.x, b.y};
#pragma unroll
                    for (int q = 0; q < 4; ++q) m = max(m, max(w[q] & 0x7fffu, (w[q] >> 16) & 0x7fffu));
                }
                m = __reduce_max_sync(FULL, m);
                if (lane == 0) x_max[t * 16 + part] = m;
            }
            consumer_bar();
            bool spread = false;
            for (int t = warp / wpt; t < T; t += NCW / wpt) {
                uint32_t m = 0u;
                for (int q = 0; q < wpt; ++q) m = max(m, x_max[t * 16 + q]);
                const int sh = min(120, 141 - (int)(m >> 7));
                const float f = __uint_as_float((uint32_t)(127 + sh) << 23);
                // the smallest magnitude that fits, less one: magnitudes less one are compared, so that zeros fit
                const uint32_t least = (uint32_t)max(((int)(m >> 7) - 31) * 128 - 1, 0);
                if (lane == 0 && part == 0) x_inv[t] = __uint_as_float((uint32_t)(127 - sh) << 23);
                for (int i = i0 + lane; i < i1; i += 32) {
                    const uint2 a = *own(t, i, 0), b = *own(t, i, 1);
                    const uint32_t w[4] = {a.x, a.y, b.x, b.y};
                    uint32_t o[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        spread |= ((w[q] & 0x7fffu) - 1u < least) | (((w[q] >> 16) & 0x7fffu) - 1u < least);
                        const float lo = __uint_as_float(w[q] << 16) * f, hi = __uint_as_float(w[q] & 0xffff0000u) * f;
                        asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(o[q]) : "f"(hi), "f"(lo));
                    }
                    *own(t, i, 0) = make_uint2(o[0], o[1]);
                    *own(t, i, 1) = make_uint2(o[2], o[3]);
                }
            }
            if (spread) x_spread = 1;
            consumer_bar();
            if (__builtin_expect(*(volatile int *)&x_spread != 0, 0)) {
                if (tid < T) x_inv[tid] = 1.0f;
                fetch(false);
                consumer_bar();
            }
        }

        int slot = 0, n = 0;
        uint32_t phase = 0;
        bool ok = true;
        auto stage_wait = [&]() {
            if (ok) ok = d2d_tc::mbar_wait_warp(smem_addr(&bar_full[slot]), phase, P.status);
        };
        auto stage_done = [&]() {
            __syncwarp();
            if (lane == 0) d2d_tc::mbar_arrive(smem_addr(&bar_empty[slot]));
            if (++slot == S.stages) { slot = 0; phase ^= 1u; }
        };
        // this thread's hidden value in a round: neuron nr of its unit, token tok
        const int nr = tid / T8, tok = tid % T8;
        const bool mine = tid < 16 * T8 && tok < T;
        // ldmatrix addresses: row of this lane inside a 16-row operand tile, and which 16-byte piece of a pair
        const int lrow = (lane & 7) + ((lane >> 3) & 1) * 8, lhalf = lane >> 4;
        const uint32_t xs_addr = smem_addr(xs);

        // ---- up projection (and gate) of this CTA's unit of round r; the sums, bias added, go to this thread's places in
        // zs[place].  A warp takes one 128-byte column block.
        auto up = [&](int r, int place) {
            if (rank >= slots(r, n)) return;
            const int u = unit_of(r, rank, unit_list);
            float bias = 0.0f;
            int sc[3] = {0, 0, 0};                                // exponents of the scales of W1, W_gate and W2
            if (mine) {
                if (P.b1) bias = __bfloat162float(P.b1[u * 16 + nr]);
                if (Q8) {
                    const int e = expert_of(S, u * 16 + nr);
                    sc[0] = P.k1[e]; sc[2] = P.k2[e];
                    if (S.gated) sc[1] = P.kg[e];
                }
            }
            constexpr int CH = NT8 == 1 ? 2 : 1;                  // chains of matrix instructions per accumulator
            float s[2][NT8 * CH][4];
#pragma unroll
            for (int m = 0; m < 2; ++m)
#pragma unroll
                for (int t = 0; t < NT8 * CH; ++t) s[m][t][0] = s[m][t][1] = s[m][t][2] = s[m][t][3] = 0.0f;
            const bool spread = Q8 && *(volatile int *)&x_spread != 0;        // (read here: a register less)
            if (Q8 && __builtin_expect(spread, 0)) {
                const up_rows a = {smem_addr(bar_full), smem_addr(bar_empty), smem_addr(ring), smem_addr(xs), xp, T, d,
                                   nq, n_mat, S.stages, warp, slot, phase, ok ? P.status : nullptr};
                const up_sums<NT8, CH> o = TPW * NT8 <= 4 ? up_spread_rows_call<NT8, CH>(a) : up_spread_rows<NT8, CH>(a);
#pragma unroll
                for (int m = 0; m < 2; ++m)
#pragma unroll
                    for (int t = 0; t < NT8 * CH; ++t)
#pragma unroll
                        for (int i = 0; i < 4; ++i) s[m][t][i] = o.v[m][t][i];
                slot = o.slot; phase = o.phase; ok = ok && o.ok;
            }
#pragma unroll 1
            for (int q = spread ? nq : 0; q < nq; ++q) {
                const int k0 = q * SEG + warp * SUB;
#pragma unroll
                for (int m = 0; m < 2; ++m) {
                    if (m == 1 && !S.gated) break;
                    stage_wait();
                    if (k0 < d) {                                 // warp-uniform: d is a multiple of a block's columns
                        unsigned char *st = ring + (size_t)slot * STAGE_BYTES + warp * SUB_BYTES;
                        if (!Q8) {
                            const uint32_t sa = smem_addr(st);
#pragma unroll
                            for (int h = 0; h < 2; ++h) {                     // 32 columns at a time
                                uint32_t a0[4], a1[4];
                                ldmatrix4<false>(a0, sa + swz(lrow, h * 64 + lhalf * 16));
                                ldmatrix4<false>(a1, sa + swz(lrow, h * 64 + 32 + lhalf * 16));
#pragma unroll
                                for (int t = 0; t < NT8; ++t) {
                                    uint32_t b[4];
                                    ldmatrix4<false>(b, xs_addr + min(t * 8 + (lane & 7), T - 1) * xp + (k0 + h * 32) * 2 + (lane >> 3) * 16);
                                    mma16816(s[m][t * CH], a0[0], a0[1], a0[2], a0[3], b[0], b[1]);
                                    mma16816(s[m][t * CH + CH - 1], a1[0], a1[1], a1[2], a1[3], b[2], b[3]);
                                }
                            }
                        } else {
                            // Two 16-code pieces of all rows at a time: lane (g, c) gets codes 4 c .. 4 c + 3 of rows g and g + 8 of each, that
                            // is a matrix instruction's operand but for the order of its 16 columns, which the token rows share.  (Plain
                            // 16-byte loads, half of them exchanged between registers so that they do not meet in a bank, and
                            // addresses worked out load by load here and in the down projection kept the ALU pipe busy for 58 % of the
                            // kernel, where the loops were bound by it: Llama-shaped layer, tau = 0.2, 41.8 -> 37.4 us at 1 token, 55.8 ->
                            // 49.7 at 2, 60.0 -> 52.9 at 6.)
                            const uint32_t sa = smem_addr(st) + lrow * 128 + ((lhalf ^ (lrow & 7)) << 4);
#pragma unroll
                            for (int h = 0; h < 4; ++h) {
                                uint32_t q[4], w[8];
                                ldmatrix4<false>(q, sa ^ (uint32_t)(h * 32));
                                widen16(make_uint4(q[0], q[1], q[2], q[3]), w);
#pragma unroll
                                for (int t = 0; t < NT8; ++t) {
                                    const uint4 xb = lds16(xs_addr + min(t * 8 + g, T - 1) * xp + (k0 + h * 32) * 2 + c * 16);
                                    mma16816_f16(s[m][t * CH], w[0], w[2], w[1], w[3], xb.x, xb.y);
                                    mma16816_f16(s[m][t * CH + CH - 1], w[4], w[6], w[5], w[7], xb.z, xb.w);
                                }
                            }
                        }
                    }
                    stage_done();
                }
            }
            // the warps' partial sums meet
            consumer_bar();                                       // the sums of the previous round have been read
#pragma unroll
            for (int m = 0; m < 2; ++m) {
                if (m == 1 && !S.gated) break;
#pragma unroll
                for (int t = 0; t < NT8; ++t) {
                    if (CH == 2) {
#pragma unroll
                        for (int i = 0; i < 4; ++i) s[m][0][i] += s[m][CH - 1][i];
                    }
                    float *r = red + (size_t)((m * NCW + warp) * 16 + g) * T8 + t * 8 + 2 * c;
                    *reinterpret_cast<float2 *>(r) = make_float2(s[m][t * CH][0], s[m][t * CH][1]);
                    *reinterpret_cast<float2 *>(r + 8 * T8) = make_float2(s[m][t * CH][2], s[m][t * CH][3]);
                }
            }
            consumer_bar();
            if (mine) {
                float *z = zs + (size_t)place * 3 * 16 * T8 + tid;
                float v[2] = {0.0f, 0.0f};
                // (codes: scales only when both sums are there, and without ldexpf: 34.5 instead of 35.6 us for the Llama-shaped layer at 1
                // token that keeps 163 experts, 45.7 instead of 47.1 at 2, tau = 0.2)
#pragma unroll
                for (int m = 0; m < 2; ++m) {
                    if (m == 1 && !S.gated) break;
                    const float *p = red + (size_t)m * NCW * 16 * T8 + tid;
#pragma unroll
                    for (int w = 0; w < NCW; ++w) v[m] += p[w * 16 * T8];
                    if (!Q8) z[m * 16 * T8] = m == 0 ? v[m] + bias : v[m];
                }
                if (Q8) {
                    z[0] = times_pow2(v[0] * x_inv[tok], sc[0]) + bias;
                    if (S.gated) z[16 * T8] = times_pow2(v[1] * x_inv[tok], sc[1]);
                    z[2 * 16 * T8] = times_pow2(1.0f, sc[2]);
                }
            }
        };

        // Waits for the router and brings mask and list of kept units into shared memory (the list is found here, from the
        // mask, where the router does not make it).
        auto mask_ready = [&]() {
            pdl_wait();
            if (P.units) {
                load_list(unit_list, tid, NC);
                n = __ldcg(P.units);
            }
            for (int i = tid; i < T * S.W; i += NC) smask[i] = __ldcg(P.mask + i);
            consumer_bar();
            if (P.units) return;
            const int u0 = min(S.n_static * NCL * CL, U), nu = U - u0;
            if (nu > 0) {
                uint32_t *un = smask + T * S.W;
                for (int w = tid; w < S.W; w += NC) {
                    uint32_t v = 0u;
                    for (int t = 0; t < T; ++t) v |= smask[t * S.W + w];
                    un[w] = v;
                }
                consumer_bar();
                const int nw = (nu + 31) / 32;
                for (int w = warp; w < nw; w += NCW) {
                    const int u = u0 + w * 32 + lane;
                    bool keep = false;
                    if (u < U)
                        for (int e = u * 16 / S.s; e <= (u * 16 + 15) / S.s; ++e) keep |= (un[e >> 5] >> (e & 31)) & 1u;
                    const uint32_t bits = __ballot_sync(FULL, keep);
                    if (lane == 0) keep_bits[w] = bits;
                }
                consumer_bar();
                if (warp == 0) {
                    int run = 0;
                    for (int w0 = 0; w0 < nw; w0 += 32) {
                        const int v = w0 + lane < nw ? __popc(keep_bits[w0 + lane]) : 0;
                        int inc = v;
#pragma unroll
                        for (int o = 1; o < 32; o <<= 1) {
                            const int m = __shfl_up_sync(FULL, inc, o);
                            if (lane >= o) inc += m;
                        }
                        if (w0 + lane < nw) keep_pre[w0 + lane] = run + inc - v;
                        run += __shfl_sync(FULL, inc, 31);
                    }
                    if (lane == 0) n_units = run;
                }
                consumer_bar();
                for (int i = tid; i < nu; i += NC)
                    if ((keep_bits[i >> 5] >> (i & 31)) & 1u) {
                        const int r = keep_pre[i >> 5] + __popc(keep_bits[i >> 5] & ((1u << (i & 31)) - 1u)), j = r / CL;
                        if (j % NCL == cid) unit_list[j / NCL * CL + r % CL] = u0 + i;
                    }
            } else if (tid == 0) {
                n_units = 0;
            }
            asm volatile("bar.sync 2, %0;" ::"n"(NC + 32) : "memory");
            n = n_units;
        };

        // ---- hidden values of rounds [r0, r1): activation and selection on this CTA's sums into its own buffers
        auto finish = [&](int r0, int r1) {
            const int j = r0 - my_static;                                      // shared rounds: their number
            for (int r = r0; r < r1; ++r) {
                if (rank >= slots(r, n) || !mine) continue;
                const int e = expert_of(S, unit_of(r, rank, unit_list) * 16 + nr);
                const float *z = zs + (size_t)min(r, my_static) * 3 * 16 * T8 + tid;
                const float up = z[0], pre = S.gated ? z[16 * T8] : up;
                float h = 0.0f;
                if ((smask[tok * S.W + (e >> 5)] >> (e & 31)) & 1u) {
                    h = S.planes == 3 ? act_accurate(S.act, pre) : act_fast(S.act, pre);
                    if (S.gated) h *= up;
                }
                // the scale of W2 is a power of two: applied to the hidden value, after its rounding
                __nv_bfloat16 *o = reinterpret_cast<__nv_bfloat16 *>(buffer(r) + (size_t)(rank * S.planes * T8 + tok) * H_ROW) + nr;
                if (S.planes == 3) {
                    __nv_bfloat16 t[3];
                    split3(Q8 ? h * z[2 * 16 * T8] : h, t);
                    o[0] = t[0]; o[T8 * H_ROW / 2] = t[1]; o[2 * T8 * H_ROW / 2] = t[2];
                } else {
                    const __nv_bfloat16 hb = __float2bfloat16_rn(h);
                    o[0] = Q8 ? __float2bfloat16_rn(__bfloat162float(hb) * z[2 * 16 * T8]) : hb;
                }
            }
            if (CL > 1) {
                const int q = j < 0 ? 0 : j + (my_static > 0 ? 1 : 0);
                __syncwarp();
                if (lane == 0) d2d_tc::mbar_arrive(smem_addr(&h_done[q & 1]));
            } else {
                consumer_bar();
            }
        };
        // (A CTA's own slot of a shared round's buffer is written again two rounds later.  The consumers have read it by then: the
        // barriers of that round's up projection come behind their down projection.  So has the warp that sends it, which takes no
        // part in those: that down projection waits for its arrival at h_full, and it arrives when it has read the slot.)

        // ---- down projection of round r onto this CTA's columns.  A tile's 16 columns: bf16 weights g and g + 8 of lane (g, c);
        // codes 4 g and 4 g + 1 of a 32-column pair of tiles, 4 g + 2 and 4 g + 3 in its second tile.
        float acc[ACC][NT8][4];
#pragma unroll
        for (int i = 0; i < ACC; ++i)
#pragma unroll
            for (int t = 0; t < NT8; ++t) acc[i][t][0] = acc[i][t][1] = acc[i][t][2] = acc[i][t][3] = 0.0f;
        const int DC = d / CL;
        // codes: where neurons 2 c and 2 c + 1 of the lane's four columns lie in a unit's rows
        const uint32_t dn0 = (uint32_t)(warp / (SUB / 32) * SUB_BYTES) + swz(2 * c, warp % (SUB / 32) * 32 + g * 4),
                       dn1 = (uint32_t)(warp / (SUB / 32) * SUB_BYTES) + swz(2 * c + 1, warp % (SUB / 32) * 32 + g * 4);
        auto down = [&](int r, int R) {
            const int j = r - my_static, nv = slots(r, n);
            if (ok && CL > 1) ok = mbar_wait_cluster(smem_addr(&h_full[j < 0 ? 2 : j & 1]), j < 0 ? 0u : (j >> 1) & 1u, P.status);
            const unsigned char *hb0 = buffer(r) + g * H_ROW + c * 4;
            for (int k0 = 0; k0 < nv; k0 += S.sps) {
                const int k1 = min(nv, k0 + S.sps);
#pragma unroll
                for (int part = 0; part < PARTS; ++part) {
                    stage_wait();
                    unsigned char *stage = ring + (size_t)slot * STAGE_BYTES;
#pragma unroll(NT8 == 1 || PARTS > 1 ? 1 : 4)
                    for (int k = k0; k < k1; ++k) {
                        uint32_t hb[3][NT8][2];
#pragma unroll
                        for (int p = 0; p < 3; ++p)
#pragma unroll
                            for (int t = 0; t < NT8; ++t) {
                                if (p > 0 && (NT8 > 1 || S.planes == 1)) break;
                                const unsigned char *hr = hb0 + ((k * S.planes + p) * T8 + t * 8) * H_ROW;
                                hb[p][t][0] = *reinterpret_cast<const uint32_t *>(hr);
                                hb[p][t][1] = *reinterpret_cast<const uint32_t *>(hr + 16);
                            }
                        auto products = [&](float (&o)[NT8][4], const uint32_t (&a)[4]) {
#pragma unroll
                            for (int t = 0; t < NT8; ++t) mma16816(o[t], a[0], a[1], a[2], a[3], hb[0][t][0], hb[0][t][1]);
                            if (NT8 == 1 && S.planes == 3) {
                                mma16816(o[0], a[0], a[1], a[2], a[3], hb[1][0][0], hb[1][0][1]);
                                mma16816(o[0], a[0], a[1], a[2], a[3], hb[2][0][0], hb[2][0][1]);
                            }
                        };
                        const unsigned char *piece = stage + (k - k0) * S.nb * SUB_BYTES;
                        if (!Q8) {
#pragma unroll
                            for (int i = 0; i < TPP; ++i) {
                                const int tile = warp + NCW * i;
                                if (PARTS == 1 && tile * 16 >= DC) break;
                                // matrices: neurons 0-7 and 8-15 (lane / 16), columns 0-7 and 8-15 (lane / 8 % 2)
                                uint32_t a[4];
                                ldmatrix4<true>(a, smem_addr(piece + tile * 16 / SUB * SUB_BYTES) +
                                                       swz((lane & 7) + lhalf * 8, tile * 16 % SUB * 2 + ((lane >> 3) & 1) * 16));
                                products(acc[part * TPP + i], a);
                            }
                        } else {
#pragma unroll
                            for (int i = 0; i < (TPP + 1) / 2; ++i) {
                                const int pair = warp + NCW * i;
                                if (PARTS == 1 && pair * 32 >= DC) break;
                                uint32_t r[4];                    // neurons 2c, 2c + 1, 2c + 8, 2c + 9: four columns each
#pragma unroll
                                for (int q = 0; q < 4; ++q)
                                    r[q] = *reinterpret_cast<const uint32_t *>(piece + ((q & 1) ? dn1 : dn0) + (i * NCW * 32 / SUB * SUB_BYTES + (q >> 1) * 1024));
                                const uint32_t a0[4] = {pair_of<0>(r[0], r[1]), pair_of<1>(r[0], r[1]), pair_of<0>(r[2], r[3]), pair_of<1>(r[2], r[3])};
                                const uint32_t a1[4] = {pair_of<2>(r[0], r[1]), pair_of<3>(r[0], r[1]), pair_of<2>(r[2], r[3]), pair_of<3>(r[2], r[3])};
                                products(acc[part * TPP + 2 * i], a0);
                                products(acc[part * TPP + 2 * i + 1], a1);
                            }
                        }
                    }
                    stage_done();
                }
            }
            // the buffer's next use is the shared round after the next
            if (CL > 1 && j >= 0 && r + 2 < R && lane == 0) d2d_tc::mbar_arrive(smem_addr(&h_read[j & 1]));
        };

        // Order of work: the up projections of the static rounds; then, with the selection there, hidden values one round
        // ahead of the down projections.  The up projection of the first shared round waits until the static rounds are
        // done: their down stages can then be requested before the list is known.
        int R = 0;
        bool ready = false;
        for (int ru = 0, rf = 0, rd = 0;;) {                                   // next round's up / finish / down
            if (!ready && ru == my_static) {
                mask_ready();
                ready = true;
                R = rounds_for(n);
                if (tid == 0) {
                    n_s = n;
                    rounds_s = R;
                    d2d_tc::mbar_arrive(smem_addr(&bar_go));
                }
            }
            if (ready && rd == R) break;
            if (!ready || (rf == ru && up_next(ru, rd, R))) {
                up(ru, min(ru, my_static));
                ++ru;
            } else if (rf < ru && rf <= rd + 1) {
                const int to = rf < my_static ? my_static : rf + 1;
                finish(rf, to);
                rf = to;
            } else {
                down(rd, R);
                ++rd;
            }
        }
        cluster_arrive();                                                      // this CTA sends nothing to the others any more
        // ---- this CTA's sums.  Codes: a lane has four adjacent columns of two tokens; bf16: four lanes (g of a group of four)
        // exchange their four values each, so that every lane has four adjacent columns of one token: 16 bytes per reduction.
        if (R > 0) {
            if (Q8) {
#pragma unroll
                for (int i = 0; i < ACC / 2; ++i) {
                    constexpr int PAIRS = (TPP + 1) / 2;                       // of a stage
                    const int col = (i / PAIRS) * STAGE_BLOCKS * SUB + ((i % PAIRS) * NCW + warp) * 32 + g * 4;
#pragma unroll
                    for (int t = 0; t < NT8; ++t) {
                        const float(&v)[4] = acc[2 * i][t], (&w)[4] = acc[2 * i + 1][t];
                        const int tk = t * 8 + 2 * c;
                        float *o = P.y32 + (size_t)tk * d + rank * DC + col;
                        if (tk < T && col < DC) red_add4(o, make_float4(v[0], v[2], w[0], w[2]));
                        if (tk + 1 < T && col < DC) red_add4(o + d, make_float4(v[1], v[3], w[1], w[3]));
                    }
                }
            } else {
#pragma unroll
                for (int i = 0; i < TPW; ++i) {
                    const int tile = (i % TPP) * NCW + warp, col0 = (i / TPP) * STAGE_BLOCKS * SUB + tile * 16;
#pragma unroll
                    for (int t = 0; t < NT8; ++t) {
                        const float(&v)[4] = acc[i][t];
                        const bool o1 = g & 1, o2 = g & 2;
                        // 4 x 4 transpose over the lanes: value j of all four goes to lane j of the group
                        const float x0 = __shfl_xor_sync(FULL, o1 ? v[0] : v[1], 4), x1 = __shfl_xor_sync(FULL, o1 ? v[2] : v[3], 4);
                        const float a0 = o1 ? x0 : v[0], a1 = o1 ? v[1] : x0, b0 = o1 ? x1 : v[2], b1 = o1 ? v[3] : x1;   // (a0, a1): value o1, (b0, b1): value 2 + o1 of the lane pair
                        const float y0 = __shfl_xor_sync(FULL, o2 ? a0 : b0, 8), y1 = __shfl_xor_sync(FULL, o2 ? a1 : b1, 8);
                        const float4 o = o2 ? make_float4(y0, y1, b0, b1) : make_float4(a0, a1, y0, y1);
                        const int tk = t * 8 + 2 * c + (o1 ? 1 : 0), col = (o2 ? 8 : 0) + (g & 4);
                        if (tk < T && col0 + col < DC) red_add4(P.y32 + (size_t)tk * d + rank * DC + col0 + col, o);
                    }
                }
            }
        }
        // ---- the CTA that is last to add to these columns finishes them: + b2, bf16
        consumer_bar();
        if (tid == 0) {
            // releases the whole CTA's additions (the barrier before it) and acquires everybody's: one round trip, where two fences
            // around the addition made three
            asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;" : "=r"(my_ticket) : "l"(P.ticket + rank) : "memory");
            if (my_ticket == (unsigned)NCL - 1) P.ticket[rank] = 0u;
        }
        consumer_bar();
        const int per_row = my_ticket == (unsigned)NCL - 1 ? DC / 4 : 0;
#pragma unroll 4
        for (int i = tid; i < T * per_row; i += NC) {
            const int t = i / per_row, col = rank * DC + (i - t * per_row) * 4;
            const float4 v = __ldcg(reinterpret_cast<const float4 *>(P.y32 + (size_t)t * d + col));
            float bb[4] = {0.f, 0.f, 0.f, 0.f};
            if (P.b2) {
                const uint2 q = __ldg(reinterpret_cast<const uint2 *>(P.b2 + col));
                bb[0] = __uint_as_float(q.x << 16); bb[1] = __uint_as_float(q.x & 0xffff0000u);
                bb[2] = __uint_as_float(q.y << 16); bb[3] = __uint_as_float(q.y & 0xffff0000u);
            }
            const __nv_bfloat162 lo = __floats2bfloat162_rn(v.x + bb[0], v.y + bb[1]), hi = __floats2bfloat162_rn(v.z + bb[2], v.w + bb[3]);
            *reinterpret_cast<uint2 *>(P.y + (size_t)t * d + col) = make_uint2(*reinterpret_cast<const uint32_t *>(&lo), *reinterpret_cast<const uint32_t *>(&hi));
        }
    }
    cluster_wait();                                                            // nobody leaves while another CTA may still send to it
}

constexpr size_t kSmemLimit = 218 * 1024;

int nt8_for(int T) { return T <= 8 ? 1 : T <= 16 ? 2 : 4; }

// Shared memory beside the ring, with `rows` rows of x
template <typename WT> size_t fixed_smem(const FfnShape &S, size_t rows)
{
    const size_t t8 = 8 * (size_t)nt8_for(S.T);
    return 1024 + rows * x_pitch(S.d) + (size_t)(S.gated ? 2 : 1) * NCW * 16 * t8 * 4 + (size_t)(S.n_static + 1) * 3 * 16 * t8 * 4 +
           (size_t)(S.n_static + 2) * S.cl * S.planes * t8 * H_ROW + (size_t)(S.T + 1) * S.W * 4;
}

// Output tiles per warp for clusters of cl CTAs; 0: the shape cannot be cut that way.  A unit's rows of W2T are cut into
// cl pieces of whole 128-byte blocks, several pieces to a stage or whole stages to a piece, and 16 x 8-token tiles of
// output accumulators take at most 32 registers.
template <typename WT> int tiles_per_warp(int d, int cl, int T)
{
    const int blocks = d / sub_cols<WT>();
    if (d % sub_cols<WT>() || blocks % cl) return 0;
    const int nb = blocks / cl, n = d2d_cdiv(d / cl, NCW * 16), tpw = n <= 1 ? 1 : n <= 2 ? 2 : n <= 4 ? 4 : n <= 8 ? 8 : 0;
    if (nb > STAGE_BLOCKS && nb != STAGE_BLOCKS * (tpw / (sub_cols<WT>() / 16))) return 0;
    return tpw * nt8_for(T) <= 8 ? tpw : 0;
}

// Fills in the launch parameters for n layers; false: no cluster size fits the shape.
template <typename WT> bool plan(FfnShape &S, int n_layers)
{
    const int U = S.d_ff / 16, sms = d2d_tc_sm_count();
    int best = 0;
    // Fewest rounds first (the rounds stream the weights), then the larger cluster (fewer sums to merge).  Clusters of four
    // reach 132 of 148 SMs, smaller ones all of them.  The smallest batches, which keep a fraction of the experts, do not run all
    // rounds: there the larger cluster wins unless it would make a quarter more of them (Llama-shaped layer, clusters of two / four:
    // 45.6 / 43.6 us at 1 token, 43.9 / 42.0 with 8-bit weights; 60.5 / 62.6 at 7 tokens, 55.2 / 61.0 at 4 with 8-bit weights).  One or two rows of sums are cheaper to merge than hidden values to
    // exchange (1.2 us).
    for (int cl = S.T * S.d <= 2048 && tiles_per_warp<WT>(S.d, 1, S.T) ? 1 : 4; cl >= 1; cl /= 2) {
        const int clusters = (cl == 4 ? sms * 33 / 37 : sms) / n_layers / cl;
        if (clusters < 1 || tiles_per_warp<WT>(S.d, cl, S.T) == 0) continue;
        const int rounds = d2d_cdiv(d2d_cdiv(U, cl), clusters);
        // A cluster's list of kept units holds up to cl entries a round.  One layer never needs more than 128; several large
        // ones, which share the clusters, can (four of d_ff = 17408 in clusters of four: 34 rounds).
        if (rounds * cl > MAX_LIST) continue;
        if (best == 0 || (S.planes == 3 ? rounds * 5 < best * 4 : rounds < best)) {
            best = rounds;
            S.cl = cl;
            S.clusters = d2d_cdiv(d2d_cdiv(U, cl), rounds);
        }
    }
    if (best == 0) return false;
    const int blocks = S.d / sub_cols<WT>();
    S.up_blocks = blocks < STAGE_BLOCKS ? blocks : STAGE_BLOCKS;
    S.pass = (double)n_layers * (S.gated ? 3.0 : 2.0) * S.d_ff * S.d * sizeof(WT) > 64e6;       // half of L2
    S.nb = blocks / S.cl;
    S.sps = S.nb >= STAGE_BLOCKS ? 1 : STAGE_BLOCKS / S.nb < S.cl ? STAGE_BLOCKS / S.nb : S.cl;
    // Rounds a cluster starts on before the selection is known: what the ring holds beside the up stages, which are used up
    // by then.  None for the smallest batches, which keep a fraction of the experts: most of what would be fetched early
    // would be thrown away.
    const int per_up = d2d_cdiv(S.d, seg_cols<WT>()) * (S.gated ? 2 : 1), per_down = d2d_cdiv(S.d, seg_cols<WT>());
    const int most = nt8_for(S.T) > 2 ? 2 : 4;
    S.n_static = most;                                       // (the largest, while the ring is sized)
    // A batch is taken if its whole token block fits beside three stages; the ring then also gets the room of the rows it lacks.
    const auto stages_with = [&](size_t rows) {
        const size_t f = fixed_smem<WT>(S, rows);
        return f >= kSmemLimit ? 0 : (int)((kSmemLimit - f) / STAGE_BYTES);
    };
    if (stages_with(8 * (size_t)nt8_for(S.T)) < 3) return false;
    S.stages = stages_with((size_t)S.T);
    if (S.stages > MAX_STAGES) S.stages = MAX_STAGES;
    const int fit = (S.stages + per_up) / (per_up + per_down);
    S.n_static = S.planes == 3 ? 0 : fit < 1 ? 1 : fit < most ? fit : most;
    return true;
}

FfnShape shape_for(const d2d_layer_desc &D, int T)
{
    FfnShape S = {};
    S.T = T; S.d = D.d; S.d_ff = D.d_ff; S.E = D.n_experts; S.s = D.expert_size; S.inv_s = (uint32_t)((0x100000000ull + D.expert_size - 1) / D.expert_size);      // (0 for s = 1: not used)
    S.W = (D.n_experts + 31) / 32;
    S.act = D.act; S.gated = D.gated ? 1 : 0;
    S.planes = T <= d2d_decode_max_tokens(D) ? 3 : 1;
    return S;
}

template <typename WT, int TPW, int NT8>
d2d_status launch(const FfnShape &S, int n_layers, const d2d_decode_ffn_args &a, const void *x, bool after_router, cudaStream_t st)
{
    auto kern = decode_ffn_kernel<WT, TPW, NT8>;
    static bool attr_set[64] = {};                          // the attribute is per device
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return D2D_ERR_CUDA;
    if (!__atomic_load_n(&attr_set[dev], __ATOMIC_ACQUIRE)) {
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemLimit) != cudaSuccess) return D2D_ERR_CUDA;
        __atomic_store_n(&attr_set[dev], true, __ATOMIC_RELEASE);
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(S.clusters * S.cl, n_layers, 1);
    cfg.blockDim = dim3(S.cl > 1 ? NT : NT - 32, 1, 1);        // clusters of one have nobody to talk to
    cfg.dynamicSmemBytes = fixed_smem<WT>(S, (size_t)S.T) + (size_t)S.stages * STAGE_BYTES;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = S.cl; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = after_router && d2d_tc_pdl_enabled() ? 2 : 1;
    const cudaError_t err = cudaLaunchKernelEx(&cfg, kern, (const __nv_bfloat16 *)x, S, a);
    D2D_LAUNCHED(1);
    return err == cudaSuccess ? D2D_OK : D2D_ERR_CUDA;
}

template <typename WT>
d2d_status dispatch(FfnShape S, int n, const d2d_decode_ffn_args &a, const void *x, bool after, cudaStream_t st)
{
    if (!plan<WT>(S, n)) return D2D_ERR_UNSUPPORTED;
    d2d_decode_ffn_args b = a;
    for (int l = 0; l < n; ++l) b.l[l].tm_w2t = a.l[l].tm_w2t_cl[S.cl == 4 ? 2 : S.cl == 2 ? 1 : 0];
    const int tpw = tiles_per_warp<WT>(S.d, S.cl, S.T), nt = nt8_for(S.T);
    switch (tpw * 10 + nt) {
    case 11: return launch<WT, 1, 1>(S, n, b, x, after, st);
    case 12: return launch<WT, 1, 2>(S, n, b, x, after, st);
    case 14: return launch<WT, 1, 4>(S, n, b, x, after, st);
    case 21: return launch<WT, 2, 1>(S, n, b, x, after, st);
    case 22: return launch<WT, 2, 2>(S, n, b, x, after, st);
    case 24: return launch<WT, 2, 4>(S, n, b, x, after, st);
    case 41: return launch<WT, 4, 1>(S, n, b, x, after, st);
    case 42: return launch<WT, 4, 2>(S, n, b, x, after, st);
    case 81: return launch<WT, 8, 1>(S, n, b, x, after, st);
    }
    return D2D_ERR_UNSUPPORTED;
}

template <typename WT> bool make_map(CUtensorMap *m, const void *w, int rows, int d, int blocks)
{
    const cuuint64_t dims[3] = {(cuuint64_t)sub_cols<WT>(), (cuuint64_t)rows, (cuuint64_t)(d / sub_cols<WT>())};
    const cuuint64_t strides[2] = {(cuuint64_t)d * sizeof(WT), 128};
    const cuuint32_t box[3] = {(cuuint32_t)sub_cols<WT>(), 16, (cuuint32_t)(blocks < STAGE_BLOCKS ? blocks : STAGE_BLOCKS)};
    return d2d_tc_encode_map(m, sizeof(WT) == 1, 3, w, dims, strides, box);
}

template <typename WT> d2d_status make_maps(d2d_layer *L, const void *w1, const void *wg, const void *w2t)
{
    const int d = L->desc.d, rows = L->desc.d_ff, blocks = d / sub_cols<WT>();
    if (d % sub_cols<WT>() || rows % 16) return D2D_OK;
    bool ok = make_map<WT>(&L->tm_dec[0], w1, rows, d, blocks) && (!wg || make_map<WT>(&L->tm_dec[1], wg, rows, d, blocks));
    for (int i = 0; i < 3; ++i)
        if (blocks % (1 << i) == 0) ok = ok && make_map<WT>(&L->tm_dec[2 + i], w2t, rows, d, blocks >> i);
    L->dec_maps = ok;
    return ok ? D2D_OK : D2D_ERR_CUDA;
}

}  // namespace

// The layer's tensor maps (its weights stay where they are for the layer's lifetime): W1, W_gate, and W2T as clusters of
// 1, 2 and 4 CTAs read it.  L->dec_maps stays 0 for shapes the kernel does not take.
d2d_status d2d_decode_ffn_maps(d2d_layer *L)
{
    L->dec_maps = 0;
    if (L->desc.dtype != D2D_BF16) return D2D_OK;
    return L->q_w1 ? make_maps<uint8_t>(L, L->q_w1, L->q_wg, L->q_w2t) : make_maps<__nv_bfloat16>(L, L->w1, L->w_gate, L->w2t);
}

// The cut of a batch as d2d_decode_ffn takes it, for d2d_decode_plan_for
bool d2d_decode_ffn_plan(const d2d_layer_desc &D, int n_layers, int T, bool fp8, d2d_decode_plan *out)
{
    if (!d2d_decode_ffn_supports(D, n_layers, T, fp8)) return false;
    FfnShape S = shape_for(D, T);
    if (!(fp8 ? plan<uint8_t>(S, n_layers) : plan<__nv_bfloat16>(S, n_layers))) return false;
    out->token_block = 8 * nt8_for(T);
    out->cluster_size = S.cl;
    out->clusters = S.clusters;
    out->rounds = d2d_cdiv(d2d_cdiv(S.d_ff / 16, S.cl), S.clusters);
    out->static_rounds = S.n_static;
    out->stages = S.stages;
    out->list_entries = out->rounds * S.cl;
    out->list_capacity = MAX_LIST;
    return true;
}

// Whole 16-neuron units, rows of whole 128-byte blocks, a batch whose rows fit shared memory beside three stages.
bool d2d_decode_ffn_supports(const d2d_layer_desc &D, int n_layers, int T, bool fp8)
{
    if (D.dtype != D2D_BF16 || T < 1 || T > 32 || D.d_ff % 16 || D.d_ff / 16 > MAX_UNITS) return false;
    FfnShape S = shape_for(D, T);
    return fp8 ? plan<uint8_t>(S, n_layers) : plan<__nv_bfloat16>(S, n_layers);
}

int d2d_decode_ffn_first_shared(const d2d_layer_desc &D, int n_layers, int T, bool fp8)
{
    FfnShape S = shape_for(D, T);
    if (!(fp8 ? plan<uint8_t>(S, n_layers) : plan<__nv_bfloat16>(S, n_layers))) return 0;
    return S.n_static * S.clusters * S.cl;
}

d2d_status d2d_decode_ffn(const d2d_layer_desc &D, int n_layers, const d2d_decode_ffn_args &a, const void *x, int T, bool after_router,
                          cudaStream_t st)
{
    const bool fp8 = a.l[0].k1 != nullptr;
    if (n_layers < 1 || n_layers > D2D_MAX_GROUP) return D2D_ERR_UNSUPPORTED;
    const FfnShape S = shape_for(D, T);
    return fp8 ? dispatch<uint8_t>(S, n_layers, a, x, after_router, st) : dispatch<__nv_bfloat16>(S, n_layers, a, x, after_router, st);
}
