// Decode batches of bf16 layers (a few tokens per call): interface of the cluster router (decode_router.cu) and of the
// streaming expert kernel (decode_ffn.cu), and the warp-level building blocks they share.
#pragma once

#include "d2d_common.cuh"
#include "tc_common.cuh"

// Outputs and weights of one layer's router; a group of layers runs as one grid (blockIdx.y = layer).
struct d2d_decode_router_layer {
    const __nv_bfloat16 *w_r1, *b_r1, *w_r2, *b_r2;
    float *R;                  // [T, E] scores or NULL
    float *zero;               // float32 accumulator of the expert kernel that follows, cleared here (or NULL)
    uint32_t *mask;            // [T, W]
    int32_t *k;                // [T]
    int32_t *counts, *offsets, *perm, *tok_off, *tok_exp, *n_sel;      // lists, or all NULL
    int32_t *status;
    long long capacity;
    int32_t *units;            // NULL, or [0] entries, [1 ..] kept experts' 16-neuron units from unit u0 on, ascending
    int u0, upe;               // upe: units per expert
};
struct d2d_decode_router_args {
    d2d_decode_router_layer l[D2D_MAX_GROUP];
};

struct d2d_decode_ffn_layer {
    CUtensorMap tm_w1, tm_wg, tm_w2t;          // bf16 weights, or e4m3 codes when k1 is given: d2d_layer::tm_dec
    const CUtensorMap *tm_w2t_cl;              // host: W2T for clusters of 1, 2, 4; the launch picks tm_w2t from them
    const __nv_bfloat16 *b1, *b2;
    const int32_t *k1, *kg, *k2;
    const uint32_t *mask;
    const int32_t *units;                      // the router's list of kept units (see there) or NULL: found from the mask
    float *y32;                                // [T, d] zero at launch
    unsigned int *ticket;                      // zero at launch, left at zero
    __nv_bfloat16 *y;
    int32_t *status;
};
struct d2d_decode_ffn_args {
    d2d_decode_ffn_layer l[D2D_MAX_GROUP];
};

bool d2d_decode_router_supports(const d2d_layer_desc &D, int T);
// do_mask = 0: scores only (R).  zero_words: floats cleared at every layer's `zero`.
d2d_status d2d_decode_router(const d2d_layer_desc &D, int n_layers, const d2d_decode_router_args &a, const void *x, int T, float tau,
                             int do_mask, int zero_words, cudaStream_t st);

d2d_status d2d_decode_ffn_maps(d2d_layer *L);
// First unit that is not fixed to a CTA by its index (units from there on are shared out when the selection is known)
int d2d_decode_ffn_first_shared(const d2d_layer_desc &D, int n_layers, int T, bool fp8);
// Router and experts of n layers of one shape, two launches.  scratch[l]: d2d_decode_scratch_bytes each.
size_t d2d_decode_scratch_bytes(const d2d_layer_desc &D, int T);
d2d_status d2d_decode_layers(const d2d_layer *const *layers, int n, const void *x, int T, float tau, const d2d_routing *routing, float *R,
                             void *const *scratch, void *y, cudaStream_t st);
bool d2d_decode_ffn_supports(const d2d_layer_desc &D, int n_layers, int T, bool fp8);
bool d2d_decode_ffn_plan(const d2d_layer_desc &D, int n_layers, int T, bool fp8, d2d_decode_plan *out);
// after_router: launched right behind d2d_decode_router on `st` (weights and x are then read before it has finished)
d2d_status d2d_decode_ffn(const d2d_layer_desc &D, int n_layers, const d2d_decode_ffn_args &a, const void *x, int T, bool after_router,
                          cudaStream_t st);

// d2d_api.cu: the kernels' arguments for one layer, and whether a batch of T tokens takes the streaming expert kernel
bool d2d_use_decode_ffn(const d2d_layer *L, int n_layers, int T);
bool d2d_can_decode_ffn(const d2d_layer *L, int n_layers, int T);      // ... or would, whatever path the layer is set to
d2d_decode_router_layer d2d_decode_router_args_for(const d2d_layer *L, const d2d_routing *r, float *R, float *zero);
d2d_decode_ffn_layer d2d_decode_ffn_args_for(const d2d_layer *L, const d2d_routing *r, float *y32, unsigned int *ticket, void *y);

#ifdef __CUDACC__
namespace d2d_decode {

// D[16 x 8] += A[16 x 16] B[16 x 8]^T, bf16 operands, float32 accumulators.  With lane = 4 g + c: a0 / a1 hold rows g /
// g + 8 at two of the 16 k positions, a2 / a3 the same rows at two others, b0 / b1 column g at the same positions; d0, d1
// are row g, columns 2c and 2c + 1, d2, d3 row g + 8.  Which k positions a lane holds is free as long as A and B agree.
// Loop bounds and branches around it should be warp-uniform for the compiler (a warp index taken from a shuffle, no bounds
// that depend on the lane): otherwise the warp is re-converged around every instruction, which measured 300 cycles per step.
__device__ __forceinline__ void mma16816(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1)
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// Row p + 0..2 of the three-term bf16 expansion of a float32 value: v = t0 + t1 + t2 exactly (8 + 8 + 8 mantissa bits),
// so that a bf16 matrix instruction multiplies it without losing precision.
__device__ __forceinline__ void split3(float v, __nv_bfloat16 (&t)[3])
{
    t[0] = __float2bfloat16_rn(v);
    const float r1 = v - __bfloat162float(t[0]);
    t[1] = __float2bfloat16_rn(r1);
    t[2] = __float2bfloat16_rn(r1 - __bfloat162float(t[1]));
}

__device__ __forceinline__ uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void cp_async8(uint32_t dst, const void *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Wait for a barrier that other CTAs of the cluster complete (whole warps, about a second at most)
__device__ __forceinline__ bool mbar_wait_cluster(uint32_t bar, uint32_t parity, int32_t *status)
{
    return d2d_tc::mbar_wait_warp<true>(bar, parity, status);
}

}  // namespace d2d_decode
#endif
