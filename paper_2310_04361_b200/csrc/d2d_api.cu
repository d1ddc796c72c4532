// Host side of the C ABI declared in include/d2d.h: argument validation, weight packing,
// workspace carving and kernel dispatch.  No computation happens on the host.
#include <limits.h>
#include <math.h>
#include <new>
#include <string.h>

#include "d2d_common.cuh"
#include <stdlib.h>
#include "decode.cuh"
#include "gemm_tc.cuh"
#include "moe_gather.cuh"
#include "moe_sorted.cuh"

bool d2d_token_path_supports(const d2d_layer_desc &D);
d2d_status d2d_launch_moe_ffn_token(const d2d_layer *L, const void *x, int T, const d2d_routing *r, void *y,
                                    cudaStream_t st);

unsigned long long d2d_launch_counter = 0;
static int g_test_fault = 0;       // d2d_test_inject_fault: consumed by the next d2d_expert_up_fwd

namespace {

bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

bool has_lists(const d2d_routing *r) { return r->counts && r->offsets && r->perm && r->n_sel; }

// lists_optional: the per-expert lists (counts, offsets, perm, n_sel) may be absent as a set (d2d_layer_fwd then
// does not build them); mask, k and status are always required
bool routing_ok(const d2d_routing *r, bool lists_optional)
{
    if (!r || !r->mask || !r->k || !r->status) return false;
    const bool none = !r->counts && !r->offsets && !r->perm && !r->n_sel && !r->tok_off && !r->tok_exp;
    if (lists_optional && none) return true;
    if (!has_lists(r)) return false;
    if ((r->tok_off == nullptr) != (r->tok_exp == nullptr)) return false;
    return r->perm_capacity >= 0;
}

// Workspace layout of the layer-level calls: [ u: T*d_h f32 | R: T*E f32 | select scratch | ffn scratch ]
struct ws_layout {
    size_t u_off, r_off, sel_off, ffn_off, total;
};

// What a call with exactly T tokens needs
ws_layout layout_for(const d2d_layer *L, int T)
{
    ws_layout w;
    const size_t Tn = (size_t)(T > 0 ? T : 1);
    size_t off = 0;
    w.u_off = off;
    off += 256 + d2d_align_up(Tn * (size_t)L->desc.d_h * sizeof(float), 256);   // ticket area + hidden activations
    w.r_off = off;
    off += d2d_align_up(Tn * (size_t)L->desc.n_experts * sizeof(float), 256);
    w.sel_off = off;
    off += d2d_select_ws_bytes((int)Tn, L->desc.n_experts);
    w.ffn_off = off;
    off += d2d_moe_ffn_ws_bytes(L, (int)Tn);
    w.total = off;
    return w;
}

}  // namespace

// Up to this many tokens a bf16 layer takes CUDA-core arithmetic (the streaming decode kernels then carry float32 hidden
// activations as three bf16 terms, so that results are as precise as those of small_batch_ffn.cu), above it tensor-core
// arithmetic with bf16 hidden activations.  Measured with small_batch_ffn.cu, which still serves the shapes the streaming
// kernels do not take, before those existed (us per layer call, small_batch_ffn.cu / tensor-core path): GPT-2-medium-shaped FFN
// (64 KB of weights per expert) T = 3: 31 / 39, T = 4: 33 / 39, T = 5: 41 / 40, T = 8: 43 / 39; Llama-shaped layer (786 KB per expert) T = 1: 84 / 129, T = 2: 108 / 133, T = 3: 221 / 133,
// T = 4: 229 / 127.  So 4 tokens for small experts, 2 for large ones; D2D_DECODE_MAX_TOKENS overrides both.
int d2d_decode_max_tokens(const d2d_layer_desc &D)
{
    static const int v = [] {
        const char *e = getenv("D2D_DECODE_MAX_TOKENS");
        const int n = e ? atoi(e) : -1;
        return n > 8 ? 8 : n;
    }();
    if (v >= 0) return v;
    const size_t expert_bytes = (size_t)(D.gated ? 3 : 2) * D.expert_size * D.d * 2;
    return expert_bytes > ((size_t)256 << 10) ? 2 : 4;
}

static bool use_dense_masked(const d2d_layer *L, int T)
{
    return L->desc.dtype == D2D_BF16 && T > d2d_decode_max_tokens(L->desc) && L->desc.d_ff % 8 == 0 && d2d_gemm_tc_available();
}

// Up to this many tokens the expert-per-CTA kernel (each kept expert's slice read once) is used.
static bool use_small_ffn(const d2d_layer *L, int T)
{
    const int lim = L->desc.dtype == D2D_BF16 ? d2d_decode_max_tokens(L->desc) : 8;      // fp32 layers have no tensor-core path
    return T <= lim && d2d_small_ffn_supports(L->desc);
}

// Batches of a few tokens of bf16 layers: cluster router and streaming expert kernel (decode_router.cu, decode_ffn.cu).
// A path forced through d2d_layer_set_expert_path concerns the tensor-core batches: those keep it.
bool d2d_use_decode_ffn(const d2d_layer *L, int n_layers, int T)
{
    if (T > d2d_decode_max_tokens(L->desc) && L->expert_path != D2D_PATH_AUTO) return false;
    return d2d_can_decode_ffn(L, n_layers, T);
}

bool d2d_can_decode_ffn(const d2d_layer *L, int n_layers, int T)
{
    return L->dec_maps && d2d_decode_ffn_supports(L->desc, n_layers, T, L->q_w1 != nullptr);
}

d2d_decode_ffn_layer d2d_decode_ffn_args_for(const d2d_layer *L, const d2d_routing *r, float *y32, unsigned int *ticket, void *y)
{
    d2d_decode_ffn_layer a = {};
    a.tm_w1 = L->tm_dec[0]; a.tm_wg = L->tm_dec[1]; a.tm_w2t_cl = L->tm_dec + 2;
    a.b1 = (const __nv_bfloat16 *)L->b1; a.b2 = (const __nv_bfloat16 *)L->b2;
    if (L->q_w1) {                                             // 8-bit expert weights: the kernel reads the codes
        a.k1 = L->q_k1; a.kg = L->q_kg; a.k2 = L->q_k2;
    }
    a.mask = r->mask; a.y32 = y32; a.ticket = ticket; a.y = (__nv_bfloat16 *)y; a.status = r->status;
    return a;
}

d2d_decode_router_layer d2d_decode_router_args_for(const d2d_layer *L, const d2d_routing *r, float *R, float *zero)
{
    d2d_decode_router_layer a = {};
    a.w_r1 = (const __nv_bfloat16 *)L->w_r1; a.b_r1 = (const __nv_bfloat16 *)L->b_r1;
    a.w_r2 = (const __nv_bfloat16 *)L->w_r2; a.b_r2 = (const __nv_bfloat16 *)L->b_r2;
    a.R = R; a.zero = zero;
    if (r) {
        a.mask = r->mask; a.k = r->k; a.counts = r->counts; a.offsets = r->offsets; a.perm = r->perm;
        a.tok_off = r->tok_off; a.tok_exp = r->tok_exp; a.n_sel = r->n_sel; a.status = r->status; a.capacity = (long long)r->perm_capacity;
    }
    return a;
}

// [ticket (256 bytes) | float32 accumulator [T, d] | list of units]
size_t d2d_decode_scratch_bytes(const d2d_layer_desc &D, int T)
{
    return 256 + d2d_align_up((size_t)T * D.d * 4, 256) + d2d_align_up((size_t)(1 + D.d_ff / 16) * 4, 256);
}

d2d_status d2d_decode_layers(const d2d_layer *const *layers, int n, const void *x, int T, float tau, const d2d_routing *routing, float *R,
                             void *const *scratch, void *y, cudaStream_t st)
{
    const d2d_layer_desc &D = layers[0]->desc;
    d2d_decode_router_args ra = {};
    d2d_decode_ffn_args fa = {};
    // experts of whole units: the router lists the units the experts share out; otherwise they find them from the mask
    const int U = D.d_ff / 16, upe = D.expert_size % 16 ? 0 : D.expert_size / 16;
    const int u0 = upe ? d2d_decode_ffn_first_shared(D, n, T, layers[0]->q_w1 != nullptr) : U;
    const bool list = u0 < U && u0 % upe == 0;
    for (int l = 0; l < n; ++l) {
        float *y32 = (float *)((char *)scratch[l] + 256);
        ra.l[l] = d2d_decode_router_args_for(layers[l], &routing[l], R, y32);           // the router clears the accumulator
        fa.l[l] = d2d_decode_ffn_args_for(layers[l], &routing[l], y32, layers[l]->tickets + 16, (char *)y + (size_t)l * T * D.d * 2);
        if (list) {
            ra.l[l].units = (int32_t *)((char *)y32 + d2d_align_up((size_t)T * D.d * 4, 256));
            ra.l[l].u0 = u0; ra.l[l].upe = upe;
            fa.l[l].units = ra.l[l].units;
        }
    }
    const d2d_status rc = d2d_decode_router(D, n, ra, x, T, tau, 1, T * D.d, st);
    return rc != D2D_OK ? rc : d2d_decode_ffn(D, n, fa, x, T, true, st);
}

size_t d2d_layer_ws_bytes(const d2d_layer *L, int T) { return layout_for(L, T).total; }

// Whether a batch may take the sorted form (moe_sorted.cu), by shape and size: from 1.1e11 FLOP of up projection on (23300 tokens of the
// paper's shape).  Shorter batches win where few pairs are kept (expert step, us, dense pair / sorted form at p = 0.02, 0.05, 0.1, 0.2: 12608
// tokens 105 / 60, 75, 84, 104; 8000 tokens 69 / 52, 59, 66, 79), but where the dense pair runs in the end the four kernels of the other
// form cost it 10 to 20 us (14000 tokens, p = 0.3, routing and expert step 125 / 136; 30000, p = 0.45, 240 / 238).
static bool sorted_shape(const d2d_layer_desc &D, int T)
{
    return 2.0 * (double)T * D.d * D.d_ff >= 1.1e11 && d2d_sorted_supports(D, T) && d2d_gemm_tc_splits(T, D.d, D.d_ff) == 1;
}

size_t d2d_moe_ffn_ws_bytes(const d2d_layer *L, int T)
{
    size_t need = 256;
    if (d2d_decode_ffn_supports(L->desc, 1, T, L->q_w1 != nullptr)) need = d2d_decode_scratch_bytes(L->desc, T);
    if (use_small_ffn(L, T) && d2d_small_ffn_ws_bytes(L, T) > need) need = d2d_small_ffn_ws_bytes(L, T);
    // hidden activations H [T, d_ff] bf16 of the dense-masked path
    if (L->desc.dtype == D2D_BF16 && T > d2d_decode_max_tokens(L->desc)) {
        size_t h = d2d_align_up((size_t)T * L->desc.d_ff * 2, 256);
        h += d2d_align_up(d2d_gemm_tc_partial_floats(T, L->desc.d, L->desc.d_ff) * 4, 256);      // split-K partial sums
        if (sorted_shape(L->desc, T)) h += d2d_sorted_layout_for(L->desc, T).total;
        if (h > need) need = h;
    }
    return need;
}

// Density up to which the automatic choice takes the gathered pair for this shape and batch size.  The gathered kernel is bound
// by the rate at which token rows can be copied into the A stages (about the same time per 128 x 64 tile of gathered rows
// whatever the MMA width), so with full-width groups a gathered row costs about 1.2 x a dense one, and the kernel has a fixed
// part (the scan of the mask, a ragged tile per group visit) worth about five tiles per CTA.  Against a dense up projection of
// T / 128 x Nd tiles (Nd = 256-column tiles across d_ff) on S SMs that fixed part is T0 = 5 * 128 * 1.2 * S / Nd tokens' worth
// of dense time, so the pair is taken while the fraction of kept (token, group) pairs
//     u = 1 - (1 - rho)^g  <  U - T0 / T,
// U = 0.85 for 256 MMA columns (less for narrower groups).
// Gated layers run in pairs of CTAs: U = 0.73 and three tiles.  Llama-shaped layer, up projections back to back (us, gathered /
// masked dense): 8192 tokens, u 0.62 and 0.24: 883 / 951 and 386 / 943; 2560 tokens: 310 / 300 and 192 / 300, that is 85 + 0.159 u T
// against 0.1165 T; the kernels of the form that is not taken and the zero fill cost the choice another 40.
// Plain layers: U was fitted to a dense pair without CTA pairs and TMA stores; the present one is faster, so the rule takes the
// gathered pair in a band of densities where the dense one would be level or ahead.  Paper's shape, 50432 tokens, expert step with
// each forced and with the choice, one interleaved loop under sustained load (us, dense / gathered / automatic; the rule's limit):
//     rho 0.4    366 /  390 /  413   0.3    366 /  357 /  378   0.2    363 /  319 /  337   (0.42)
// (the last includes 14 to 24 us for the kernels of the forms that are not taken, which are launched and return).
int d2d_tc_sm_count();      // gemm_tc.cu

// Smallest up projection for which the automatic choice is made, see path_before_launch.  Gated layers with the library's own limit on
// the density: from where that limit lets the gathered pair in at 3.5 % of the pairs (1330 tokens of the Llama-shaped layer);
// below, the choice would only cost them the overlap with the router.  Above it the choice is what lets sparse batches take the gathered
// pair, and costs dense ones that overlap and the launches.  Llama-shaped layer, interleaved (us, dense form / with the choice, * =
// which took the gathered pair):
//     1400 tokens  rho 0.22  338 / 372   0.07  333 / 366    0.03  318 / 291*
//     1500         rho 0.22  339 / 377   0.07  335 / 366    0.03  319 / 292*
//     1760         rho 0.22  385 / 440   0.07  361 / 347*   0.03  348 / 300*
// The line was at 3.2e11 for a while, which kept the first column and gave away the last (370 instead of 297 at 1760 tokens).
static double auto_min_up_flop(const d2d_layer *L) { return L->desc.gated && L->gather_rho_max < 0.0 ? 2.4e11 : 2e11; }

static double default_gather_rho_max(const d2d_layer_desc &D, int g, int T)
{
    if (g <= 0 || T <= 0) return -1.0;
    const int n_mma = g * D.expert_size * (D.gated ? 2 : 1);
    double U = n_mma >= 256 ? (D.gated ? 0.73 : 0.85) : n_mma >= 192 ? 0.64 : n_mma >= 128 ? 0.43 : 0.25;
    const double nd = ceil((double)D.d_ff * (D.gated ? 2.0 : 1.0) / 256.0);
    const double T0 = (D.gated ? 3.0 : 5.0) * 128.0 * 1.2 * (double)d2d_tc_sm_count() / nd;
    const double u_max = U - T0 / (double)T;
    if (u_max <= 0.0) return 0.0;
    return 1.0 - pow(1.0 - u_max, 1.0 / g);
}

// Density up to which the automatic choice takes the fused gathered kernel.  Its merge moves 4 d bytes of vector reductions per
// kept (token, group) pair through each SM's path to L2, next to the token and weight rows coming in, and its float32
// accumulator is written once and read once more than the other paths' output.  It is taken while at most 8 % of the (token,
// group) pairs are kept.  Measured (d = 768, 128-neuron groups, 50432 tokens, us, fused / gathered pair at 1 / 2 / 5 / 8 / 10 /
// 15 % of the pairs): 140 / 220, 150 / 226, 175 / 235, 220 / 249, 256 / 263, 335 / 294.
static double default_fused_rho_max(int g)
{
    if (g <= 0) return 0.0;
    return 1.0 - pow(1.0 - 0.08, 1.0 / g);
}

// The form of the expert step as far as it is known before the launch: the one that is set, or the dense pair where the shape or the
// size leaves no choice.
// The automatic choice costs a few launches that return at once and the overlap of the router with the masked dense
// kernel's main loops (ViT-shaped layer, 1.2e11 FLOP: 241 us against 224 us at every density when the line was drawn), so it
// is made only for problems whose up projection takes long enough (2e11 FLOP, about 150 us of tensor-core time) that this is
// little.  What the line gives away: on the ViT-shaped layer the gathered pair wins below rho = 0.03 (205 against 219 us at
// 0.023), and on the paper's shape at 12608 tokens (6e10 FLOP, expert step) the fused kernel wins up to rho = 0.17 (58 / 73 / 87
// against 110 us at 0.01 / 0.05 / 0.1).
static int path_before_launch(const d2d_layer *L, int T, bool counted)
{
    const d2d_layer_desc &D = L->desc;
    int path = L->expert_path;
    if (L->gather_group <= 0) path = D2D_PATH_DENSE;
    const double up_flop = 2.0 * (double)T * D.d * D.d_ff * (D.gated ? 2.0 : 1.0);
    if (path == D2D_PATH_AUTO && (up_flop < auto_min_up_flop(L) || !counted)) path = D2D_PATH_DENSE;
    return path;
}

// Largest number of selected pairs with which the automatic choice takes the sorted form, -1: never.  Tiles of 128 ordered tokens can
// tell apart about as many patterns of kept experts as there are tiles: with an entropy of h(rho) bits per decision a tile fixes
// log2(T / 128) / h of the E experts and has all of the others in its union, which leaves 1 - (1 - rho) log2(T / 128) / (E h) of
// the work.  (Independent decisions are the worst case; correlated ones leave less.)  The form is level with the dense pair where 0.73
// is left: expert step of the paper's shape, us, sorted / dense, a box each: 50432 tokens p = 0.1 175 / 342, 0.2 266 / 348, 0.3 341 /
// 356, 0.4 396 / 370 (the limit: 0.32); 25000 tokens 0.1 130 / 183, 0.2 172 / 178, 0.3 189 / 178 (0.28); and the choice itself costs 10 to
// 14 where the dense pair runs in the end (p = 0.5: 25000 tokens 222 / 208, 40000 356 / 344, 50432 437 / 424).
// in_layer_call: behind a router, which overlaps a dense up projection that is not chosen: only batches that had a choice anyway (they
// paid for the kernels of two other forms).  Layer call, us, with this choice / the dense pair forced / with the fused, gathered and dense
// forms that were the choice before: 42600 tokens, rho = 0.06 147 / 322 / 268, 0.14 250 / 353 / 381, 0.28 350 / 364 / 415, above the limit
// 0.33 404 / 373 / 448, 0.51 411 / 390 / 392; 80000 tokens, 0.09 356 / 632 / 658, 0.33 669 / 674 / 812; 32 experts of 64 neurons, d = 1024,
// 60000 tokens (the limit: 0.235), 0.05 234 / 405 / 341, 0.12 388 / 439 / 469, 0.18 445 / 429 / 528, 0.22 486 / 447 / 487: there the
// form is level a little earlier, at 0.17.
static double default_fused_rho_max(int g);
static long long sorted_n_sel_max(const d2d_layer *L, int T, bool in_layer_call)
{
    const d2d_layer_desc &D = L->desc;
    if (L->expert_path != D2D_PATH_AUTO || L->gather_rho_max >= 0.0 || !sorted_shape(D, T)) return -1;
    if (L->fused_group > 0 && L->fused_rho_max != default_fused_rho_max(L->fused_group)) return -1;
    if (in_layer_call && 2.0 * (double)T * D.d * D.d_ff < auto_min_up_flop(L)) return -1;
    const double patterns = log2((double)T / 128.0) / D.n_experts;
    double lo = 0.0, hi = 0.5;
    for (int i = 0; i < 14; ++i) {
        const double rho = 0.5 * (lo + hi), h = -rho * log2(rho) - (1.0 - rho) * log2(1.0 - rho);
        (1.0 - (1.0 - rho) * fmin(patterns / h, 1.0) <= 0.73 ? lo : hi) = rho;
    }
    return (long long)(lo * (double)T * (double)D.n_experts);
}

// The masked dense pair's arguments
static d2d_gemm_args dense_up_args(const d2d_layer *L, const void *x, int T, const d2d_routing *r, void *H)
{
    const d2d_layer_desc &D = L->desc;
    d2d_gemm_args up = {};
    up.a = x; up.b = L->w1; up.b_gate = D.gated ? L->w_gate : nullptr; up.b_cat = L->w1g; up.b_cat_block = 128; up.bias = L->b1; up.out = H;
    up.M = T; up.N = D.d_ff; up.K = D.d; up.epilogue = D2D_EPI_UP_MASKED; up.act = D.act;
    up.mask = r->mask; up.mask_words = (D.n_experts + 31) / 32; up.expert_size = D.expert_size; up.status = r->status;
    return up;
}
static d2d_gemm_args dense_down_args(const d2d_layer *L, const void *H, int T, void *y, int32_t *status)
{
    const d2d_layer_desc &D = L->desc;
    d2d_gemm_args dn = {};
    dn.a = H; dn.b = L->w2; dn.bias = L->b2; dn.out = y;
    dn.M = T; dn.N = D.d; dn.K = D.d_ff; dn.epilogue = D2D_EPI_BIAS_BF16; dn.status = status;
    return dn;
}

// The sorted form up to n_sel_max selected pairs, the masked dense pair above
static d2d_status launch_sorted_or_dense(const d2d_layer *L, const void *x, int T, const d2d_routing *r, void *y, void *ws, cudaStream_t st,
                                         const int32_t *n_sel, long long n_sel_max)
{
    char *const scratch = (char *)ws + d2d_align_up((size_t)T * L->desc.d_ff * 2, 256);
    d2d_status rc = d2d_moe_sorted(L, x, T, r, y, ws, scratch, L->sorted_ctr, (int *)(L->tickets + 56), n_sel, n_sel_max, st);
    if (rc != D2D_OK) return rc;
    d2d_gemm_args up = dense_up_args(L, x, T, r, ws), dn = dense_down_args(L, ws, T, y, r->status);
    up.n_sel = dn.n_sel = n_sel;
    up.n_sel_max = dn.n_sel_max = n_sel_max;
    rc = d2d_gemm_tc(up, st);
    return rc != D2D_OK ? rc : d2d_gemm_tc(dn, st);
}

// Expert step of bf16 batches above the decode sizes, on the tensor cores.
//   up projection    two kernels that compute the same H = G * A(x W1^T + b1):
//     masked dense   one GEMM over all of d_ff, the selection applied as a mask in the epilogue; its time does not
//                    depend on the selection (every expert is kept by some token of a 128-token tile)
//     gathered       per group of adjacent experts, a contraction over the tokens that keep the group (moe_gather.cu);
//                    its time is proportional to the number of (token, group) pairs
//   down projection  y = H W2^T + b2 as a dense GEMM: exactly b2 + the sum over kept experts, since the h of an expert
//                    the token did not keep is zero (written as zero by the masked dense kernel, or zero-filled from
//                    the mask while H is staged when the gathered kernel, which writes only kept cells, may have run)
// Which up projection runs is decided per call from the number of selected pairs of THIS batch.  D2D_PATH_AUTO
// launches both kernels with complementary rules on a device word (n_sel) that is valid once the preceding kernel of
// the stream has completed; the one that is not needed returns at once, so no host synchronisation is involved.
// up_counter (optional): a zeroed device counter; its presence also states that the kernel launched just before
// on this stream is the router, which writes only the mask (and R, k), so that a forced masked dense up projection
// may overlap it with its main loops and draw its tiles dynamically.
static d2d_status launch_tc_experts(const d2d_layer *L, const void *x, int T, const d2d_routing *r, void *y,
                                    void *ws, cudaStream_t st, int *up_counter, const int32_t *n_sel, bool lists)
{
    const d2d_layer_desc &D = L->desc;
    const long long n_sel_sorted = n_sel ? sorted_n_sel_max(L, T, n_sel != r->n_sel) : -1;
    if (n_sel_sorted >= 0) return launch_sorted_or_dense(L, x, T, r, y, ws, st, n_sel, n_sel_sorted);
    const int path = path_before_launch(L, T, n_sel != nullptr);
    const double rho_max = L->gather_rho_max >= 0.0 ? L->gather_rho_max : default_gather_rho_max(D, L->gather_group, T);
    long long n_sel_max = (long long)(rho_max * (double)T * (double)D.n_experts);
    d2d_status rc;
    // Fused gathered step (plain layers): up projection, activation, down projection and the merge in one kernel whose
    // time is proportional to the kept (token, group) pairs; the float32 accumulator takes the place of H.
    long long n_sel_fused = -1;
    if (L->fused_group > 0 && (path == D2D_PATH_FUSED || (path == D2D_PATH_AUTO && L->fused_rho_max > 0.0))) {
        d2d_gather_args fa = {};
        fa.x = x; fa.w1 = L->w1; fa.b1 = L->b1; fa.mask = r->mask;
        fa.T = T; fa.d = D.d; fa.d_ff = D.d_ff; fa.n_experts = D.n_experts; fa.s = D.expert_size; fa.g = L->fused_group;
        fa.act = D.act; fa.status = r->status; fa.ctr = L->gather_ctr;
        if (path == D2D_PATH_AUTO) {
            // three ranges of n_sel: (.., fused] fused kernel, (fused, max] gathered pair, (max, ..) dense pair
            n_sel_fused = (long long)(L->fused_rho_max * (double)T * (double)D.n_experts);
            if (n_sel_max < n_sel_fused) n_sel_max = n_sel_fused;
            fa.n_sel = n_sel; fa.n_sel_min = -1; fa.n_sel_max = n_sel_fused;
        }
        rc = d2d_moe_gather_ffn(fa, (float *)ws, y, L->w2, L->b2, st);
        if (rc != D2D_OK || path == D2D_PATH_FUSED) return rc;
    } else if (path == D2D_PATH_FUSED) {
        return D2D_ERR_UNSUPPORTED;
    }
    // decode-sized batches: split K of the down projection over the SMs, partial sums in the float32 scratch behind H
    const int k_splits = d2d_gemm_tc_splits(T, D.d, D.d_ff);
    float *partial = k_splits > 1 ? (float *)((char *)ws + d2d_align_up((size_t)T * D.d_ff * 2, 256)) : nullptr;
    // Wide layers: the cells the gathered kernel leaves alone are zero-filled, so that the TMA-fed dense down projection can follow
    // whichever up projection ran; otherwise the down projection that applies the selection while it stages H follows the gathered
    // kernel.  In front of both up projections: on the side stream beside the gathered kernel, behind the dense one, it saved nothing there
    // (Llama-shaped layer, us, there / here: 3500 tokens at tau = 0.6 557 / 562, 6000 at 0.5 998 / 997, 8192 at 0.4 1657 / 1651), and where
    // the dense form runs the events and waits between the streams held up the down projection (1536 tokens 384 / 372, 2048 479 / 463, 2560
    // 591 / 574).
    const bool zero_fill = path != D2D_PATH_DENSE && D.d >= 2048;
    const long long hi = path == D2D_PATH_AUTO ? n_sel_max : LLONG_MAX;
    if (zero_fill) {
        rc = d2d_moe_zero_unkept(ws, r->mask, T, D.d_ff, D.n_experts, D.expert_size, L->gather_group, n_sel, n_sel_fused, hi, st);
        if (rc != D2D_OK) return rc;
    }
    if (path != D2D_PATH_GATHER) {
        d2d_gemm_args up = dense_up_args(L, x, T, r, ws);
        const bool forced = path == D2D_PATH_DENSE;
        up.tile_counter = forced ? up_counter : nullptr;
        up.pdl_late_wait = forced && up_counter != nullptr;
        up.n_sel = forced ? nullptr : n_sel; up.n_sel_max = n_sel_max;
        if (forced && k_splits > 1) { up.zero = partial; up.zero_floats = (long long)d2d_gemm_tc_partial_floats(T, D.d, D.d_ff); }
        rc = d2d_gemm_tc(up, st);
        if (rc != D2D_OK) return rc;
    }
    if (path != D2D_PATH_DENSE) {
        d2d_gather_args ga = {};
        ga.x = x; ga.w1 = L->w1; ga.w_gate = D.gated ? L->w_gate : nullptr; ga.b1 = L->b1; ga.mask = r->mask; ga.H = ws;
        ga.T = T; ga.d = D.d; ga.d_ff = D.d_ff; ga.n_experts = D.n_experts; ga.s = D.expert_size; ga.g = L->gather_group;
        ga.act = D.act; ga.status = r->status; ga.ctr = L->gather_ctr;
        ga.n_sel = n_sel; ga.n_sel_min = n_sel_fused; ga.n_sel_max = hi;
        rc = d2d_moe_gather_up(ga, st);
        if (rc != D2D_OK) return rc;
    }
    if (path != D2D_PATH_DENSE && !zero_fill) {
        rc = d2d_moe_down_masked(D, ws, r->mask, L->w2, L->b2, y, T, r->status, st, path == D2D_PATH_AUTO ? n_sel : nullptr, n_sel_fused, n_sel_max);
        if (rc != D2D_OK || path == D2D_PATH_GATHER) return rc;
    }
    d2d_gemm_args dn = dense_down_args(L, ws, T, y, r->status);
    // after a zero fill this kernel serves the gathered range too: it only has to stay out of the fused kernel's range
    dn.n_sel = path == D2D_PATH_AUTO && (!zero_fill || n_sel_fused >= 0) ? n_sel : nullptr;
    dn.n_sel_max = zero_fill ? n_sel_fused : n_sel_max;
    dn.k_splits = k_splits;
    dn.partial = partial;
    dn.partial_zero = path == D2D_PATH_DENSE;
    if (lists) dn.lists = d2d_list_job_for(r, 1, T, D.n_experts, false);
    return d2d_gemm_tc(dn, st);
}

d2d_status d2d_launch_moe_ffn(const d2d_layer *L, const void *x, int T, const d2d_routing *r, void *y,
                              void *ws, size_t ws_bytes, cudaStream_t st, int *up_counter, int small_fused, const int32_t *n_sel, bool lists)
{
    if (ws_bytes < d2d_moe_ffn_ws_bytes(L, T)) return D2D_ERR_WORKSPACE;
    if (d2d_use_decode_ffn(L, 1, T)) {
        // the ticket and the float32 accumulator must start at zero
        if (cudaMemsetAsync(ws, 0, 256 + (size_t)T * L->desc.d * 4, st) != cudaSuccess) return D2D_ERR_CUDA;
        d2d_decode_ffn_args a = {};
        a.l[0] = d2d_decode_ffn_args_for(L, r, (float *)((char *)ws + 256), (unsigned int *)ws, y);
        return d2d_decode_ffn(L->desc, 1, a, x, T, false, st);
    }
    if (use_small_ffn(L, T)) return has_lists(r) ? d2d_small_ffn(L, x, T, r, y, ws, st, small_fused) : D2D_ERR_INVALID_ARG;
    if (use_dense_masked(L, T)) return launch_tc_experts(L, x, T, r, y, ws, st, up_counter, n_sel ? n_sel : r->n_sel, lists);
    return d2d_launch_moe_ffn_token(L, x, T, r, y, st);
}

extern "C" {

uint64_t d2d_launch_count(void) { return __atomic_load_n(&d2d_launch_counter, __ATOMIC_RELAXED); }

const char *d2d_status_str(d2d_status s)
{
    switch (s) {
    case D2D_OK: return "ok";
    case D2D_ERR_INVALID_ARG: return "invalid argument";
    case D2D_ERR_UNSUPPORTED: return "unsupported shape or option";
    case D2D_ERR_WORKSPACE: return "workspace too small";
    case D2D_ERR_CUDA: return "CUDA runtime or launch failure";
    case D2D_ERR_NONFINITE: return "non-finite router score";
    case D2D_ERR_TIMEOUT: return "bounded wait ran out inside a kernel";
    case D2D_ERR_CAPACITY: return "more selected pairs than perm_capacity";
    }
    return "unknown status";
}

// Gated bf16 layers: W1 and W_gate once more, interleaved in blocks of 128 rows (the gated up projection fetches both
// tiles with one TMA box).  Built from the layer's own packed copies (again after they were replaced by dequantised values).
static d2d_status build_gate_cat(d2d_layer *L, cudaStream_t st)
{
    const d2d_layer_desc &D = L->desc;
    const int cat_block = 128;
    const size_t cat_rows = (size_t)2 * cat_block * d2d_cdiv(D.d_ff, cat_block);
    const size_t row_b = (size_t)D.d * L->elem;
    char *cat = (char *)L->w1g;
    if (cudaMemsetAsync(cat, 0, cat_rows * row_b, st) != cudaSuccess) return D2D_ERR_CUDA;
    for (int r0 = 0, b = 0; r0 < D.d_ff; r0 += cat_block, ++b) {
        const size_t rows = (size_t)(D.d_ff - r0 < cat_block ? D.d_ff - r0 : cat_block);
        char *dst = cat + (size_t)b * 2 * cat_block * row_b;
        if (cudaMemcpyAsync(dst, (const char *)L->w1 + (size_t)r0 * row_b, rows * row_b, cudaMemcpyDeviceToDevice, st) != cudaSuccess ||
            cudaMemcpyAsync(dst + (size_t)cat_block * row_b, (const char *)L->w_gate + (size_t)r0 * row_b, rows * row_b,
                            cudaMemcpyDeviceToDevice, st) != cudaSuccess)
            return D2D_ERR_CUDA;
    }
    return D2D_OK;
}

d2d_status d2d_layer_create(const d2d_layer_desc *desc, const d2d_weights *w, void *stream, d2d_layer **out)
{
    if (out) *out = nullptr;
    if (!desc || !w || !out) return D2D_ERR_INVALID_ARG;
    const d2d_layer_desc &D = *desc;
    if (D.d <= 0 || D.d_ff <= 0 || D.n_experts <= 0 || D.expert_size <= 0 || D.d_h <= 0) return D2D_ERR_INVALID_ARG;
    if ((int64_t)D.n_experts * D.expert_size != D.d_ff) return D2D_ERR_INVALID_ARG;
    if (D.dtype != D2D_F32 && D.dtype != D2D_BF16) return D2D_ERR_INVALID_ARG;
    if (D.act < D2D_ACT_RELU || D.act > D2D_ACT_SILU) return D2D_ERR_INVALID_ARG;
    if (D.d % 8 || D.d_h % 8) return D2D_ERR_INVALID_ARG;
    if (!w->w_r1 || !w->w_r2 || !w->w1 || !w->w2) return D2D_ERR_INVALID_ARG;
    if ((D.gated != 0) != (w->w_gate != nullptr)) return D2D_ERR_INVALID_ARG;
    if (!d2d_token_path_supports(D)) return D2D_ERR_UNSUPPORTED;

    int dev = 0, sms = 0;
    D2D_CUDA_TRY(cudaGetDevice(&dev));
    D2D_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));

    d2d_layer *L = new (std::nothrow) d2d_layer();
    if (!L) return D2D_ERR_CUDA;
    memset(L, 0, sizeof(*L));
    L->desc = D;
    L->elem = D.dtype == D2D_F32 ? 4 : 2;
    L->sm_count = sms;
    const size_t el = L->elem;
    const size_t n_wr1 = (size_t)D.d_h * D.d, n_wr2 = (size_t)D.n_experts * D.d_h, n_w = (size_t)D.d_ff * D.d;

    struct piece { void **dst; const void *src; size_t n; bool transpose; };
    piece pieces[] = {
        {&L->w_r1, w->w_r1, n_wr1, false}, {&L->b_r1, w->b_r1, (size_t)D.d_h, false},
        {&L->w_r2, w->w_r2, n_wr2, false}, {&L->b_r2, w->b_r2, (size_t)D.n_experts, false},
        {&L->w1, w->w1, n_w, false},       {&L->b1, w->b1, (size_t)D.d_ff, false},
        {&L->w_gate, w->w_gate, n_w, false}, {&L->w2t, w->w2, n_w, true},
        {&L->b2, w->b2, (size_t)D.d, false}, {&L->w2, w->w2, n_w, false},
    };
    size_t total = 256;                                   // the ticket words (see d2d_layer::tickets)
    L->gather_group = d2d_gather_group_for(D, 0);
    L->gather_rho_max = -1.0;                             // the default for the shape and the batch size of each call
    L->expert_path = D2D_PATH_AUTO;
    L->fused_group = d2d_gather_ffn_group_for(D);
    L->fused_rho_max = default_fused_rho_max(L->fused_group);
    L->gather_ctr_words = (int)d2d_align_up(D.n_experts + 64, 64);      // enough for any group size: E / g counters + the exit ticket
    const int sorted_at = L->gather_ctr_words;
    if (d2d_sorted_supports(D, 1)) L->gather_ctr_words += D2D_SORTED_CTR_WORDS;
    const size_t ctr_off = total;
    total += d2d_align_up((size_t)L->gather_ctr_words * sizeof(int), 256);
    for (const piece &p : pieces)
        if (p.src) total += d2d_align_up(p.n * el, 256);
    // gated bf16 layers: W1 and W_gate once more, interleaved in blocks of 128 rows for the tensor-core up projection
    const int cat_block = 128;
    const size_t cat_rows = (size_t)2 * cat_block * d2d_cdiv(D.d_ff, cat_block);
    const bool want_cat = D.gated && D.dtype == D2D_BF16;
    const size_t cat_off = total;
    if (want_cat) total += d2d_align_up(cat_rows * D.d * el, 256);
    cudaStream_t st = (cudaStream_t)stream;
    if (cudaMalloc(&L->slab, total) != cudaSuccess) {
        delete L;
        return D2D_ERR_CUDA;
    }
    L->slab_bytes = total;
    L->tickets = (unsigned int *)L->slab;
    L->gather_ctr = (int *)((char *)L->slab + ctr_off);
    L->sorted_ctr = L->gather_ctr + sorted_at;
    size_t off = ctr_off + d2d_align_up((size_t)L->gather_ctr_words * sizeof(int), 256);
    d2d_status rc = cudaMemsetAsync(L->slab, 0, off, st) == cudaSuccess ? D2D_OK : D2D_ERR_CUDA;
    for (const piece &p : pieces) {
        if (!p.src || rc != D2D_OK) continue;
        void *dst = (char *)L->slab + off;
        off += d2d_align_up(p.n * el, 256);
        *p.dst = dst;
        if (p.transpose) {
            rc = d2d_launch_transpose(p.src, dst, D.d, D.d_ff, el, st);
        } else if (cudaMemcpyAsync(dst, p.src, p.n * el, cudaMemcpyDeviceToDevice, st) != cudaSuccess) {
            rc = D2D_ERR_CUDA;
        }
        if (rc != D2D_OK) break;
    }
    if (rc == D2D_OK && want_cat) {
        L->w1g = (char *)L->slab + cat_off;
        rc = build_gate_cat(L, st);
    }
    if (rc == D2D_OK) rc = d2d_decode_ffn_maps(L);
    if (rc == D2D_OK && cudaStreamSynchronize(st) != cudaSuccess) rc = D2D_ERR_CUDA;
    if (rc == D2D_OK && (cudaStreamCreateWithFlags(&L->side_stream, cudaStreamNonBlocking) != cudaSuccess ||
                         cudaEventCreateWithFlags(&L->ev_fork, cudaEventDisableTiming) != cudaSuccess ||
                         cudaEventCreateWithFlags(&L->ev_join, cudaEventDisableTiming) != cudaSuccess))
        rc = D2D_ERR_CUDA;
    if (rc == D2D_OK) {
        bool ok = cudaStreamCreateWithFlags(&L->copy_in, cudaStreamNonBlocking) == cudaSuccess &&
                  cudaStreamCreateWithFlags(&L->copy_out, cudaStreamNonBlocking) == cudaSuccess &&
                  cudaEventCreateWithFlags(&L->ev_begin, cudaEventDisableTiming) == cudaSuccess &&
                  cudaEventCreateWithFlags(&L->ev_end, cudaEventDisableTiming) == cudaSuccess &&
                  cudaMallocHost((void **)&L->status_host, sizeof(int32_t) * d2d_layer::kHostChunks) == cudaSuccess;
        for (int c = 0; c < d2d_layer::kHostChunks && ok; ++c)
            ok = cudaEventCreateWithFlags(&L->ev_in[c], cudaEventDisableTiming) == cudaSuccess &&
                 cudaEventCreateWithFlags(&L->ev_done[c], cudaEventDisableTiming) == cudaSuccess;
        if (!ok) rc = D2D_ERR_CUDA;
    }
    if (rc != D2D_OK) {
        d2d_layer_destroy(L);
        return rc;
    }
    *out = L;
    return D2D_OK;
}

d2d_status d2d_layer_destroy(d2d_layer *layer)
{
    if (!layer) return D2D_OK;
    if (layer->ev_join) cudaEventDestroy(layer->ev_join);
    if (layer->ev_fork) cudaEventDestroy(layer->ev_fork);
    if (layer->side_stream) cudaStreamDestroy(layer->side_stream);
    for (int c = 0; c < d2d_layer::kHostChunks; ++c) {
        if (layer->ev_in[c]) cudaEventDestroy(layer->ev_in[c]);
        if (layer->ev_done[c]) cudaEventDestroy(layer->ev_done[c]);
    }
    if (layer->ev_begin) cudaEventDestroy(layer->ev_begin);
    if (layer->ev_end) cudaEventDestroy(layer->ev_end);
    if (layer->copy_in) cudaStreamDestroy(layer->copy_in);
    if (layer->copy_out) cudaStreamDestroy(layer->copy_out);
    if (layer->status_host) cudaFreeHost(layer->status_host);
    if (layer->q_slab) cudaFree(layer->q_slab);
    cudaError_t e = cudaFree(layer->slab);
    delete layer;
    return e == cudaSuccess ? D2D_OK : D2D_ERR_CUDA;
}

d2d_status d2d_layer_create_fp8(const d2d_layer_desc *desc, const d2d_weights *w, void *stream, d2d_layer **out)
{
    if (out) *out = nullptr;
    if (!desc || desc->dtype != D2D_BF16) return D2D_ERR_UNSUPPORTED;
    if (desc->d % 16 || ((int64_t)desc->expert_size * desc->d) % 16) return D2D_ERR_UNSUPPORTED;   // 16-byte pieces of codes
    d2d_layer *L = nullptr;
    d2d_status rc = d2d_layer_create(desc, w, stream, &L);
    if (rc != D2D_OK) return rc;
    const d2d_layer_desc &D = L->desc;
    cudaStream_t st = (cudaStream_t)stream;
    const size_t n_w = (size_t)D.d_ff * D.d, n_mat = D.gated ? 3 : 2;
    const size_t codes_b = d2d_align_up(n_w, 256), exps_b = d2d_align_up((size_t)D.n_experts * sizeof(int32_t), 256);
    if (cudaMalloc(&L->q_slab, n_mat * (codes_b + exps_b)) != cudaSuccess) {
        d2d_layer_destroy(L);
        return D2D_ERR_CUDA;
    }
    char *q = (char *)L->q_slab;
    L->q_w1 = (uint8_t *)q; L->q_k1 = (int32_t *)(q + codes_b); q += codes_b + exps_b;
    L->q_w2t = (uint8_t *)q; L->q_k2 = (int32_t *)(q + codes_b); q += codes_b + exps_b;
    if (D.gated) { L->q_wg = (uint8_t *)q; L->q_kg = (int32_t *)(q + codes_b); }
    const int per = D.expert_size * D.d;
    // the packed bf16 copies are replaced by the dequantised values, so every path of the layer computes with them
    rc = d2d_quantize_experts_e4m3(L->w1, L->q_w1, L->q_k1, D.n_experts, per, st);
    if (rc == D2D_OK) rc = d2d_quantize_experts_e4m3(L->w2t, L->q_w2t, L->q_k2, D.n_experts, per, st);
    if (rc == D2D_OK && D.gated) rc = d2d_quantize_experts_e4m3(L->w_gate, L->q_wg, L->q_kg, D.n_experts, per, st);
    if (rc == D2D_OK) rc = d2d_launch_transpose(L->w2t, L->w2, D.d_ff, D.d, L->elem, st);      // W2 [d, d_ff] from the transposed copy
    if (rc == D2D_OK && L->w1g) rc = build_gate_cat(L, st);
    if (rc == D2D_OK) rc = d2d_decode_ffn_maps(L);
    if (rc == D2D_OK && cudaStreamSynchronize(st) != cudaSuccess) rc = D2D_ERR_CUDA;
    if (rc != D2D_OK) {
        d2d_layer_destroy(L);
        return rc;
    }
    *out = L;
    return D2D_OK;
}

d2d_status d2d_layer_get_fp8(const d2d_layer *layer, int32_t which, uint8_t *codes, int32_t *exps, void *stream)
{
    if (!layer || which < 0 || which > 2 || (!codes && !exps)) return D2D_ERR_INVALID_ARG;
    const uint8_t *c = which == 0 ? layer->q_w1 : which == 1 ? layer->q_wg : layer->q_w2t;
    const int32_t *k = which == 0 ? layer->q_k1 : which == 1 ? layer->q_kg : layer->q_k2;
    if (!c || !k) return D2D_ERR_UNSUPPORTED;
    const d2d_layer_desc &D = layer->desc;
    cudaStream_t st = (cudaStream_t)stream;
    if (codes && cudaMemcpyAsync(codes, c, (size_t)D.d_ff * D.d, cudaMemcpyDeviceToDevice, st) != cudaSuccess) return D2D_ERR_CUDA;
    if (exps && cudaMemcpyAsync(exps, k, (size_t)D.n_experts * sizeof(int32_t), cudaMemcpyDeviceToDevice, st) != cudaSuccess) return D2D_ERR_CUDA;
    return D2D_OK;
}

d2d_status d2d_layer_set_expert_path(d2d_layer *layer, d2d_expert_path path, int32_t group, double rho_max)
{
    if (!layer || path < D2D_PATH_AUTO || path > D2D_PATH_FUSED || group < 0) return D2D_ERR_INVALID_ARG;
    if (path == D2D_PATH_FUSED) {
        // the group size applies to the fused kernel, whose groups hold at most 128 neurons
        const d2d_layer_desc &D = layer->desc;
        int g = d2d_gather_ffn_group_for(D);
        if (g <= 0) return D2D_ERR_UNSUPPORTED;
        if (group > 0) {
            const int gs = group * D.expert_size;
            if ((group & (group - 1)) || group > 32 || D.n_experts % group || gs % 16 || gs > 128) return D2D_ERR_UNSUPPORTED;
            g = group;
        }
        layer->fused_group = g;
        layer->expert_path = path;
        return D2D_OK;
    }
    const int g = d2d_gather_group_for(layer->desc, group);
    if (g <= 0 && (path == D2D_PATH_GATHER || group > 0)) return D2D_ERR_UNSUPPORTED;
    layer->gather_group = g;
    layer->expert_path = path;
    layer->gather_rho_max = rho_max >= 0.0 ? (rho_max > 1.0 ? 1.0 : rho_max) : -1.0;
    return D2D_OK;
}

d2d_status d2d_layer_set_fused_rho_max(d2d_layer *layer, double rho_max)
{
    if (!layer) return D2D_ERR_INVALID_ARG;
    if (layer->fused_group <= 0) return rho_max > 0.0 ? D2D_ERR_UNSUPPORTED : D2D_OK;
    layer->fused_rho_max = rho_max >= 0.0 ? (rho_max > 1.0 ? 1.0 : rho_max) : default_fused_rho_max(layer->fused_group);
    return D2D_OK;
}

d2d_status d2d_layer_expert_path_for(const d2d_layer *layer, int32_t T, int64_t n_sel, int32_t *path)
{
    if (!layer || !path || T <= 0 || n_sel < 0) return D2D_ERR_INVALID_ARG;
    const d2d_layer_desc &D = layer->desc;
    int p = layer->expert_path;
    if (p == D2D_PATH_FUSED && layer->fused_group <= 0) return D2D_ERR_UNSUPPORTED;
    if (p != D2D_PATH_FUSED && layer->gather_group <= 0) p = D2D_PATH_DENSE;
    if (p == D2D_PATH_AUTO) {
        const double up_flop = 2.0 * (double)T * D.d * D.d_ff * (D.gated ? 2.0 : 1.0);
        const double pairs = (double)T * (double)D.n_experts;
        const double rho_max = layer->gather_rho_max >= 0.0 ? layer->gather_rho_max : default_gather_rho_max(D, layer->gather_group, T);
        if (up_flop < auto_min_up_flop(layer)) p = D2D_PATH_DENSE;
        else if (layer->fused_group > 0 && layer->fused_rho_max > 0.0 && n_sel <= (long long)(layer->fused_rho_max * pairs)) p = D2D_PATH_FUSED;
        else if (n_sel <= (long long)(rho_max * pairs) || (layer->fused_group > 0 && n_sel <= (long long)(layer->fused_rho_max * pairs))) p = D2D_PATH_GATHER;
        else p = D2D_PATH_DENSE;
    }
    *path = p;
    return D2D_OK;
}

d2d_status d2d_layer_get_sorted(const d2d_layer *layer, int32_t T, int64_t *n_sel_max)
{
    if (!layer || !n_sel_max || T <= 0) return D2D_ERR_INVALID_ARG;
    *n_sel_max = use_dense_masked(layer, T) ? sorted_n_sel_max(layer, T, false) : -1;
    return D2D_OK;
}

d2d_status d2d_decode_plan_for(const d2d_layer_desc *desc, int32_t n_layers, int32_t T, int32_t fp8_experts, d2d_decode_plan *plan)
{
    if (!desc || !plan || n_layers < 1 || n_layers > D2D_MAX_GROUP || T < 1) return D2D_ERR_INVALID_ARG;
    if (desc->d <= 0 || desc->d_ff <= 0 || desc->n_experts <= 0 || desc->expert_size <= 0 || desc->d_h <= 0 ||
        (int64_t)desc->n_experts * desc->expert_size != desc->d_ff)
        return D2D_ERR_INVALID_ARG;
    d2d_decode_plan p = {};
    if (!d2d_decode_ffn_plan(*desc, n_layers, T, fp8_experts != 0, &p)) return D2D_ERR_UNSUPPORTED;
    p.router = d2d_decode_router_supports(*desc, T) ? 1 : 0;
    *plan = p;
    return D2D_OK;
}

d2d_status d2d_layer_get_fused(const d2d_layer *layer, int32_t *group, double *rho_max)
{
    if (!layer) return D2D_ERR_INVALID_ARG;
    if (group) *group = layer->fused_group;
    if (rho_max) *rho_max = layer->fused_rho_max;
    return D2D_OK;
}

d2d_status d2d_layer_get_expert_path(const d2d_layer *layer, int32_t *path, int32_t *group, double *rho_max)
{
    if (!layer) return D2D_ERR_INVALID_ARG;
    if (path) *path = layer->expert_path;
    if (group) *group = layer->expert_path == D2D_PATH_FUSED ? layer->fused_group : layer->gather_group;
    if (rho_max) *rho_max = layer->gather_rho_max;
    return D2D_OK;
}

d2d_status d2d_layer_reset_counters(d2d_layer *layer, void *stream)
{
    if (!layer) return D2D_ERR_INVALID_ARG;
    const size_t bytes = 256 + d2d_align_up((size_t)layer->gather_ctr_words * sizeof(int), 256);
    return cudaMemsetAsync(layer->slab, 0, bytes, (cudaStream_t)stream) == cudaSuccess ? D2D_OK : D2D_ERR_CUDA;
}

size_t d2d_workspace_bytes(const d2d_layer *layer, int32_t max_tokens)
{
    if (!layer || max_tokens < 0) return 0;
    return d2d_largest_up_to(max_tokens, [&](int T) { return layout_for(layer, T).total; });
}

size_t d2d_select_workspace_bytes(int32_t T, int32_t E)
{
    if (T < 0 || E <= 0) return 0;
    return d2d_select_ws_bytes(T, E);
}

d2d_status d2d_router_fwd(const d2d_layer *layer, const void *x, int32_t T, float *R,
                          void *ws, size_t ws_bytes, void *stream)
{
    if (!layer || T < 0) return D2D_ERR_INVALID_ARG;
    if (T == 0) return D2D_OK;
    if (!x || !R || !ws || !aligned16(x) || !aligned16(R) || !aligned16(ws)) return D2D_ERR_INVALID_ARG;
    const ws_layout w = layout_for(layer, T);
    if (ws_bytes < w.total) return D2D_ERR_WORKSPACE;
    return d2d_launch_router(layer, x, T, R, (float *)((char *)ws + w.u_off), (cudaStream_t)stream);
}

static d2d_status select_common(const float *R, int32_t T, int32_t E, float tau, int topk, d2d_routing *out,
                                void *ws, size_t ws_bytes, void *stream, bool mask_is_input)
{
    if (T < 0 || E <= 0 || !routing_ok(out, false)) return D2D_ERR_INVALID_ARG;
    if (!mask_is_input && T > 0 && (!R || !aligned16(R))) return D2D_ERR_INVALID_ARG;
    if (!mask_is_input && topk == 0 && !(tau >= 0.0f && tau <= 1.0f)) return D2D_ERR_INVALID_ARG;   // also rejects NaN
    if (topk < 0 || (topk > 0 && E > 2048)) return topk < 0 ? D2D_ERR_INVALID_ARG : D2D_ERR_UNSUPPORTED;
    if (T > 0 && (!ws || ws_bytes < d2d_select_ws_bytes(T, E))) return D2D_ERR_WORKSPACE;
    return d2d_launch_select(mask_is_input ? nullptr : R, T, E, tau, topk, out, ws, (cudaStream_t)stream);
}

d2d_status d2d_select_dynk(const float *R, int32_t T, int32_t E, float tau, d2d_routing *out,
                           void *ws, size_t ws_bytes, void *stream)
{
    return select_common(R, T, E, tau, 0, out, ws, ws_bytes, stream, false);
}

d2d_status d2d_select_topk(const float *R, int32_t T, int32_t E, int32_t kk, d2d_routing *out,
                           void *ws, size_t ws_bytes, void *stream)
{
    if (kk <= 0) return D2D_ERR_INVALID_ARG;
    return select_common(R, T, E, 0.0f, kk, out, ws, ws_bytes, stream, false);
}

d2d_status d2d_routing_from_mask(int32_t T, int32_t E, d2d_routing *out, void *ws, size_t ws_bytes, void *stream)
{
    return select_common(nullptr, T, E, 0.0f, 0, out, ws, ws_bytes, stream, true);
}

d2d_status d2d_routing_of_mask(const uint32_t *mask, int32_t T, int32_t E, d2d_routing *out, void *ws, size_t ws_bytes, void *stream)
{
    if (T < 0 || E <= 0 || !routing_ok(out, false) || (T > 0 && !mask)) return D2D_ERR_INVALID_ARG;
    if (T > 0 && (!ws || ws_bytes < d2d_select_ws_bytes(T, E))) return D2D_ERR_WORKSPACE;
    if (T == 0) return d2d_launch_select(nullptr, 0, E, 0.0f, 0, out, ws, (cudaStream_t)stream);
    return d2d_launch_select_mask_of(mask, T, E, out, ws, (cudaStream_t)stream);
}

d2d_status d2d_moe_ffn_fwd(const d2d_layer *layer, const void *x, int32_t T, const d2d_routing *routing,
                           void *y, void *ws, size_t ws_bytes, void *stream)
{
    if (!layer || T < 0) return D2D_ERR_INVALID_ARG;
    if (T == 0) return D2D_OK;
    if (!x || !y || !aligned16(x) || !aligned16(y) || !routing_ok(routing, false)) return D2D_ERR_INVALID_ARG;
    const ws_layout w = layout_for(layer, T);
    if (!ws || ws_bytes < w.total) return D2D_ERR_WORKSPACE;
    return d2d_launch_moe_ffn(layer, x, T, routing, y, (char *)ws + w.ffn_off, w.total - w.ffn_off,
                              (cudaStream_t)stream);
}

d2d_status d2d_expert_up_fwd(const d2d_layer *layer, const void *x, int32_t T, const d2d_routing *routing,
                             void *H, void *stream)
{
    if (!layer || T < 0) return D2D_ERR_INVALID_ARG;
    if (T == 0) return D2D_OK;
    if (!x || !H || !aligned16(x) || !aligned16(H) || !routing_ok(routing, false)) return D2D_ERR_INVALID_ARG;
    if (layer->desc.dtype != D2D_BF16 || layer->desc.d_ff % 8 || !d2d_gemm_tc_available()) return D2D_ERR_UNSUPPORTED;
    d2d_gemm_args up = dense_up_args(layer, x, T, routing, H);
    up.test_skip_load = __atomic_exchange_n(&g_test_fault, 0, __ATOMIC_RELAXED) == 1;
    return d2d_gemm_tc(up, (cudaStream_t)stream);
}

d2d_status d2d_test_inject_fault(int32_t kind)
{
    if (kind != 0 && kind != 1) return D2D_ERR_INVALID_ARG;
    __atomic_store_n(&g_test_fault, kind, __ATOMIC_RELAXED);
    return D2D_OK;
}

d2d_status d2d_expert_up_gather_fwd(const d2d_layer *layer, const void *x, int32_t T, const d2d_routing *routing,
                                    void *H, void *stream)
{
    if (!layer || T < 0) return D2D_ERR_INVALID_ARG;
    if (T == 0) return D2D_OK;
    if (!x || !H || !aligned16(x) || !aligned16(H) || !routing_ok(routing, false)) return D2D_ERR_INVALID_ARG;
    if (layer->gather_group <= 0) return D2D_ERR_UNSUPPORTED;
    const d2d_layer_desc &D = layer->desc;
    d2d_gather_args ga = {};
    ga.x = x; ga.w1 = layer->w1; ga.w_gate = D.gated ? layer->w_gate : nullptr; ga.b1 = layer->b1; ga.mask = routing->mask; ga.H = H;
    ga.T = T; ga.d = D.d; ga.d_ff = D.d_ff; ga.n_experts = D.n_experts; ga.s = D.expert_size; ga.g = layer->gather_group;
    ga.act = D.act; ga.status = routing->status; ga.ctr = layer->gather_ctr;
    ga.n_sel = routing->n_sel; ga.n_sel_min = -1; ga.n_sel_max = LLONG_MAX;
    return d2d_moe_gather_up(ga, (cudaStream_t)stream);
}

d2d_status d2d_expert_down_masked_fwd(const d2d_layer *layer, const void *H, int32_t T, const d2d_routing *routing, void *y,
                                      void *stream)
{
    if (!layer || T < 0) return D2D_ERR_INVALID_ARG;
    if (T == 0) return D2D_OK;
    if (!H || !y || !aligned16(H) || !aligned16(y) || !routing_ok(routing, true)) return D2D_ERR_INVALID_ARG;
    if (!d2d_moe_down_masked_supports(layer->desc)) return D2D_ERR_UNSUPPORTED;
    return d2d_moe_down_masked(layer->desc, H, routing->mask, layer->w2, layer->b2, y, T, routing->status, (cudaStream_t)stream);
}

d2d_status d2d_expert_down_fwd(const d2d_layer *layer, const void *H, int32_t T, void *y, int32_t *status, void *stream)
{
    if (!layer || T < 0) return D2D_ERR_INVALID_ARG;
    if (T == 0) return D2D_OK;
    if (!H || !y || !aligned16(H) || !aligned16(y)) return D2D_ERR_INVALID_ARG;
    if (layer->desc.dtype != D2D_BF16 || layer->desc.d_ff % 8 || !d2d_gemm_tc_available()) return D2D_ERR_UNSUPPORTED;
    return d2d_gemm_tc(dense_down_args(layer, H, T, y, status), (cudaStream_t)stream);
}

// The forms of a layer call, in the order in which they are tried.
enum layer_form {
    FORM_DECODE,             // decode batches: cluster router with selection and lists, streaming experts
    FORM_FUSED_ROUTER,       // router and mask in one kernel, tensor-core experts, lists beside them
    FORM_FUSED_ROUTER_LISTS, // the same router, then the lists, then experts that walk them
    FORM_F32_SMALL,          // float32 layers that fit one SM's shared memory: one launch
    FORM_TOKEN_FUSED,        // other small float32 problems: one launch
    FORM_SMALL_ROUTER,       // decode batches the streaming kernels do not take: router that selects as well
    FORM_MASKED,             // hidden layer, then scores and selection; tensor-core experts, lists beside them
    FORM_PLAIN,              // scores, selection, experts, one after the other
};

static layer_form form_for(const d2d_layer *L, int T, bool lists)
{
    const d2d_layer_desc &D = L->desc;
    const bool masked = use_dense_masked(L, T) && !use_small_ffn(L, T);
    if (d2d_decode_router_supports(D, T) && d2d_use_decode_ffn(L, 1, T)) return FORM_DECODE;
    if (d2d_router_fused_supports(D, T)) return masked ? FORM_FUSED_ROUTER : FORM_FUSED_ROUTER_LISTS;
    if (d2d_layer_f32_small_supports(D, T, lists)) return FORM_F32_SMALL;
    if (T > 8 && d2d_layer_token_fused_supports(D, T, lists)) return FORM_TOKEN_FUSED;
    if (lists && d2d_small_router_supports(D, T)) return FORM_SMALL_ROUTER;
    // (Also where one CTA could select, which would take a kernel more and a pass over the batch, and where the cluster router could
    // score: behind the router in two kernels the up projection starts at once.)
    if (masked && (!d2d_small_select_supports(T, D.n_experts) || d2d_router_scores_supports(D, T))) return FORM_MASKED;
    return FORM_PLAIN;
}

// Whether the form's expert kernels walk the per-expert lists (the others read the mask, and build the lists if they are wanted)
// or have always been called with them (up to 64 tokens of a router in two kernels)
static bool needs_lists(const d2d_layer *L, int T, layer_form f)
{
    return f == FORM_FUSED_ROUTER_LISTS || f == FORM_SMALL_ROUTER || f == FORM_PLAIN ||
           (f == FORM_MASKED && d2d_small_select_supports(T, L->desc.n_experts));
}

// The per-expert lists on the layer's side stream, behind what is queued on `st`
static d2d_status fork_lists(const d2d_layer *L, int T, d2d_routing *r, void *ws, cudaStream_t st)
{
    if (cudaEventRecord(L->ev_fork, st) != cudaSuccess || cudaStreamWaitEvent(L->side_stream, L->ev_fork, 0) != cudaSuccess) return D2D_ERR_CUDA;
    return d2d_launch_select(nullptr, T, L->desc.n_experts, 0.0f, 0, r, ws, L->side_stream, 1, L->tickets + 48);
}
static d2d_status join_lists(const d2d_layer *L, cudaStream_t st)
{
    return cudaEventRecord(L->ev_join, L->side_stream) == cudaSuccess && cudaStreamWaitEvent(st, L->ev_join, 0) == cudaSuccess ? D2D_OK : D2D_ERR_CUDA;
}

// Whether the down projection builds the lists on the side: the dense pair, few tokens, no token-major dual
static bool lists_ride(const d2d_layer *L, int T, const d2d_routing *r)
{
    const d2d_layer_desc &D = L->desc;
    return !r->tok_off && path_before_launch(L, T, true) == D2D_PATH_DENSE &&
           d2d_lists_ride(T, D.n_experts, d2d_gemm_tc_splits(T, D.d, D.d_ff), 2.0 * T * D.d * D.d_ff);
}

d2d_status d2d_layer_fwd(const d2d_layer *layer, const void *x, int32_t T, float tau, void *y,
                         float *R_out, d2d_routing *routing, void *ws, size_t ws_bytes, void *stream)
{
    if (!layer || T < 0 || !routing_ok(routing, true)) return D2D_ERR_INVALID_ARG;
    if (!(tau >= 0.0f && tau <= 1.0f)) return D2D_ERR_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    const int E = layer->desc.n_experts;
    const bool lists = has_lists(routing);
    bool fork = false, ride = false;                         // lists beside the experts: on the side stream, or by the down projection
    if (T == 0) return lists ? d2d_launch_select(nullptr, 0, E, tau, 0, routing, ws, st) : D2D_OK;
    if (!x || !y || !aligned16(x) || !aligned16(y) || (R_out && !aligned16(R_out))) return D2D_ERR_INVALID_ARG;
    const ws_layout w = layout_for(layer, T);
    if (!ws || !aligned16(ws) || ws_bytes < w.total) return D2D_ERR_WORKSPACE;
    const layer_form form = form_for(layer, T, lists);
    if (!lists && needs_lists(layer, T, form)) return D2D_ERR_INVALID_ARG;
    char *base = (char *)ws;
    float *R = R_out ? R_out : (float *)(base + w.r_off);
    void *ffn_ws = base + w.ffn_off;
    const size_t ffn_bytes = w.total - w.ffn_off;
    // the fused routers and router_scores also add up k: the number of selected pairs, which decides between the two up projections
    int32_t *ksum = (int32_t *)(layer->tickets + 40);
    d2d_status rc;
    switch (form) {
    case FORM_DECODE: return d2d_decode_layers(&layer, 1, x, T, tau, routing, R_out, &ffn_ws, y, st);
    case FORM_F32_SMALL: return d2d_layer_f32_small(layer, x, T, tau, y, R_out, routing, lists, layer->tickets + 52, st);
    case FORM_TOKEN_FUSED:
        if (cudaMemsetAsync(routing->status, 0, sizeof(int32_t), st) != cudaSuccess) return D2D_ERR_CUDA;
        return d2d_layer_token_fused(layer, x, T, tau, y, R_out, routing, lists, layer->tickets + 52, st);
    case FORM_FUSED_ROUTER:
        // The scores are written only when the caller asked for them: mask and k come out of the same kernel.  The tensor-core
        // expert kernels read only the mask: the per-expert lists (when the caller wants them) are built on the side stream while
        // they run (the small metadata CTAs fit beside the persistent CTAs), join at the end.
        rc = d2d_router_fused(layer, x, T, tau, 1, R_out, routing->mask, routing->k, routing->status, st, ksum);
        ride = lists && lists_ride(layer, T, routing);
        fork = lists && !ride;
        if (rc == D2D_OK && fork) rc = fork_lists(layer, T, routing, base + w.sel_off, st);
        if (rc != D2D_OK) return rc;
        // tile counter of the up projection: layer-owned, zero at creation and reset by the kernel that used it, so no memset node
        // sits in front of the router (the up projection may begin while the router is still running)
        rc = d2d_launch_moe_ffn(layer, x, T, routing, y, ffn_ws, ffn_bytes, st, (int *)(layer->tickets + 32), 0, ksum + 4, ride);
        return fork && join_lists(layer, st) != D2D_OK ? D2D_ERR_CUDA : rc;
    case FORM_FUSED_ROUTER_LISTS:
        if (cudaMemsetAsync(routing->status, 0, sizeof(int32_t), st) != cudaSuccess) return D2D_ERR_CUDA;
        rc = d2d_router_fused(layer, x, T, tau, 1, R_out, routing->mask, routing->k, routing->status, st, nullptr);
        if (rc == D2D_OK) rc = d2d_launch_select(nullptr, T, E, tau, 0, routing, base + w.sel_off, st, 1);
        break;
    case FORM_SMALL_ROUTER: {
        // the router kernel's last CTA selects as well (one launch for router + selection)
        const bool small = use_small_ffn(layer, T);
        float *y32 = (float *)(base + w.ffn_off + 256);
        rc = d2d_small_router(layer, x, T, R, base + w.u_off, st, routing, tau, 1, small ? y32 : nullptr, small ? T * layer->desc.d : 0);
        if (rc != D2D_OK) return rc;
        return d2d_launch_moe_ffn(layer, x, T, routing, y, ffn_ws, ffn_bytes, st, nullptr, small ? 1 : 0);
    }
    case FORM_MASKED:
        // router shapes the fused kernel does not take: the hidden layer by a GEMM, then scores, mask, k and the number of selected
        // pairs by one kernel (two where the scores do not fit it); lists as above
        if (d2d_router_scores_supports(layer->desc, T)) {
            rc = d2d_router_scores(layer, x, base + w.u_off + 256, T, tau, R_out, routing->mask, routing->k, routing->status, st, ksum);
        } else {
            rc = d2d_launch_router(layer, x, T, R, (float *)(base + w.u_off), st);
            if (rc == D2D_OK) rc = d2d_launch_dynk_mask(R, T, E, tau, routing, ksum, st);
        }
        ride = lists && lists_ride(layer, T, routing);
        fork = lists && !ride;
        if (rc == D2D_OK && fork) rc = fork_lists(layer, T, routing, base + w.sel_off, st);
        if (rc != D2D_OK) return rc;
        rc = d2d_launch_moe_ffn(layer, x, T, routing, y, ffn_ws, ffn_bytes, st,
                                d2d_router_scores_supports(layer->desc, T) ? (int *)(layer->tickets + 32) : nullptr, 0, ksum + 4, ride);
        return fork && join_lists(layer, st) != D2D_OK ? D2D_ERR_CUDA : rc;
    case FORM_PLAIN:
        rc = d2d_launch_router(layer, x, T, R, (float *)(base + w.u_off), st);
        if (rc == D2D_OK) rc = d2d_launch_select(R, T, E, tau, 0, routing, base + w.sel_off, st);
        break;
    }
    if (rc != D2D_OK) return rc;
    return d2d_launch_moe_ffn(layer, x, T, routing, y, ffn_ws, ffn_bytes, st);
}

// Ends a host call: its n status words come back with everything else queued on `st` (a blocking copy after the
// synchronisation was a second round trip of 10 us); returns the largest (0 = ok).
static d2d_status finish_host_call(const d2d_layer *layer, const int32_t *status_dev, int n, cudaStream_t st)
{
    D2D_CUDA_TRY(cudaMemcpyAsync(layer->status_host, status_dev, sizeof(int32_t) * (size_t)n, cudaMemcpyDeviceToHost, st));
    D2D_CUDA_TRY(cudaStreamSynchronize(st));
    int32_t worst = 0;
    for (int i = 0; i < n; ++i) worst = layer->status_host[i] > worst ? layer->status_host[i] : worst;
    return (d2d_status)worst;
}

// Whether a batch can do without the per-expert lists
static bool lists_optional(const d2d_layer *L, int T) { return !needs_lists(L, T, form_for(L, T, false)); }

// Carves routing buffers + x/y staging + the layer workspace out of one device buffer.
struct host_call_layout {
    size_t x_off, y_off, mask_off, k_off, counts_off, offsets_off, perm_off, scalars_off, ws_off;      // the layer's workspace is last
};

static host_call_layout host_layout(const d2d_layer *L, int T)
{
    host_call_layout h;
    const size_t Tn = (size_t)(T > 0 ? T : 1), E = (size_t)L->desc.n_experts, W = (E + 31) / 32;
    size_t off = 0;
    auto take = [&](size_t bytes) { size_t o = off; off += d2d_align_up(bytes, 256); return o; };
    h.x_off = take(Tn * L->desc.d * L->elem);
    h.y_off = take(Tn * L->desc.d * L->elem);
    h.mask_off = take(Tn * W * 4);
    h.k_off = take(Tn * 4);
    h.counts_off = take(E * 4);
    h.offsets_off = take((E + 1) * 4);
    h.perm_off = take(Tn * E * 4);
    h.scalars_off = take((2 + d2d_layer::kHostChunks) * 4);     // n_sel, then one status word per chunk
    h.ws_off = off;
    return h;
}

size_t d2d_layer_fwd_host_workspace_bytes(const d2d_layer *layer, int32_t max_tokens)
{
    if (!layer || max_tokens < 0) return 0;
    return host_layout(layer, max_tokens).ws_off + d2d_workspace_bytes(layer, max_tokens > 0 ? max_tokens : 1);      // chunks are smaller batches
}

// How a host call cuts T tokens: bounds[0 .. chunks], returns the number of chunks.  Which of the three legs (copy in, layer, copy out) is
// the slowest decides: a bf16 token's FLOP take as long as its bytes over PCIe (54 GB/s) with 18000 hidden neurons times matrices at
// 0.97 PFLOP/s, with 26000 at the sustained 1.4, which batches of a chunk's size do not reach.  At 18432 (d = 1536, plain) both cuts are
// level (us, equal chunks / sizes by the layer: 1600 tokens 258 / 256, 3600 412 / 405); float32 layers take the equal ones, since each
// chunk costs them most of a round of CTAs (d = 512, d_ff = 9216: 1600 tokens 7328 in two / 8091, 2000 8367 / 9519).
static int cut_host_batch(const d2d_layer *L, int T, int *bounds)
{
    const size_t row_bytes = (size_t)T * L->desc.d * L->elem;
    // Under 3 MB two chunks pay where there are many narrow rows, from 2 MB on (us, one / two chunks: d = 256, 4000 tokens 128 / 115,
    // 5800 160 / 139; d = 128, 6000 102 / 99, 12000 162 / 143; float32, d = 64, 12000 458 / 420; d = 128, 3600 667 / 717, 6000 1006 / 1031)
    const bool large = row_bytes >= ((size_t)3 << 20);
    if (T < 1024 || !(large || (T >= 3584 && row_bytes >= ((size_t)2 << 20)))) return 1;
    int n_chunks = 2, first = 0, middle = 0;                 // sizes: first, middle, .., middle, the rest
    if (L->desc.dtype == D2D_BF16 && large && (L->desc.gated ? 3 : 2) * (int64_t)L->desc.d_ff >= 18000) {
        // The layer: the call takes about (copy-in of the first chunk) + (all layer calls) + (copy-out of the last), if a chunk is
        // copied in while the layer works on the one before and out while it works on the next: sizes may grow and shrink by the
        // ratio of the two times, 1.3.  Multiples of 256, the rows of a pair's tile.  Llama-shaped layer, us, sizes of before (3/16,
        // 5/16, 5/16, 3/16 from 3584 tokens on, two or three equal ones below) / these: 8192 tokens 2288 / 2187, 6000 1734 / 1684, 4096
        // 1209 / 1139, 3400 1082 / 958, 2500 944 / 773, 2000 710 / 678; two of 512 443 at 1024 tokens, three 482.
        n_chunks = T >= 3328 ? 4 : T >= 1536 ? 3 : 2;
        auto round256 = [](int v) { return v < 384 ? 256 : (v + 128) / 256 * 256; };
        first = n_chunks == 2 ? d2d_cdiv(d2d_cdiv(T, 2), 128) * 128 : round256((n_chunks == 4 ? 7 : 10) * (T / 32));
        middle = n_chunks == 2 ? first : round256((T - 2 * first) / (n_chunks - 2));
    } else {
        // The copies: equal chunks, as many as pay for their launches.  us with 2 / 3 / 4, GPT-2-medium-shaped layer: 2048 tokens 192 /
        // 207 / 215, 3000 256 / 245 / 258, 3450 - / 265 / 284, 3600 302 / 290 / 269, 6000 464 / 423 / 390; BERT-shaped: 3000 203 / 201 / 216,
        // 4096 256 / 236 / 247, 4500 - / 253 / 257, 4800 293 / 268 / 256, 6000 364 / 328 / 307; d = 256: 8000 tokens 179 / 166 / 186, 13000
        // 264 / 251 / 232.
        n_chunks = row_bytes > ((size_t)7 << 20) ? 4 : large && T >= 2560 ? 3 : 2;
        first = middle = d2d_cdiv(d2d_cdiv(T, n_chunks), 128) * 128;
    }
    for (int c = 1; c < n_chunks; ++c) bounds[c] = first + (c - 1) * middle < T ? first + (c - 1) * middle : T;
    return n_chunks;
}

d2d_status d2d_layer_fwd_host(const d2d_layer *layer, const void *x_host, int32_t T, float tau, void *y_host,
                              void *ws, size_t ws_bytes, void *stream)
{
    if (!layer || T < 0) return D2D_ERR_INVALID_ARG;
    if (T == 0) return D2D_OK;
    if (!x_host || !y_host || !ws || !aligned16(ws)) return D2D_ERR_INVALID_ARG;
    const host_call_layout h = host_layout(layer, T);
    cudaStream_t st = (cudaStream_t)stream;
    char *base = (char *)ws;
    const size_t tok_bytes = (size_t)layer->desc.d * layer->elem;
    const size_t row_bytes = (size_t)T * tok_bytes;
    d2d_routing r;
    memset(&r, 0, sizeof(r));
    r.mask = (uint32_t *)(base + h.mask_off);
    r.k = (int32_t *)(base + h.k_off);
    r.counts = (int32_t *)(base + h.counts_off);
    r.offsets = (int32_t *)(base + h.offsets_off);
    r.perm = (int32_t *)(base + h.perm_off);
    r.n_sel = (int32_t *)(base + h.scalars_off);
    r.status = r.n_sel + 1;
    r.perm_capacity = (int64_t)T * layer->desc.n_experts;
    // Tokens are independent, so a large batch is cut into chunks (multiples of 128 tokens) and pipelined: the copy of
    // chunk c+1 to the device (copy-in stream), the layer on chunk c (`stream`) and the copy of chunk c-1 back to the
    // host (copy-out stream) run at the same time; PCIe carries both directions at once.  The routing buffers and the
    // layer workspace are reused chunk after chunk, which is safe because the layer calls are serial on `stream`.
    int bounds[d2d_layer::kHostChunks + 1] = {0, T, T, T, T};
    int n_chunks = cut_host_batch(layer, T, bounds);
    if (const char *e = getenv("D2D_HOST_CHUNKS")) {          // 1 .. 4 equal chunks, for tuning
        const int n = atoi(e);
        if (n >= 1 && n <= d2d_layer::kHostChunks && T >= 128 * n) {
            n_chunks = n;
            const int chunk = d2d_cdiv(d2d_cdiv(T, n), 128) * 128;
            for (int c = 1; c <= d2d_layer::kHostChunks; ++c) bounds[c] = c * chunk < T && c < n ? c * chunk : T;
        }
    }
    size_t layer_bytes = layout_for(layer, T).total;
    for (int c = 0; n_chunks > 1 && c < n_chunks; ++c) {
        const size_t n = layout_for(layer, bounds[c + 1] - bounds[c]).total;
        if (n > layer_bytes) layer_bytes = n;
    }
    if (ws_bytes < h.ws_off + layer_bytes) return D2D_ERR_WORKSPACE;
    if (n_chunks == 1) {
        D2D_CUDA_TRY(cudaMemcpyAsync(base + h.x_off, x_host, row_bytes, cudaMemcpyHostToDevice, st));
        if (lists_optional(layer, T)) r.counts = r.offsets = r.perm = r.n_sel = nullptr;      // nobody sees them
        d2d_status rc = d2d_layer_fwd(layer, base + h.x_off, T, tau, base + h.y_off, nullptr, &r,
                                      base + h.ws_off, layer_bytes, st);
        if (rc != D2D_OK) return rc;
        D2D_CUDA_TRY(cudaMemcpyAsync(y_host, base + h.y_off, row_bytes, cudaMemcpyDeviceToHost, st));
        return finish_host_call(layer, r.status, 1, st);
    }
    // the copies may not start before work already queued on `stream` (which may still use ws) has finished
    D2D_CUDA_TRY(cudaEventRecord(layer->ev_begin, st));
    D2D_CUDA_TRY(cudaStreamWaitEvent(layer->copy_in, layer->ev_begin, 0));
    D2D_CUDA_TRY(cudaStreamWaitEvent(layer->copy_out, layer->ev_begin, 0));
    for (int c = 0; c < n_chunks; ++c) {
        const int t0 = bounds[c], tc = bounds[c + 1] - bounds[c];
        if (tc <= 0) continue;
        D2D_CUDA_TRY(cudaMemcpyAsync(base + h.x_off + (size_t)t0 * tok_bytes, (const char *)x_host + (size_t)t0 * tok_bytes,
                                     (size_t)tc * tok_bytes, cudaMemcpyHostToDevice, layer->copy_in));
        D2D_CUDA_TRY(cudaEventRecord(layer->ev_in[c], layer->copy_in));
    }
    d2d_status rc = D2D_OK;
    int32_t *const status0 = r.status, *const counts = r.counts, *const offsets = r.offsets, *const perm = r.perm, *const n_sel = r.n_sel;
    int n_used = 0;
    for (int c = 0; c < n_chunks; ++c) {
        const int t0 = bounds[c], tc = bounds[c + 1] - bounds[c];
        if (tc <= 0) continue;
        r.status = status0 + n_used;                         // one status word per chunk (the layer call clears its own)
        ++n_used;
        const bool lists = !lists_optional(layer, tc);       // nobody sees them
        r.counts = lists ? counts : nullptr;
        r.offsets = lists ? offsets : nullptr;
        r.perm = lists ? perm : nullptr;
        r.n_sel = lists ? n_sel : nullptr;
        D2D_CUDA_TRY(cudaStreamWaitEvent(st, layer->ev_in[c], 0));
        rc = d2d_layer_fwd(layer, base + h.x_off + (size_t)t0 * tok_bytes, tc, tau, base + h.y_off + (size_t)t0 * tok_bytes,
                           nullptr, &r, base + h.ws_off, layer_bytes, st);
        if (rc != D2D_OK) break;
        D2D_CUDA_TRY(cudaEventRecord(layer->ev_done[c], st));
        D2D_CUDA_TRY(cudaStreamWaitEvent(layer->copy_out, layer->ev_done[c], 0));
        D2D_CUDA_TRY(cudaMemcpyAsync((char *)y_host + (size_t)t0 * tok_bytes, base + h.y_off + (size_t)t0 * tok_bytes,
                                     (size_t)tc * tok_bytes, cudaMemcpyDeviceToHost, layer->copy_out));
    }
    // join both copy streams back into `stream` (also on the error path, so nothing is left running on them)
    cudaEventRecord(layer->ev_end, layer->copy_out);
    cudaStreamWaitEvent(st, layer->ev_end, 0);
    cudaEventRecord(layer->ev_end, layer->copy_in);
    cudaStreamWaitEvent(st, layer->ev_end, 0);
    if (rc != D2D_OK) return rc;
    return finish_host_call(layer, status0, n_used, st);
}

}  // extern "C"
