"""Work that users of the dynamic-k MoE layer have it do, through the public entry points of `api`.

A layer replaces a Transformer FFN or an attention projection at inference time, so what is called in earnest is
decoding (a token per running sequence), prefill and encoder batches (all tokens of the prompts or images at once), the
Q/K/V projections of one attention layer as a group, the latency protocol with given gating decisions, and the
host-buffer call of a program whose activations live in host memory.  Shapes, thresholds and distributions are those of
`workloads.CONFIGS`; weights and tokens are drawn on the GPU.

A case: `call` ("layer" | "group" | "mask" | "host"), `shape` (a name in CONFIGS), `T` tokens, `tau` (or `p`, the
Bernoulli probability of "mask"), `fp8` (8-bit expert weights), `layers` (of a group), `fresh` (the caller leaves the
output buffers to the call instead of keeping them).
"""
import math

import torch

from paper_2310_04361_b200 import api, workloads

DEVICE = "cuda:0"


def _case(call, shape, T, tau=0.0, p=0.0, fp8=False, layers=1, fresh=False):
    return {"call": call, "shape": shape, "T": int(T), "tau": float(tau), "p": float(p), "fp8": bool(fp8),
            "layers": int(layers), "fresh": bool(fresh)}


def listed():
    return [dict(c, name=name) for name, c in [
        # one user's decode step through a GPT-2-medium-sized FFN: latency and launches only
        ("gpt2_ffn decode 1", _case("layer", "gpt2_ffn", 1, 0.5)),
        # a decode step of a server with an odd number of running sequences
        ("gpt2_ffn decode 13", _case("layer", "gpt2_ffn", 13, 0.5)),
        # the prefill of one ragged prompt, by a program that keeps no buffers between calls
        ("gpt2_ffn prefill 333", _case("layer", "gpt2_ffn", 333, 0.2, fresh=True)),
        # Q, K and V of a converted attention layer in a small decode batch
        ("gpt2_attn qkv 8", _case("group", "gpt2_attn", 8, 0.5, layers=3)),
        # one user's decode step through a Llama-sized gated FFN with 8-bit expert weights: bytes of the kept experts
        ("llama fp8 decode 1", _case("layer", "llama", 1, 0.2, fp8=True)),
        # a small decode batch of the same layer with bf16 weights
        ("llama decode 7", _case("layer", "llama", 7, 0.2)),
        # the smallest float32 layer
        ("tiny f32 128", _case("layer", "tiny", 128, 0.5)),
        # an encoder batch: 32 sequences of 128 tokens
        ("bert 4096", _case("layer", "bert", 4096, 0.3)),
        # an image batch: 128 images of 197 tokens (a ragged last tile)
        ("vit 25216", _case("layer", "vit", 25216, 0.3)),
        # the headline: a Llama-sized prefill batch
        ("llama prefill 8192", _case("layer", "llama", 8192, 0.4)),
        # the latency protocol of the paper's Sec. 4.4: gating decisions given as a mask
        ("paper mask 50432", _case("mask", "paper", 50432, p=0.1)),
        # the headline batch from and to page-locked host memory
        ("llama host 8192", _case("host", "llama", 8192, 0.4)),
    ]]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["decode", "prefill", "encoder", "llama", "group", "fp8", "f32", "mask", "host"])
    fresh = rng.random() < 0.25
    tau = round(rng.uniform(0.2, 0.7), 3)
    if kind == "decode":
        return _case("layer", rng.choice(["gpt2_ffn", "gpt2_attn"]), _log_int(rng, 1, 64), tau, fresh=fresh)
    if kind == "prefill":
        return _case("layer", rng.choice(["gpt2_ffn", "gpt2_attn"]), _log_int(rng, 65, 4096), tau, fresh=fresh)
    if kind == "encoder":
        return _case("layer", rng.choice(["bert", "vit"]), _log_int(rng, 128, 25216), tau, fresh=fresh)
    if kind == "llama":
        return _case("layer", "llama", _log_int(rng, 1, 6144), tau)
    if kind == "group":
        return _case("group", "gpt2_attn", _log_int(rng, 1, 512), tau, layers=rng.choice([2, 3, 4]))
    if kind == "fp8":
        return _case("layer", "llama", rng.randint(1, 8), tau, fp8=True)
    if kind == "f32":
        return _case("layer", "tiny", _log_int(rng, 1, 1024), tau, fresh=fresh)
    if kind == "mask":
        return _case("mask", "paper", _log_int(rng, 197, 50432), p=round(math.exp(rng.uniform(math.log(0.02), math.log(0.5))), 3))
    return _case("host", rng.choice(["gpt2_ffn", "bert", "llama"]), _log_int(rng, 64, 6144), tau)


def _weights(cfg, g):
    """The layer's parameters with the distributions of workloads.make_weights, drawn on the GPU."""
    dt = api.torch_dtype(cfg.dtype)

    def normal(shape, std):
        return (torch.randn(shape, generator=g, device=DEVICE) * std).to(dt)

    return {
        "w_r1": normal((cfg.d_h, cfg.d), 1.0 / math.sqrt(cfg.d)), "b_r1": normal((cfg.d_h,), 0.1),
        "w_r2": normal((cfg.E, cfg.d_h), 1.0 / math.sqrt(cfg.d_h)), "b_r2": normal((cfg.E,), 0.1),
        "w1": normal((cfg.d_ff, cfg.d), 0.02),
        "b1": None if cfg.b1_shift is None else torch.full((cfg.d_ff,), cfg.b1_shift, device=DEVICE).to(dt),
        "w_gate": normal((cfg.d_ff, cfg.d), 0.02) if cfg.gated else None,
        "w2": normal((cfg.d, cfg.d_ff), 0.02), "b2": normal((cfg.d,), 0.02) if cfg.has_b2 else None,
    }


def _tokens(cfg, T, g):
    """T token rows as workloads.make_tokens draws them: N(0, 1) times a lognormal scale of the token."""
    x = torch.randn((T, cfg.d), generator=g, device=DEVICE)
    if cfg.token_sigma > 0:
        x = x * torch.exp(torch.randn((T, 1), generator=g, device=DEVICE) * cfg.token_sigma)
    return x.to(api.torch_dtype(cfg.dtype))


def _mask_words(T, E, p, g):
    """Bernoulli(p) decisions as the mask words of the C ABI: expert i = bit i % 32 of word i // 32."""
    W = (E + 31) // 32
    keep = torch.zeros((T, W * 32), dtype=torch.int64, device=DEVICE)
    keep[:, :E] = torch.rand((T, E), generator=g, device=DEVICE) < p
    words = (keep.view(T, W, 32) << torch.arange(32, device=DEVICE)).sum(-1)
    return torch.where(words >= 1 << 31, words - (1 << 32), words).to(torch.int32)


def prepare(case, seed):
    cfg, T = workloads.CONFIGS[case["shape"]], case["T"]
    g = torch.Generator(device=DEVICE)
    g.manual_seed(int(seed))
    layers = [api.Layer.from_config(cfg, _weights(cfg, g), device=DEVICE, fp8_experts=case["fp8"]) for _ in range(case["layers"])]
    s = {"case": case, "layer": layers[0], "x": _tokens(cfg, T, g), "y": None, "routing": None}
    if case["call"] == "group":
        s["group"] = api.LayerGroup(layers)
        s["group"].workspace(T)
        s["routing"] = [L.new_routing(T) for L in layers]
        s["y"] = torch.empty((len(layers), T, cfg.d), dtype=s["x"].dtype, device=DEVICE)
    elif case["call"] == "host":
        s["x"] = s["x"].cpu().pin_memory()
        s["y"] = torch.empty_like(s["x"]).pin_memory()
        s["ws"] = layers[0].host_workspace(T)
    else:
        layers[0].workspace(T)
        if case["call"] == "mask":
            s["mask"] = _mask_words(T, cfg.E, case["p"], g)
        elif not case["fresh"]:
            s["routing"] = layers[0].new_routing(T)
        if not case["fresh"]:
            s["y"] = torch.empty_like(s["x"])
    return s


def run(s):
    case, layer = s["case"], s["layer"]
    # Beside y, a layer call's answer is what each token kept: the mask words and k.  (The per-expert lists follow from
    # the mask, and one decision at a tie of the threshold moves every entry behind it, so they come back where the
    # decisions are given and every whole number is determined.)
    if case["call"] == "layer":
        y, r = layer.layer_fwd(s["x"], case["tau"], y=s["y"], routing=s["routing"])
        return {"y": y, "mask": r.mask, "k": r.k}
    if case["call"] == "group":
        y, rs = s["group"].group_fwd(s["x"], case["tau"], y=s["y"], routings=s["routing"])
        return {"y": y, "mask": [r.mask for r in rs], "k": [r.k for r in rs]}
    if case["call"] == "mask":
        r = api.routing_from_mask(s["mask"], layer.E)
        y = layer.moe_ffn_fwd(s["x"], r, y=s["y"])
        return {"y": y, "k": r.k, "counts": r.counts, "offsets": r.offsets, "perm": r.perm, "scalars": r.scalars}
    return {"y": layer.layer_fwd_host(s["x"], case["tau"], s["y"], s["ws"])}


def _kept(case, cfg):
    """Expected fraction of experts that a token keeps.  Scores are close to |N(0, 1)| times a constant, so with the
    largest of E at its median m it is P(|N(0, 1)| >= tau m) (0.39 for 128 experts at tau = 0.3, 0.21 for 344 at 0.4)."""
    if case["call"] == "mask":
        return case["p"]
    lo, hi, tail = 0.0, 8.0, 1.0 - 0.5 ** (1.0 / cfg.E)
    for _ in range(60):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if math.erfc(mid / math.sqrt(2.0)) > tail else (lo, mid)
    return math.erfc(case["tau"] * lo / math.sqrt(2.0))


def work(case):
    cfg, T, n = workloads.CONFIGS[case["shape"]], case["T"], case["layers"]
    elem = 4 if cfg.dtype == "f32" else 2
    rho = _kept(case, cfg)
    used = cfg.E * (1.0 - (1.0 - rho) ** T)                        # experts that at least one token keeps
    pairs = rho * T * cfg.E
    words = (cfg.E + 31) // 32
    by = T * cfg.d * elem * (1 + n)                                # x once, y of every layer
    by += n * used * cfg.n_mat * cfg.s * cfg.d * (1 if case["fp8"] else elem)
    by += n * 4 * (T * words + T + pairs + 2 * cfg.E)              # mask, k, token lists, counts and offsets
    fl = n * pairs * 2.0 * cfg.n_mat * cfg.d * cfg.s
    if case["call"] != "mask":
        by += n * elem * cfg.d_h * (cfg.d + cfg.E)                 # router
        fl += n * 2.0 * T * cfg.d_h * (cfg.d + cfg.E)
    return {"bytes": by, "flops": fl}


def tolerance(case):
    # float32: sums of up to 256 products in another order.  bf16: outputs and hidden activations are rounded to 8
    # bits; an expert whose score lies on the threshold to within float32 rounding may be kept or not, which changes
    # that token's row (`max`) and its mask word and k (`differ`).
    if workloads.CONFIGS[case["shape"]].dtype == "f32":
        return {"rel": 1e-5, "max": 1e-3, "differ": 0.002}
    return {"rel": 1e-2, "max": 0.3, "differ": 0.0 if case["call"] == "mask" else 0.002}
