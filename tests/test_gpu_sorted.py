"""Expert step on tokens ordered by the experts they keep (layers of at most 32 experts): against the oracle on sampled tokens and,
bit for bit, against the masked dense pair, at batches that begin and end tiles and buckets everywhere."""
import dataclasses

import numpy as np
import pytest
import torch

import oracle
from paper_2310_04361_b200 import workloads as wl

pytestmark = pytest.mark.gpu
TOL_Y = 2e-2


@pytest.fixture(scope="module")
def api():
    from paper_2310_04361_b200 import api
    return api


def _keep(kind, T, E, rng):
    if kind == "one mask":                                     # one bucket
        return np.broadcast_to(np.arange(E) % 5 == 0, (T, E)).copy()
    if kind == "nothing":                                      # no up projection at all
        return np.zeros((T, E), bool)
    if kind == "two kinds":                                    # a bucket that ends inside a tile, the other reaches the ragged end
        k = np.zeros((T, E), bool)
        k[: T // 2 + 7, 0] = True
        k[T // 2 + 7:, E - 1] = True
        return k[rng.permutation(T)]
    p = float(kind)
    k = rng.random((T, E)) < p
    k[::97] = False                                            # tokens that keep nothing between others
    k[5] = True                                                # and one that keeps everything
    return k


# (E, s, d, T): the paper's experts; experts of 64 neurons; a word full of experts; few; ragged last tiles, one of one row
CASES = [(24, 128, 768, 23555, k) for k in ("0.02", "0.2", "one mask", "nothing", "two kinds")] + [
    (32, 64, 1024, 26369, "0.05"), (8, 128, 1024, 52481, "0.1"), (32, 128, 512, 26369, "0.1")]


@pytest.mark.parametrize("E,s,d,T,kind", CASES)
def test_sorted_form(api, E, s, d, T, kind):
    rng = np.random.default_rng(T + E)
    cfg = dataclasses.replace(wl.CONFIGS["paper"], E=E, d_ff=E * s, d=d, T=T)
    w, x = wl.make_weights(cfg), wl.make_tokens(cfg)
    layer = api.Layer.from_config(cfg, w)
    G = _keep(kind, T, E, rng).astype(np.uint8)
    r = api.routing_from_mask(torch.from_numpy(oracle.pack_mask(G).view(np.int32)).cuda(), E)
    assert 0 <= r.n_sel <= layer.sorted_limit(T)               # the form is what runs
    xd = api.to_device(x, cfg.dtype)
    ys = []
    for rep in range(2):                                       # the counters reset themselves; stale rows and cells would show
        layer.workspace(T).fill_(0xff)                         # bf16 NaNs
        y = torch.full((T, d), float("nan"), dtype=torch.bfloat16, device="cuda")
        layer.moe_ffn_fwd(xd, r, y=y)
        assert r.status == 0
        ys.append(y)
    layer.set_expert_path("dense")
    assert layer.sorted_limit(T) == -1
    yd = layer.moe_ffn_fwd(xd, r)
    # the same products in the same order, plus exact zeros
    for y in ys:
        assert torch.equal(y.view(torch.int16), yd.view(torch.int16))
    sample = np.unique(np.concatenate([[0, 5, 97, T - 2, T - 1], rng.integers(0, T, 120)]))
    ref = oracle.moe_ffn(x[sample], w["w1"], w["b1"], w["w_gate"], w["w2"], w["b2"], oracle.ACT_BY_NAME[cfg.act], G[sample])
    got = ys[0].float().cpu().numpy()[sample]
    assert np.isfinite(got).all() and np.abs(got - ref).max() / np.abs(ref).max() <= TOL_Y
    layer.close()


def test_above_the_limit_the_dense_pair_runs(api):
    cfg = wl.with_tokens(wl.CONFIGS["paper"], 24000)
    layer = api.Layer.from_config(cfg, wl.make_weights(cfg))
    g = torch.Generator(device="cuda").manual_seed(3)
    x = torch.randn((cfg.T, cfg.d), generator=g, device="cuda").to(torch.bfloat16)
    words = ((torch.rand((cfg.T, 32), generator=g, device="cuda") < 0.5).long()[:, :24] << torch.arange(24, device="cuda")).sum(-1)
    r = api.routing_from_mask(words.to(torch.int32)[:, None], cfg.E)
    assert r.n_sel > layer.sorted_limit(cfg.T) > 0
    y = layer.moe_ffn_fwd(x, r, y=torch.full_like(x, float("nan")))
    layer.set_expert_path("dense")
    assert torch.equal(y.view(torch.int16), layer.moe_ffn_fwd(x, r).view(torch.int16))
    layer.close()


# the paper's shape, and one whose rows are wide beside its hidden layer (the copy of the rows outweighs the rest)
@pytest.mark.parametrize("E,s,d", [(24, 128, 768), (8, 64, 2048)])
def test_a_workspace_serves_every_smaller_batch_of_ordered_tokens(api, E, s, d):
    """d2d_workspace_bytes(max_tokens) is enough for any batch of up to max_tokens tokens, also behind the largest that is ordered: the sizes
    never fall.  Sizes only: nothing is allocated or run."""
    cfg = dataclasses.replace(wl.CONFIGS["paper"], E=E, d_ff=E * s, d=d)
    layer = api.Layer.from_config(cfg, wl.make_weights(cfg))
    group = api.LayerGroup([layer])
    edge = 2048 * 128
    assert layer.sorted_limit(edge) >= 0 and layer.sorted_limit(edge + 1) == -1
    batches = sorted({*range(1, 330001, 1009), *range(edge - 200, edge + 200), 16384, 16385, 23300, 23301, 330000, 500000})
    for size in (layer.workspace_bytes, lambda T: int(api._lib.d2d_layer_fwd_host_workspace_bytes(layer.handle, T)),
                 lambda T: int(api._lib.d2d_group_workspace_bytes(group.handle, T))):
        at = [size(T) for T in batches]
        assert all(a <= b for a, b in zip(at, at[1:]))
    group.close()
    layer.close()


# tau: few pairs, some, and more than the limit (the dense pair then runs); a ragged last tile of one row, and the last batch without the
# choice; with and without the lists, which a stream of the layer's own builds beside the four kernels
@pytest.mark.parametrize("T,tau,ordered", [(43009, 0.9, True), (43009, 0.6, True), (50432, 0.7, True), (43009, 0.4, False), (42300, 0.7, False)])
def test_sorted_form_behind_a_router(api, T, tau, ordered):
    cfg = wl.with_tokens(wl.CONFIGS["paper"], T)
    w, x = wl.make_weights(cfg), wl.make_tokens(cfg)
    layer = api.Layer.from_config(cfg, w)
    xd = api.to_device(x, cfg.dtype)
    used, masks, ys = [], [], []
    ws = layer.workspace(T)
    tail = ws[layer.workspace_bytes(T) - 8 * T:layer.workspace_bytes(T)]       # masks and lists of work in the form's scratch
    for path, lists in (("auto", True), ("auto", True), ("auto", False), ("dense", False)):
        layer.set_expert_path(path)
        ws.fill_(0xff)                                         # bf16 NaNs; what a form does not write stays
        r = layer.new_routing(T, lists=lists)
        if lists:
            r.perm.fill_(-1), r.counts.fill_(-1), r.offsets.fill_(-1)
        y = torch.full((T, cfg.d), float("nan"), dtype=torch.bfloat16, device="cuda")
        layer.layer_fwd(xd, tau, y=y, routing=r)
        torch.cuda.synchronize()
        assert r.status == 0
        used.append(bool((tail != 0xff).any()))
        masks.append(r.mask_u32().copy())
        ys.append(y)
        G = oracle.unpack_mask(masks[0], cfg.E)
        if path == "auto":
            behind_the_choice = 2.0 * T * cfg.d * cfg.d_ff >= 2e11
            assert (int(G.sum()) <= layer.sorted_limit(T) and behind_the_choice) == ordered
        if lists:
            want = oracle.metadata(G)
            assert np.array_equal(r.k[:T].cpu().numpy(), G.sum(1)) and r.n_sel == want["n_sel"]
            assert np.array_equal(r.counts.cpu().numpy(), want["counts"]) and np.array_equal(r.offsets.cpu().numpy(), want["offsets"])
            assert np.array_equal(r.perm[: r.n_sel].cpu().numpy(), want["perm"])
    assert used == [ordered] * 3 + [False]
    assert all(np.array_equal(m, masks[0]) for m in masks)
    # bit for bit what the dense pair gives: the same products in the same order, plus exact zeros
    assert all(torch.equal(y.view(torch.int16), ys[-1].view(torch.int16)) for y in ys)
    sample = np.unique(np.concatenate([[0, 127, T - 1], np.random.default_rng(T).integers(0, T, 100)]))
    ref = oracle.moe_ffn(x[sample], w["w1"], w["b1"], w["w_gate"], w["w2"], w["b2"], oracle.ACT_BY_NAME[cfg.act], G[sample])
    got = ys[0].float().cpu().numpy()[sample]
    assert np.isfinite(got).all() and np.abs(got - ref).max() / np.abs(ref).max() <= TOL_Y
    layer.close()
