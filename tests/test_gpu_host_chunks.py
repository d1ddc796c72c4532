"""How a host call cuts its batch: the result is, bit for bit, that of layer calls on the expected pieces, in as many launches."""
import pytest
import torch

from paper_2310_04361_b200 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    from paper_2310_04361_b200 import api
    return api


GATED = dict(d=1536, d_ff=6144, E=96, gated=True, act="silu", b1_shift=None)       # 18432 neurons times matrices: the layer is the slowest leg
PLAIN = dict(d=1536, d_ff=9216, E=144)
NARROW = dict(d=256, d_ff=1024, E=64)
BERT = dict(d=768, d_ff=3072, E=128)
GPT2 = dict(d=1024, d_ff=4096, E=256)
F32_WIDE = dict(dtype="f32", d=512, d_ff=9216, E=72, d_h=64)
CASES = [
    # sizes by the layer: two, three and four chunks, on both sides of each line, and ragged ends
    (GATED, 1023, (1023,)), (GATED, 1024, (512, 512)), (GATED, 1535, (768, 767)), (GATED, 1536, (512, 512, 512)), (GATED, 2047, (512, 1024, 511)),
    (GATED, 3327, (1024, 1280, 1023)), (GATED, 3328, (768, 1024, 1024, 512)), (GATED, 4099, (1024, 1024, 1024, 1027)),
    (PLAIN, 1536, (512, 512, 512)), (PLAIN, 3328, (768, 1024, 1024, 512)),
    # equal ones: by tokens, and by the bytes of the rows (3 and 7 MB)
    (BERT, 2048, (1024, 1024)), (BERT, 2047, (2047,)), (BERT, 2559, (1280, 1279)), (BERT, 2560, (896, 896, 768)),
    (GPT2, 3584, (1280, 1280, 1024)), (GPT2, 3585, (1024, 1024, 1024, 513)),
    # narrow rows: two from 2 MB and 3584 tokens on
    (NARROW, 4095, (4095,)), (NARROW, 4096, (2048, 2048)), (NARROW, 6143, (3072, 3071)), (NARROW, 6144, (2048, 2048, 2048)),
    (dict(d=320, d_ff=1024, E=64), 3583, (3583,)), (dict(d=320, d_ff=1024, E=64), 3584, (1792, 1792)),
    # float32 takes the equal ones
    (F32_WIDE, 1600, (896, 704)),
]


@pytest.mark.parametrize("shape,T,sizes", CASES)
def test_host_call_is_the_layer_call_on_its_chunks(api, shape, T, sizes):
    assert sum(sizes) == T
    cfg = wl.LayerConfig("host", **{**dict(dtype="bf16", d_h=128, act="gelu_erf", token_sigma=0.5, b1_shift=-0.3), **shape}, T=T, seed=61)
    layer = api.Layer.from_config(cfg, wl.make_weights(cfg))
    x = torch.from_numpy(wl.make_tokens(cfg)).to(api.torch_dtype(cfg.dtype)).pin_memory()
    y = torch.full_like(x, float("nan")).pin_memory()
    ws = layer.host_workspace(T)
    before = api._lib.d2d_launch_count()
    layer.layer_fwd_host(x, 0.3, y, ws)
    launches = api._lib.d2d_launch_count() - before
    xd, want, at = x.cuda(), [], 0
    before = api._lib.d2d_launch_count()
    for n in sizes:
        want.append(layer.layer_fwd(xd[at:at + n], 0.3, routing=layer.new_routing(n, lists=cfg.dtype == "f32"))[0])     # float32: this form needs them
        at += n
    assert api._lib.d2d_launch_count() - before == launches
    want = torch.cat(want).cpu()
    bits = torch.int32 if cfg.dtype == "f32" else torch.int16
    assert torch.isfinite(y).all() and torch.equal(y.view(bits), want.view(bits))
    layer.close()
