"""The cut of a decode batch (d2d_decode_plan_for), on the host: what the kernel keeps per cluster fits where it keeps it."""
import itertools

import pytest

WIDTHS = (64, 128, 256, 640, 768, 896, 1024, 1536, 2048, 2304, 3072, 4096, 5120, 8192)


@pytest.fixture(scope="module")
def api():
    from paper_2310_04361_b200 import build
    build.build()
    from paper_2310_04361_b200 import api
    return api


def _desc(api, d, d_ff, s=16, gated=False, d_h=128):
    return api.LayerDesc(d=d, d_ff=d_ff, n_experts=d_ff // s, expert_size=s, d_h=d_h, dtype=api.D2D_BF16, act=api.ACTS["gelu_erf"],
                         gated=int(gated))


@pytest.mark.parametrize("n_layers", [1, 2, 3, 4])
def test_lists_of_kept_units_fit(api, n_layers):
    """Every layer and group the kernel takes, up to the largest d_ff and a step beyond: a cluster's list has room for all
    of its units, the clusters cover them, and the ring is long enough to be one."""
    taken = 0
    for d, gated, fp8, T in itertools.product(WIDTHS, (False, True), (False, True), (1, 3, 5, 8, 9, 16, 17, 32)):
        for d_ff in (16, 1024, 3072, 11008, 16384, 17408, 33792, 49152, 65536, 65552):
            p = api.decode_plan(_desc(api, d, d_ff, gated=gated), T, n_layers, fp8)
            if p is None:
                continue
            taken += 1
            what = (d, d_ff, gated, fp8, T)
            assert d_ff <= 65536 and p.list_entries <= p.list_capacity, what
            assert p.cluster_size * p.clusters * n_layers <= 148 and p.stages >= 3, what
            assert p.rounds * p.cluster_size * p.clusters * 16 >= d_ff, what
    assert taken > 1000


def _instance(p, d, fp8):
    """Which instance of the expert kernel a plan takes: codes or not, 16-column output tiles per warp, token block."""
    tiles = -(-(d // p.cluster_size) // 256)
    return fp8, next(t for t in (1, 2, 4, 8) if tiles <= t), p.token_block


def test_the_gpu_tests_run_every_instance(api):
    from test_gpu_parity import DECODE_CASES
    reachable, refused = set(), set()
    for d, fp8, T, d_ff, n in itertools.product(range(64, 8193, 64), (False, True), (1, 3, 8, 9, 16, 17, 32), (16, 2048, 11008), (1, 3)):
        p = api.decode_plan(_desc(api, d, d_ff), T, n, fp8)
        if p is not None:
            reachable.add(_instance(p, d, fp8))
    run = set()
    for shape, T, fp8 in DECODE_CASES:
        desc = _desc(api, shape["d"], shape["d_ff"], shape["d_ff"] // shape["E"], shape.get("gated", False), shape.get("d_h", 128))
        p = api.decode_plan(desc, T, 1, fp8)
        if p is not None and p.router:
            run.add(_instance(p, shape["d"], fp8))
        else:
            refused.add((shape["d"], T))
    assert run == reachable and len(run) == 18
    assert refused >= {(1024, 17), (640, 33)}


# largest batch of one layer that the decode kernels take, as the documents state it: width, gated, 8-bit weights
@pytest.mark.parametrize("d,d_ff,E,gated,d_h,fp8,most", [
    (512, 2048, 128, False, 128, False, 32), (640, 2560, 160, False, 128, False, 32), (768, 3072, 128, False, 128, False, 16),
    (768, 3072, 128, False, 128, True, 32), (1024, 4096, 256, False, 128, False, 16), (1024, 4096, 256, False, 128, True, 16),
    (2048, 8192, 256, False, 128, False, 16), (4096, 11008, 344, True, 256, False, 8), (4096, 11008, 344, True, 256, True, 8)])
def test_largest_decode_batch(api, d, d_ff, E, gated, d_h, fp8, most):
    desc = _desc(api, d, d_ff, d_ff // E, gated, d_h)
    taken = [T for T in range(1, 40) if (p := api.decode_plan(desc, T, 1, fp8)) is not None and p.router]
    assert taken == list(range(1, most + 1))
