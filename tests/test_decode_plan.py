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
