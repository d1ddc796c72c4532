"""Waits on barriers that another CTA of the cluster signals acquire at cluster scope.

A missing scope does not show in results (the hardware orders more than the model promises), so this reads the source: every
barrier that a remote arrival or a remote asynchronous store names is only waited for in the forms that have the scope."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2310_04361_b200", "csrc")
# how a file names the barrier in a remote signal, and its waits whose scope is the cluster
FILES = {
    "gemm_tc.cu": (r"mbar_arrive_cluster\(map_to_cta\(smem_u32\(&(\w+)", {"sched_full", "sched_empty", "bar_acc_empty"}),
    "decode_ffn.cu": (r"arrive_cluster\(cluster_addr\(smem_addr\(&(\w+)", {"h_full", "h_empty"}),
    "decode_router.cu": (r"cluster_rank_addr\((?:smem_addr\(&)?(bar\w*)", {"bar", "bar_s"}),
}


@pytest.mark.parametrize("name", sorted(FILES))
def test_waits_for_remote_signals_have_cluster_scope(name):
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
    pattern, expected = FILES[name]
    signalled = set(re.findall(pattern, text))
    assert signalled == expected, "a barrier signalled across the cluster was added or renamed: look at its waits"
    if "bar" in signalled:                        # decode_router.cu: the local name of bar_u's address
        signalled = signalled - {"bar"} | {"bar_u"}
    waits = re.findall(r"\b(\w*wait\w*|mbar_test)(<[^<>]*>)?\(\s*(?:smem_u32\(|smem_addr\()?&(\w+)", text)
    for call, _, bar in waits:
        if bar in signalled:
            assert call in ("peer_wait", "peer_wait_warp", "mbar_wait_cluster"), (call, bar)
    assert {bar for _, _, bar in waits} >= signalled


def test_the_cluster_forms_acquire_at_cluster_scope():
    tc = open(os.path.join(CSRC, "tc_common.cuh")).read()
    for form in ("test_wait", "try_wait"):
        assert len(re.findall(rf"if \(CLUSTER\)\s*asm volatile\(\s*\"[^;]*;[^;]*mbarrier\.{form}\.parity\.acquire\.cluster\.", tc)) == 1
    gemm = open(os.path.join(CSRC, "gemm_tc.cu")).read()
    assert re.search(r"peer_wait = .*mbar_wait<64, 32, PAIR>", gemm) and re.search(r"peer_wait_warp = .*mbar_wait_warp<PAIR>", gemm)
    assert "mbar_wait_warp<true>" in open(os.path.join(CSRC, "decode.cuh")).read()
