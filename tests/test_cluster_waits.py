"""Barriers that another CTA of the cluster signals: the signals release and the waits acquire at cluster scope.

A missing scope does not show in results (the hardware orders more than the model promises), so this reads the source: every
barrier that a remote arrival or a remote asynchronous store names is only waited for in the forms that have the scope, and
every arrival at another CTA's barrier releases."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2310_04361_b200", "csrc")
# how a file names the barrier in a remote signal, and its waits whose scope is the cluster
FILES = {
    "gemm_tc.cu": (r"mbar_arrive_cluster\(map_to_cta\(smem_u32\(&(\w+)", {"sched_full", "sched_empty", "bar_acc_empty"}),
    "moe_gather.cu": (r"(?:mbar_arrive_cluster\(|NOTE_BYTES,\s*)map_to_cta\(smem_u32\(&(\w+)", {"tile_full", "tile_empty", "bar_full", "bar_acc_empty"}),
    "decode_ffn.cu": (r"cluster_addr\((?:smem_addr\(&)?(h_\w+|full\b)", {"h_full", "h_empty"}),
    "decode_router.cu": (r"cluster_rank_addr\((?:smem_addr\(&)?(bar\w*)", {"bar", "bar_s"}),
}


def source(name):
    return re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())


def body(text, head):
    """A definition from `head` to the closing brace in the first column."""
    start = text.index(head)
    return text[start:text.index("\n}", start)]


@pytest.mark.parametrize("name", sorted(FILES))
def test_waits_for_remote_signals_have_cluster_scope(name):
    text = source(name)
    if name == "moe_gather.cu":                   # the pair kernel and what it calls; the file's other kernels have no peers
        own = body(text, "bool forward_tile(")
        text = body(text, "bool mma_tile(") + own + body(text, "void run_scheduler(") + body(text, "moe_gather_up_kernel(")
    pattern, expected = FILES[name]
    signalled = set(re.findall(pattern, text))
    aliases = dict(re.findall(r"uint32_t (\w+) = smem_addr\(&(\w+)", text)) if name == "decode_ffn.cu" else {}
    signalled = {aliases.get(bar, bar) for bar in signalled}
    assert signalled == expected, "a barrier signalled across the cluster was added or renamed: look at its waits"
    if "bar" in signalled:                        # decode_router.cu: the local name of bar_u's address
        signalled = signalled - {"bar"} | {"bar_u"}
    if name == "moe_gather.cu":                   # the peer waits for its own gather threads there, and signals the leader
        text = text.replace(own, "")
    waits = re.findall(r"\b(\w*wait\w*|mbar_test)(<[^<>]*>)?\(\s*(?:smem_u32\(|smem_addr\()?&(\w+)", text)
    for call, scope, bar in waits:
        if bar in signalled:
            assert call in ("peer_wait", "peer_wait_warp", "mbar_wait_cluster") or (call, scope) == ("mbar_wait_warp", "<PAIR>"), (call, scope, bar)
    assert {bar for _, _, bar in waits} >= signalled


def test_the_cluster_forms_acquire_at_cluster_scope():
    tc = open(os.path.join(CSRC, "tc_common.cuh")).read()
    for form in ("test_wait", "try_wait"):
        assert len(re.findall(rf"if \(CLUSTER\)\s*asm volatile\(\s*\"[^;]*;[^;]*mbarrier\.{form}\.parity\.acquire\.cluster\.", tc)) == 1
    gemm = open(os.path.join(CSRC, "gemm_tc.cu")).read()
    assert re.search(r"peer_wait = .*mbar_wait<64, 32, PAIR>", gemm) and re.search(r"peer_wait_warp = .*mbar_wait_warp<PAIR>", gemm)
    assert "mbar_wait_warp<true>" in open(os.path.join(CSRC, "decode.cuh")).read()


@pytest.mark.parametrize("name", sorted(f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh"))))
def test_arrivals_at_other_ctas_release(name):
    """Arrivals at a barrier of another CTA (`shared::cluster`) release at cluster scope: the waiter goes on with what the arriving
    thread, or threads it has waited for, wrote or read.  The one exception only announces bytes of asynchronous stores, whose own
    completion orders them."""
    for op in re.findall(r"mbarrier\.arrive[\w.:]*", source(name)):
        if "shared::cluster" in op:
            assert ".release.cluster." in op or op == "mbarrier.arrive.expect_tx.relaxed.cluster.shared::cluster.b64", op


def test_a_sent_slot_is_read_before_its_owner_goes_on():
    """The warp that sends a CTA's hidden values reads them from the CTA's own slot.  Two rounds later the consumers write that slot again,
    behind a wait for the barrier that this warp arrives at: so the arrival has to come behind its last read, and behind all of its lanes'."""
    text = source("decode_ffn.cu")
    talk = text[text.index("} else if (warp > NCW) {"):]
    talk = talk[:talk.index("cluster_arrive();")]
    own = [m.start() for m in re.finditer(r"mbar_arrive\(full\)", talk)]
    reads = [m.start() for m in re.finditer(r"lds16\(", talk)]
    assert len(own) == 1 and reads and reads[-1] < own[0]
    # the loop over the slot's pieces has ended, and its lanes have met
    loop = talk.index("for (int r = ")
    depth = 0
    for end in range(talk.index("{", loop), len(talk)):
        depth += {"{": 1, "}": -1}.get(talk[end], 0)
        if depth == 0:
            break
    assert reads[-1] < end < own[0] and "__syncwarp();" in talk[end:own[0]]
    # and every consumer of a shared round waits for that barrier before its down projection
    assert re.search(r"auto down = .*?mbar_wait_cluster\(smem_addr\(&h_full\[j < 0 \? 2 : j & 1\]\)", text, re.S)
