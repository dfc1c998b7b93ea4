"""Orderings inside the kernels that no result shows: a write that must follow a
wait, a barrier that must come before an access. Breaking one gives a race whose
window is a few instructions wide, so the sources are read instead (comments
taken out, the text of one function at a time)."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2508_07423_gb300", "csrc")


def body(path, name):
    """Text of the function `name` of csrc/<path>, from its parameters to its
    closing brace, without comments and with single spaces."""
    with open(os.path.join(CSRC, path)) as f:
        text = f.read()
    text = re.sub(r"//[^\n]*|/\*.*?\*/", "", text, flags=re.S)
    m = re.search(r"(__global__|__device__)[^;{}]*\b%s\(" % name, text)
    assert m, name
    i = text.index("{", m.end())
    depth, j = 1, i + 1
    while depth:
        depth += {"{": 1, "}": -1}.get(text[j], 0)
        j += 1
    return " ".join(text[m.end():j].split())


def test_fp8_loader_stores_scales_after_the_slot_wait():
    """FP8 edge step at hidden 128: a tile's scales take the place of those of two
    tiles before. Only the wait for the tile's first ring slot says that every
    thread has read them (the slot's last MMA is issued behind a barrier that
    follows those reads), so no store of a scale may come before it."""
    b = body("k_tc.cu", "p3_loader")
    wait = b.index("mbar_wait_bounded(&empty[slot]")
    stores = [m.start() for m in re.finditer(r"scales\[[^;]*\]\.[xy] = ", b)]
    assert len(stores) == 2
    assert all(s > wait for s in stores)


def test_graph_clusters_meet_before_the_first_remote_write():
    """Graph kernel, several blocks per event: the first block writes the others'
    shared memory, which exists only once they run. A cluster barrier that every
    block reaches comes before the ticket loop."""
    b = body("k_graph.cu", "k_graph_event")
    sync = b.index("if constexpr (CLUSTER) cluster.sync();")
    assert sync < b.index("return;") and sync < b.index("map_shared_rank") and sync < b.index("for (;;)")


def test_graph_clusters_read_every_ticket_before_the_next_is_written():
    """Graph kernel, several blocks per event: between a block's read of its ticket
    and the first block's next write of it lies a cluster barrier that does not
    depend on the event (whether it has masks, say): within the ticket loop only
    `if constexpr (CLUSTER)` encloses it."""
    b = body("k_graph.cu", "k_graph_event")
    loop = b[b.index("for (;;)"):]
    read, leave = loop.index("const int ev = ticket_s;"), loop.index("if (rank > 0) continue;")
    assert loop.count("atomicAdd(&w.counters[C_GRAPH_TICKET]") == 1
    opened, depths = [], []  # texts before the open braces, those of each barrier
    for m in re.finditer(r"cluster\.sync\(\)|[{}]", loop[:leave]):
        if m.group() == "{":
            opened.append(re.split(r"[{};] ", loop[:m.start()])[-1].strip())
        elif m.group() == "}":
            opened.pop()
        elif m.start() > read:
            before = re.split(r"[{};] ", loop[:m.start()])[-1].strip()
            depths.append([o for o in opened[1:] + [before] if o])
    assert ["if constexpr (CLUSTER)"] in depths, depths


@pytest.mark.parametrize("kernel", ["k_tc", "k_tc_edge_tma", "k_tc_edge_ws"])
def test_tensor_memory_before_the_next_kernel_may_start(kernel):
    """The next kernel's blocks take tensor memory and keep it while they wait for
    this kernel. So a block lets them in only after its own allocation; else its
    allocation could wait for columns that are held by blocks waiting for it."""
    b = body("k_tc.cu", kernel)
    trigger = min(b.index(t) for t in ("pdl_begin();", "pdl_trigger();") if t in b)
    alloc = b.index("tmem_alloc(")
    assert alloc < b.index("__syncthreads();", alloc) < trigger


def test_weight_ring_after_a_wait_that_ran_out():
    """FP32 kernels at hidden 128: a warp whose wait for a chunk ran out neither
    counts as done with a chunk nor refills a stage (its copy may be in flight), and
    before it ends waits for each chunk that may be, by that chunk's own parity."""
    b = body("k_mlp_f32.cu", "product")
    refill = b[b.index("__syncwarp();"):]
    assert "late < 0" in refill[:refill.index("atomicAdd")]
    d = body("k_mlp_f32.cu", "drain")
    assert "c < late + W::NST && c < total" in d
    assert "mbar_wait_bounded(full + c % W::NST, (c / W::NST) & 1" in d
    assert "ring.drain()" in body("k_mlp_f32.cu", "finish")


@pytest.mark.parametrize("kernel", ["k_gnn_f32", "k_embed_tiles"])
def test_weight_copies_land_before_a_block_can_end(kernel):
    """FP32 kernels: the bulk copies of the weights are waited for before the first
    return, else a copy could land after the block is gone."""
    b = body("k_mlp_f32.cu", kernel)
    assert b.index("pdl_begin();") < b.index("weights.landed()") < b.index("return;")
    w = body("k_mlp_f32.cu", "landed")
    assert w.count("mbar_wait_bounded(bar, 0, kRingWaitCycles)") == 2  # once more on a timeout
