"""Batches of many events of mixed size, empty ones among them, through the
C ABI. The graph kernel and the re-score receptive-field kernel give each
event its place in the batch-wide edge array and row lists by a look-back over
the totals of all earlier events (windows of 32 events, more events than
resident blocks, blocks taking events in order by a ticket), so every event
must get exactly the graph, labels and re-score rows it would get alone."""
import numpy as np
import pytest

import oracle
import paper_2508_07423_gb300 as pkg
from paper_2508_07423_gb300 import synth
from parity import compare_event

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N_EVENTS = 1200


def mixed_batch(n_events, seed):
    """Events of 0, 1, 3, 8 or 30 tracks (5 % noise): empty events, single
    hits and events of a few hundred hits, in a seeded random order."""
    rng = np.random.default_rng(seed)
    choices = np.array([0, 1, 3, 8, 30])
    parts = [synth.gen_batch(1, seed, {"kind": "fixed", "n": int(rng.choice(choices))}, 0.05,
                             first_event=i)
             for i in range(n_events)]
    return synth.concat(parts)


@pytest.fixture(scope="module")
def batch():
    b = mixed_batch(N_EVENTS, 4242)
    sizes = np.diff(b.offsets)
    assert (sizes == 0).sum() > 100 and sizes.max() > 200
    return b


def tracker(wl, b, precision, band=0.0):
    return pkg.tracker_for_workload(wl, precision=precision, rescore_band=band,
                                    max_hits=b.n_hits, max_events=b.n_events, edges_per_hit=32)


def test_many_events_fp32_match_the_oracle(batch):
    wl = synth.workload("cfg1_plain_fp32")
    sh = synth.shape_of(wl)
    model = oracle.Model(synth.workload_weights(wl), sh.embed, sh.hidden, sh.iters)
    tr = tracker(wl, batch, "fp32")
    labels = pkg.run_batch(tr, batch)
    fs = pkg.feat_scale_of(tr.cfg)
    st = tr.stats()
    n_edges = 0
    for e in range(batch.n_events):
        ev = batch.event(e)
        a = int(batch.offsets[e])
        g = tr.get_graph(e)
        n_edges += len(g["src"])
        rep = compare_event(ev, g, labels[a:a + ev.n_hits], model, wl["radius2"], wl["k_max"],
                            sh.iters, wl["cut"], fs)
        assert rep.labels_compared and rep.labels_equal, e
    assert st["edges"] == n_edges and st["events"] == batch.n_events
    tr.close()


def test_many_events_batch_equals_alone(batch):
    """A sample of events (first, last, empty neighbours, the largest) run
    alone gives the batch's graph and labels bit for bit."""
    wl = synth.workload("cfg1_plain_fp32")
    tr = tracker(wl, batch, "fp32")
    labels = pkg.run_batch(tr, batch)
    graphs = {}
    sizes = np.diff(batch.offsets)
    sample = sorted({0, 1, 31, 32, 33, 64, batch.n_events - 1, int(np.argmax(sizes))}
                    | set(np.flatnonzero(sizes == 0)[:3].tolist()))
    for e in sample:
        graphs[e] = tr.get_graph(e)
    for e in sample:
        ev = batch.event(e)
        a = int(batch.offsets[e])
        lab = pkg.run_batch(tr, ev)
        assert np.array_equal(lab, labels[a:a + ev.n_hits]), e
        g = tr.get_graph(0)
        for k in g:
            assert np.array_equal(g[k], graphs[e][k]), (e, k)
    tr.close()


def test_many_events_rescore_rows_and_logits(batch):
    """BF16 with a re-score band: band edges take the FP32 logits bit for bit
    and the row lists hold exactly the receptive field, summed over events."""
    from test_gpu_precision import receptive_field, sigmoid

    wl = synth.workload("cfg1_plain_fp32")
    band = 0.05
    out = {}
    for name, prec, bd in (("fp32", "fp32", 0.0), ("bf16", "bf16", 0.0), ("band", "bf16", band)):
        tr = tracker(wl, batch, prec, bd)
        pkg.run_batch(tr, batch)
        out[name] = ([tr.get_graph(e) for e in range(batch.n_events)], tr.stats(),
                     tr.rescore_rows())
        tr.close()
    cat = lambda gs, k: np.concatenate([g[k] for g in gs])
    l0, l1, l32 = (cat(out[n][0], "logit") for n in ("bf16", "band", "fp32"))
    inband = np.abs(sigmoid(l0) - 0.5) < band
    assert inband.any() and not inband.all()
    assert np.array_equal(l1[inband], l32[inband])
    assert np.array_equal(l1[~inband], l0[~inband])
    st = out["band"][1]
    assert st["band"] == int(inband.sum())
    re, rv = receptive_field(out["bf16"][0], band, synth.shape_of(wl).iters, batch)
    assert out["band"][2] == {"edges": re, "hits": rv}
    assert (st["rescore_edges"], st["rescore_hits"]) == (re[0], rv[0])
    # one launch per stage: sort, embedding + node encoder (2), graph, edge
    # encoder, K x (messages, node step, edge step), receptive field, FP32
    # node and edge encoders, K x 3 FP32 steps, components
    K = synth.shape_of(wl).iters
    assert st["launches"] == 1 + 2 + 1 + 1 + 3 * K + 1 + 2 + 3 * K + 1, st["launches"]


@pytest.mark.parametrize("n_events", [1, 12, 13, 30, 31, 76, 77])
@pytest.mark.parametrize("dim", [4, 7])
def test_graph_kernel_branches_match_float64(n_events, dim):
    """The graph kernel's ways through an event at the sizes where they switch:
    clusters of 8, 4, 2 blocks or one block per event (by the number of events),
    everything in shared memory, without the edges' sources, without the in-edge
    lists, without the masks, without the staged rows (by the event's size and
    the number of edges), capped and uncapped hits. Edges against the oracle's
    brute force (pairs within the radius tolerance excepted, as everywhere), the
    in-edge index through the scores of a network with one message step."""
    wl = dict(synth.workload("cfg1_plain_fp32"))
    wl["model"] = {"embed": [3, 8, dim], "hidden": 32, "iters": 1}
    sh = synth.shape_of(wl)
    model = oracle.Model(synth.workload_weights(wl), sh.embed, sh.hidden, sh.iters)
    sizes = [(150, 8, 0.02), (4, 64, 0.1), (235, 64, 0.02), (285, 64, 0.01), (520, 64, 0.002),
             (900, 5, 0.004)]
    for tracks, k_max, r2 in sizes if n_events in (1, 77) else sizes[:1]:
        big = synth.gen_batch(1, 23 + tracks, {"kind": "fixed", "n": tracks}, 0.02)
        parts = [big] + [synth.gen_batch(1, 5000 + i, {"kind": "fixed", "n": 3}, 0.1)
                         for i in range(n_events - 1)]
        b = synth.concat(parts)
        w = dict(wl, k_max=k_max, radius2=r2)
        tr = pkg.tracker_for_workload(w, precision="fp32", max_hits=b.n_hits, max_events=n_events,
                                      edges_per_hit=64)
        labels = pkg.run_batch(tr, b)
        fs = pkg.feat_scale_of(tr.cfg)
        for e in {0, n_events // 2, n_events - 1}:
            ev, a = b.event(e), int(b.offsets[e])
            rep = compare_event(ev, tr.get_graph(e), labels[a:a + ev.n_hits], model, r2, k_max,
                                sh.iters, wl["cut"], fs)
            assert not rep.bad_pairs, (tracks, e, rep.bad_pairs[:3])
            assert rep.max_score_err <= 1e-4, (tracks, e, rep.max_score_err)
        tr.close()


@pytest.mark.parametrize("line", [12, 5, 2])
@pytest.mark.parametrize("over", [0, 1])
def test_graph_of_large_events_in_every_cluster_width(line, over):
    """Events whose masks lie in global memory, and events without staged rows or
    masks, in the first and the last place of batches on both sides of each change
    of the cluster's width (1/12, 1/5 and 1/2 of the SMs): the graphs, logits and
    labels they get alone, to the bit."""
    n = torch.cuda.get_device_properties(0).multi_processor_count // line + over
    wl = synth.workload("cfg1_plain_fp32")
    for tracks, k_max, r2 in ((520, 64, 0.002), (900, 5, 0.004)):
        w = dict(wl, k_max=k_max, radius2=r2)
        big = [synth.gen_batch(1, 61 + i + tracks, {"kind": "fixed", "n": tracks}, 0.02) for i in range(2)]
        small = [synth.gen_batch(1, 7000 + i, {"kind": "fixed", "n": 3}, 0.1) for i in range(n - 2)]
        b = synth.concat([big[0]] + small + [big[1]])
        tr = pkg.tracker_for_workload(w, precision="fp32", max_hits=b.n_hits, max_events=n,
                                      edges_per_hit=64)
        labels = pkg.run_batch(tr, b)
        got = [(tr.get_graph(e), labels[b.offsets[e]:b.offsets[e + 1]]) for e in (0, n - 1)]
        for (g, lab), ev in zip(got, big):
            want_lab = pkg.run_batch(tr, ev)
            want = tr.get_graph(0)
            assert want["src"].size > 100
            for k in want:
                assert np.array_equal(g[k], want[k]), (tracks, k)
            assert np.array_equal(lab, want_lab), tracks
        tr.close()


def _cut(ev, n):
    return synth.Batch(ev.x[:n], ev.y[:n], ev.z[:n], ev.plane[:n], ev.pid[:n], np.array([0, n]))


@pytest.mark.parametrize("largest", [140, 1280, 1281])
@pytest.mark.parametrize("dim,k_max", [(4, 64), (8, 3), (16, 64)])
def test_thousands_of_small_events(largest, dim, k_max):
    """Batches of thousands of small events take smaller blocks in the graph kernel
    unless one event is large (the line lies at 1280 hits): sampled events, empty ones
    and the largest among them, get the graphs and labels they get alone, to the bit."""
    n = 16 * torch.cuda.get_device_properties(0).multi_processor_count
    wl = dict(synth.workload("cfg1_plain_fp32"), k_max=k_max, radius2=0.05)
    wl["model"] = {"embed": [3, 8, dim], "hidden": 32, "iters": 1}
    kinds = [synth.gen_batch(1, 40 + t, {"kind": "fixed", "n": t}, 0.05) for t in range(9)]
    parts = [kinds[(i * 7) % 9] for i in range(n)]
    parts[n // 3] = _cut(synth.gen_batch(1, 77, {"kind": "fixed", "n": 130}, 0.05), largest)
    b = synth.concat(parts)
    tr = pkg.tracker_for_workload(wl, precision="fp32", max_hits=b.n_hits, max_events=n,
                                  edges_per_hit=64)
    labels = pkg.run_batch(tr, b)
    sample = [0, 1, 2, n // 3 - 1, n // 3, n // 3 + 1, n - 2, n - 1]
    got = [(tr.get_graph(e), labels[b.offsets[e]:b.offsets[e + 1]]) for e in sample]
    assert sum(g["src"].size for g, _ in got) > 20
    for e, (g, lab) in zip(sample, got):
        want_lab = pkg.run_batch(tr, parts[e])
        want = tr.get_graph(0)
        for k in want:
            assert np.array_equal(g[k], want[k]), (e, k)
        assert np.array_equal(lab, want_lab), e
    tr.close()


def test_small_events_do_not_wait_for_a_whole_sm_each():
    """The graph kernel's time for 20000 events of one track, alone and with one event
    of 300 hits more: below two thirds of the time with one event of 1300 hits more, which
    sends the batch to the blocks that take an SM each (1.2 ms, the time that every such
    batch took with those blocks alone; 0.7 ms before they were introduced)."""
    wl = synth.workload("cfg3_trained_bf16")
    small = synth.gen_batch(20000, 5, {"kind": "fixed", "n": 1}, wl["noise"])
    big = synth.gen_batch(1, 6, {"kind": "fixed", "n": 150}, wl["noise"])

    def plus(n):
        return synth.Batch(*(np.concatenate([getattr(small, k), getattr(big, k)[:n]])
                             for k in ("x", "y", "z", "plane", "pid")),
                           np.concatenate([small.offsets, [small.n_hits + n]]))

    tr = pkg.tracker_for_workload(wl, precision="fp32", max_hits=small.n_hits + 1300,
                                  max_events=20001, edges_per_hit=16)
    ms = []
    for b in (small, plus(300), plus(1300)):
        pkg.run_batch(tr, b)
        best = 1e9
        for _ in range(5):
            tr.set_profiling(True)
            pkg.run_batch(tr, b)
            best = min(best, tr.stage_times()["graph"][0])
            tr.set_profiling(False)
        ms.append(best)
    tr.close()
    assert max(ms[:2]) < ms[2] * 2 / 3, ms
