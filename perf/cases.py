"""What is timed: calls of gnntrk as its users make them, on device-resident hits.

A user of the library holds a handle (resident weights and workspace) and calls
find_tracks, or find_tracks_triplets, once per event or per batch of events.
Sizes, models, radii and precisions are those of the package's workloads
(workloads.json): from one plain FP32 event to the 1000-event BF16 batch, the
hidden-64 and hidden-128 models, INT8 embedding, FP8, FP32 re-scoring near the
cut and the triplet stage. Events are the synthetic vertex-detector events of
the package, ragged in size. Handles keep the default launch configuration.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2508_07423_gb300 as pkg
from paper_2508_07423_gb300 import synth

# hits a track leaves on average (26 planes, acceptance, 2 % of them missed)
HITS_PER_TRACK = 10.72
# per workload: out-edges per hit at its own track count, and the mean track
# counts over which its radius is used in earnest (the detector's occupancy)
RANGES = {
    "cfg1_plain_fp32": (6.0, (10, 100)),
    "cfg2_run3_single": (8.0, (50, 400)),
    "cfg3_batched_bf16": (6.0, (20, 400)),
    "cfg3_trained_bf16": (1.9, (20, 400)),
    "cfg4_batched_fp8": (6.0, (50, 400)),
    "cfg4_trained_fp8": (2.08, (50, 400)),
    "cfg6_triplets": (2.08, (20, 400)),
}
GRAPH_TYPES = {"src": np.int32, "dst": np.int32, "d2": np.float32, "logit": np.float32,
               "kept": np.uint8}


def _case(name, workload, n_events, tracks, precision, band=0.0, int8=False, graph=False,
          scored=False):
    c = {"workload": workload, "n_events": n_events, "tracks": tracks, "precision": precision,
         "band": band, "int8": int8, "graph": graph, "scored": scored}
    return {"name": name, **c} if name else c


def listed():
    return [
        # one small event per call, plain FP32: the latency of the smallest call
        _case("event_fp32", "cfg1_plain_fp32", 1, 40, "fp32"),
        # one event and its scored graph read back (monitoring, physics studies)
        _case("scored_fp32", "cfg2_run3_single", 1, 200, "fp32", scored=True),
        _case("scored_bf16", "cfg2_run3_single", 1, 200, "bf16", 0.02, scored=True),
        # what a trigger's server admits at once: a few dozen events, trained model
        _case("burst_trained", "cfg3_trained_bf16", 75, 150, "bf16", 0.02),
        # a larger burst with the calibrated INT8 embedding
        _case("burst_int8", "cfg3_trained_bf16", 300, 150, "bf16", 0.02, int8=True),
        # the batched form: 1000 events, BF16 with near-cut FP32 re-scoring, one
        # captured graph per call shape
        _case("batch_bf16", "cfg3_batched_bf16", 1000, 150, "bf16", 0.02, graph=True),
        # the same events with a trained model (sparser graph, few edges near the cut)
        _case("batch_trained", "cfg3_trained_bf16", 1000, 150, "bf16", 0.02),
        # offline reprocessing in FP32
        _case("batch_fp32", "cfg3_batched_bf16", 400, 150, "fp32"),
        # the run-3 model (hidden 64, 8 steps) over 100 large events
        _case("wide_fp32", "cfg2_run3_single", 100, 200, "fp32"),
        # the hidden-128 model: FP8 alone, and trained with the band that the
        # FP8 form needs
        _case("batch_fp8", "cfg4_batched_fp8", 400, 200, "fp8"),
        _case("trained_fp8", "cfg4_trained_fp8", 400, 200, "fp8", 0.05),
        # events with close track pairs through the triplet stage
        _case("triplets", "cfg6_triplets", 500, 150, "bf16", 0.02),
    ]


# what a drawn case may be: (workload, precision, band, int8, most events)
KINDS = [
    ("cfg1_plain_fp32", "fp32", 0.0, False, 100),
    ("cfg2_run3_single", "fp32", 0.0, False, 100),
    ("cfg2_run3_single", "bf16", 0.02, False, 100),
    ("cfg3_batched_bf16", "bf16", 0.02, False, 1000),
    ("cfg3_batched_bf16", "fp32", 0.0, False, 400),
    ("cfg3_trained_bf16", "bf16", 0.02, False, 1000),
    ("cfg3_trained_bf16", "bf16", 0.02, True, 1000),
    ("cfg4_batched_fp8", "fp8", 0.0, False, 400),
    ("cfg4_trained_fp8", "fp8", 0.05, False, 400),
    ("cfg6_triplets", "bf16", 0.02, False, 500),
]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    w, prec, band, int8, most = KINDS[rng.randrange(len(KINDS))]
    tracks = _log_int(rng, *RANGES[w][1])
    # a call of that kind never holds more edges than the largest one listed
    nominal = synth.workload(w)["tracks"]
    nominal = nominal["n"] if nominal["kind"] == "fixed" else nominal["mean"]
    most = max(1, min(most, int(most * (nominal / tracks) ** 2)))
    n = _log_int(rng, 1, most)
    return _case(None, w, n, tracks, prec, band, int8, graph=rng.random() < 0.25,
                 scored=n == 1 and w != "cfg6_triplets" and rng.random() < 0.5)


def _spec(case, wl):
    if wl["tracks"]["kind"] == "fixed":
        return {"kind": "fixed", "n": case["tracks"]}
    return {**wl["tracks"], "mean": case["tracks"]}


def _events(case, seed):
    wl = synth.workload(case["workload"])
    return wl, synth.gen_batch(case["n_events"], seed, _spec(case, wl), wl["noise"], 0,
                               wl.get("pair_frac", 0.0))


def _sizes(case):
    wl = synth.workload(case["workload"])
    deg, _ = RANGES[case["workload"]]
    t0 = wl["tracks"]["n"] if wl["tracks"]["kind"] == "fixed" else wl["tracks"]["mean"]
    hits = case["n_events"] * case["tracks"] * HITS_PER_TRACK * (1 + wl["noise"]) * (
        1 + wl.get("pair_frac", 0.0))
    return wl, hits, hits * deg * case["tracks"] / t0


def _capacity(case):
    """(hits, edges) that a program sizes its handle and its buffers for: the
    expected numbers, a margin for occupancy and for the spread of the events."""
    _, hits, edges = _sizes(case)
    h = int(1.15 * hits + 100 * math.sqrt(case["tracks"] * case["n_events"]))
    return h, int(edges * (h / hits) ** 2)


def prepare(case, seed):
    """Hits on the device, a handle and output buffers of the case's capacity."""
    wl, ev = _events(case, seed)
    max_hits, max_edges = _capacity(case)
    tr = pkg.tracker_for_workload(
        wl, precision=case["precision"], rescore_band=case["band"], max_hits=max_hits,
        max_events=ev.n_events, embed_int8=case["int8"], use_graph=case["graph"])
    dev = "cuda"
    s = {
        "tracker": tr, "n_events": ev.n_events, "n_hits": ev.n_hits, "graph": None,
        "xyz": torch.from_numpy(ev.xyz_soa()).to(dev),
        "plane": torch.from_numpy(ev.plane).to(dev),
        "offsets": torch.from_numpy(ev.offsets).to(dev),
        "labels": torch.full((max_hits,), -1, dtype=torch.int32, device=dev),
        "stream": torch.cuda.Stream() if case["graph"] else None,
        "tracks": None,
    }
    if case["int8"]:  # max calibration on other events of the same kind
        cal = synth.gen_batch(100, seed + 1_000_003, _spec(case, wl), wl["noise"])
        tr.set_embed_scales(tr.embed_amax(torch.from_numpy(cal.xyz_soa()).to(dev)))
    if wl.get("triplets"):
        s["tracks"] = (torch.zeros(ev.n_events + 1, dtype=torch.int32, device=dev),
                       torch.zeros(2 * max_hits + 2, dtype=torch.int64, device=dev),
                       torch.zeros(8 * max_hits + 16, dtype=torch.int32, device=dev))
    if case["scored"]:  # host buffers of the program that reads the graphs
        s["graph"] = {k: np.zeros(max_edges, t) for k, t in GRAPH_TYPES.items()}
    if s["stream"] is not None:
        s["stream"].wait_stream(torch.cuda.current_stream())
    return s


def run(s):
    tr = s["tracker"]
    args = (s["n_events"], s["n_hits"], s["xyz"], s["plane"], s["offsets"], s["labels"])
    if s["tracks"] is not None:
        tr.find_tracks_triplets(*args, *s["tracks"], s["stream"])
        ev, off, hits = s["tracks"]
        return {"labels": s["labels"], "event_tracks": ev, "track_off": off, "track_hits": hits}
    tr.find_tracks(*args, s["stream"])
    if s["graph"] is not None:
        for k, v in tr.get_graph(0).items():
            s["graph"][k][:v.size] = v
        return {"labels": s["labels"], **s["graph"]}
    return {"labels": s["labels"]}


def work(case):
    """Hits in, labels out; one pass of the networks over the hits and edges
    (an edge layer's h_src and h_dst products once per hit, not per edge)."""
    wl, N, E = _sizes(case)
    emb, h, K = wl["model"]["embed"], wl["model"]["hidden"], wl["model"]["iters"]
    per_hit = sum(2 * a * b for a, b in zip(emb, emb[1:])) + 2 * (3 * h + h * h)
    per_hit += 4 * h * h * (K + 1) + K * 2 * (3 * h * h + h * h)
    per_edge = 2 * h * h + K * 4 * h * h + 2 * (h * h + h)
    out = 4.0
    if wl.get("triplets"):
        # 1.9 triplets per kept edge (about three quarters of the edges)
        per_edge += 1.4 * 2 * (2 * h * h + h)
        out += 8.0
    graph_out = 17.0 * E if case["scored"] else 0.0
    weights = float(len(synth.workload_weights(wl)))
    return {"bytes": N * (13.0 + out) + graph_out + weights, "flops": N * per_hit + E * per_edge}


def exact(case, seed):
    """The scored graph in 64 bits (the labels are whole numbers)."""
    if not case["scored"]:
        return None
    wl, ev = _events(case, seed)
    emb, h, K = wl["model"]["embed"], wl["model"]["hidden"], wl["model"]["iters"]
    layers = iter([(W.astype(np.float64), b.astype(np.float64))
                   for W, b in synth.weight_arrays(synth.workload_weights(wl))])

    def linear(x, wb):
        return x @ wb[0].T + wb[1]

    def net(pair, x):
        v = linear(x, pair[0])
        v = v - v.mean(axis=1, keepdims=True)
        v = v / np.sqrt((v * v).mean(axis=1, keepdims=True) + 1e-5)
        return linear(np.maximum(v, 0.0), pair[1])

    x, y, z = (a.astype(np.float64) for a in (ev.x, ev.y, ev.z))
    pi = float(np.float32(math.pi))
    e = np.stack([np.hypot(x, y) / 45, np.arctan2(y, x) / pi, z / 750], axis=1)
    n_emb = len(emb) - 1
    for i in range(n_emb):
        e = linear(e, next(layers))
        if i + 1 < n_emb:
            e = np.maximum(e, 0.0)
    # hits by (plane, input index); edges to the next two planes, by source and target
    order = np.argsort(ev.plane, kind="stable")
    plane, r2 = ev.plane.astype(np.int64), float(np.float32(wl["radius2"]))
    src, dst, dd = [], [], []
    for i in order:
        cand = order[(plane[order] == plane[i] + 1) | (plane[order] == plane[i] + 2)]
        d2 = ((e[cand] - e[i]) ** 2).sum(axis=1)
        ok = np.nonzero(d2 < r2)[0]
        if ok.size > wl["k_max"]:
            ok = np.sort(ok[np.argsort(d2[ok], kind="stable")[:wl["k_max"]]])
        src += [i] * ok.size
        dst += cand[ok].tolist()
        dd += d2[ok].tolist()
    src, dst = np.asarray(src, np.int64), np.asarray(dst, np.int64)

    pairs = [(a, next(layers)) for a in layers]
    node_enc, edge_enc, steps, cls = pairs[0], pairs[1], pairs[2:2 + 2 * K], pairs[2 + 2 * K]
    hs = net(node_enc, np.stack([x / 45, y / 45, z / 750], axis=1))
    es = net(edge_enc, np.concatenate([hs[src], hs[dst]], axis=1))
    for k in range(K):
        out, inc = np.zeros_like(hs), np.zeros_like(hs)
        np.add.at(out, src, es)
        np.add.at(inc, dst, es)
        hs = hs + net(steps[2 * k], np.concatenate([hs, out, inc], axis=1))
        es = es + net(steps[2 * k + 1], np.concatenate([es, hs[src], hs[dst]], axis=1))
    logit = net(cls, es)[:, 0]
    pad = (0, _capacity(case)[1] - logit.size)
    return {"labels": None, "src": None, "dst": None, "d2": np.pad(np.asarray(dd), pad),
            "logit": np.pad(logit, pad), "kept": None}
