"""The host emulation of the tensor-core formats, without its roundings, is the FP64
oracle's network."""
import numpy as np
import pytest

import oracle
from paper_2508_07423_gb300 import synth
from quant_net import edge_logits


@pytest.mark.parametrize("name", ["cfg3_batched_bf16", "cfg2_run3_single", "cfg4_batched_fp8"])
def test_emulation_without_roundings_is_the_oracle(name):
    wl = synth.workload(name)
    sh = synth.shape_of(wl)
    blob = synth.workload_weights(wl)
    ev = synth.gen_batch(1, 300, {"kind": "fixed", "n": 30}, wl["noise"])
    fs = tuple(float(np.float32(v)) for v in oracle.DEFAULT_FEAT_SCALE)
    ref = oracle.find_tracks_event(oracle.Model(blob, sh.embed, sh.hidden, sh.iters), ev.x, ev.y, ev.z,
                                   ev.plane, wl["radius2"], wl["k_max"], wl["cut"], feat_scale=fs)
    layers = synth.weight_arrays(blob)[len(sh.embed) - 1:]
    got = edge_logits(layers, sh.hidden, sh.iters, ev.x, ev.y, ev.z, ref.src, ref.dst, "exact")
    assert ref.src.size > 300
    assert np.abs(got - ref.logit).max() < 1e-5
