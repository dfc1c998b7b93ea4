"""The interaction network in 64 bits with the roundings of the tensor-core paths
put in by hand (numpy and torch on the host): weights and operands in BF16 or
E4M3, the encoders' operands as two BF16 parts, states stored in BF16. `fmt` is
"exact" (no rounding), "bf16" or "fp8"."""
import numpy as np
import torch


def bf16(v):
    t = torch.from_numpy(np.ascontiguousarray(v, np.float32)).to(torch.bfloat16)
    return t.to(torch.float64).numpy()


def e4m3_rows(v):
    """Rows as E4M3 codes under a scale of max |row| / 448 each, decoded."""
    v = np.asarray(v, np.float32)
    amax = np.abs(v).max(axis=1, keepdims=True)
    amax = np.where(amax > 0, amax, np.float32(448))
    q = torch.from_numpy(v * (np.float32(448) / amax)).to(torch.float8_e4m3fn)
    return q.to(torch.float64).numpy() * (amax / np.float32(448))


def two_parts(v):
    return bf16(v) + bf16(v - bf16(v))


def _ln_relu(v):
    v = v - v.mean(axis=1, keepdims=True)
    return np.maximum(v / np.sqrt((v * v).mean(axis=1, keepdims=True) + 1e-5), 0.0)


def edge_logits(layers, hidden, iters, x, y, z, src, dst, fmt):
    """Logits of the edges (src, dst); `layers` = [(W, b)] from the node encoder on."""
    same = lambda v: v
    enc, parts = (same, same) if fmt == "exact" else (bf16, two_parts)
    op = {"exact": same, "bf16": bf16, "fp8": e4m3_rows}[fmt]  # step and classifier operands
    it = iter([(W.astype(np.float64), b.astype(np.float64)) for W, b in layers])

    def net(inp, act, wt, second_act):
        (W1, b1), (W2, b2) = next(it), next(it)
        return second_act(_ln_relu(act(inp) @ wt(W1).T + b1)) @ wt(W2).T + b2

    (W1, b1), (W2, b2) = next(it), next(it)  # (the K = 3 layer stays in FP32)
    h = np.stack([x / 45, y / 45, z / 750], axis=1).astype(np.float64)
    h = parts(_ln_relu(h @ W1.T + b1)) @ enc(W2).T + b2
    e = enc(net(np.concatenate([h[src], h[dst]], axis=1), parts, enc, enc))
    h = enc(h)
    for _ in range(iters):
        out, inc = np.zeros_like(h), np.zeros_like(h)
        np.add.at(out, src, e)
        np.add.at(inc, dst, e)
        h = enc(h + net(np.concatenate([op(h), op(out), op(inc)], axis=1), same, op, op))
        ends = np.concatenate([h[src], h[dst]], axis=1)
        # (one scale for both ends of an edge at hidden 128)
        ends = op(ends) if hidden == 128 else np.concatenate([op(h)[src], op(h)[dst]], axis=1)
        e = enc(e + net(np.concatenate([op(e), ends], axis=1), same, op, op))
    (W1, b1), (W2, b2) = next(it), next(it)
    return (_ln_relu(op(e) @ op(W1).T + b1) @ W2.T + b2)[:, 0]
