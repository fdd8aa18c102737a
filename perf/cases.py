"""The work that a program using this library has it do, as measurable cases.

Five kinds of pass, each through the public calls of ``paper_1911_08020_gb300.darb``:

* ``spmm``      one product Y = W_darb X (``darb_spmm``): a fully-connected or gate layer at inference;
* ``tensor``    the same product with the tensor-core kernels asked for (``darb_spmm_ex``);
* ``retrain``   new weights into an existing handle, then a product with them (``darb_reencode`` and
                ``darb_spmm``): one turn of the prune-retrain loop;
* ``step``      one LSTM or GRU cell step, the state in and out: streaming recurrent inference;
* ``sequence``  a recurrent layer over a whole input sequence.

A case names the kind, the matrix (rows x cols, or hidden and input size), the storage type of the
weights, the law its per-row block sizes are drawn from, and the batch.  Weights are Gaussian with a
lognormal scale per row, so that rows differ in density as trained layers do; activations are N(0, 1).
``darb_assign_from_weights`` and ``darb_encode`` run once per trained layer and are part of
``prepare``, not of a pass.
"""
import math
import weakref

import numpy as np
import torch

from paper_1911_08020_gb300 import darb

# Per-row block sizes and their probabilities: the laws of this repository's own workloads.
LAWS = {
    "gemv": ((8, 16, 32, 64), (0.1, 0.2, 0.3, 0.4)),
    "lstm": ((4, 8, 16, 32), (0.1, 0.1, 0.4, 0.4)),
    "lm": ((10, 15, 20, 30), (0.25, 0.25, 0.25, 0.25)),
    "gru": ((8, 16, 32, 64), (0.2, 0.15, 0.3, 0.35)),
    "fc": ((16, 32, 64), (0.4, 0.3, 0.3)),
}


def listed():
    return [
        # The smallest call: one vector through a small fp32 layer, where launch and latency are all there is.
        {"name": "gemv_1024_f32_b1", "kind": "spmm", "rows": 1024, "cols": 1024, "dtype": "f32", "law": "gemv", "batch": 1},
        # A large fully-connected layer serving a small, a middling and a large batch.
        {"name": "fc6_b16", "kind": "spmm", "rows": 4096, "cols": 9216, "dtype": "bf16", "law": "fc", "batch": 16},
        {"name": "fc6_b64", "kind": "spmm", "rows": 4096, "cols": 9216, "dtype": "bf16", "law": "fc", "batch": 64},
        {"name": "fc6_b256", "kind": "spmm", "rows": 4096, "cols": 9216, "dtype": "bf16", "law": "fc", "batch": 256},
        # Offline scoring: a ragged layer (odd rows, columns and batch, block sizes that are no powers of two).
        {"name": "ragged_b999", "kind": "spmm", "rows": 3001, "cols": 4099, "dtype": "f32", "law": "lm", "batch": 999},
        # The caller accepts the tensor cores' rounding for a large batch.
        {"name": "fc6_tensor_b256", "kind": "tensor", "rows": 4096, "cols": 9216, "dtype": "bf16", "law": "fc", "batch": 256},
        # Prune-retrain turns: bf16 weights in power-of-two blocks, and fp32 weights in others.
        {"name": "retrain_fc6_bf16", "kind": "retrain", "rows": 4096, "cols": 9216, "dtype": "bf16", "law": "fc", "batch": 64},
        {"name": "retrain_6000x3000_f32", "kind": "retrain", "rows": 6000, "cols": 3000, "dtype": "f32", "law": "lm", "batch": 40},
        # Streaming speech: one cell step for 32 streams.
        {"name": "lstm_step_b32", "kind": "step", "cell": "lstm", "input": 256, "hidden": 1024, "dtype": "f32", "law": "lstm", "batch": 32},
        # Whole utterances: one stream, a language-model layer, and a GRU layer over a wide batch.
        {"name": "lstm_sequence_b1", "kind": "sequence", "cell": "lstm", "input": 256, "hidden": 1024, "dtype": "f32", "law": "lstm", "batch": 1, "steps": 100},
        {"name": "lm_sequence_b20", "kind": "sequence", "cell": "lstm", "input": 1500, "hidden": 1500, "dtype": "bf16", "law": "lm", "batch": 20, "steps": 35},
        {"name": "gru_sequence_b64", "kind": "sequence", "cell": "gru", "input": 1024, "hidden": 1024, "dtype": "bf16", "law": "gru", "batch": 64, "steps": 200},
    ]


def _spread(rng, lo, hi):
    """A whole number from lo to hi, spread over the logarithm."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(("spmm", "spmm", "spmm", "tensor", "retrain", "step", "sequence", "sequence"))
    case = {"kind": kind, "dtype": rng.choice(("f32", "bf16")), "law": rng.choice(sorted(LAWS))}
    if kind == "tensor":
        case["dtype"] = "bf16"   # the only weights this path takes
    if kind in ("step", "sequence"):
        case["cell"] = rng.choice(("lstm", "gru"))
        case["hidden"] = _spread(rng, 128, 1500)
        case["input"] = _spread(rng, 64, 1500)
        case["batch"] = _spread(rng, 1, 64)
        if kind == "sequence":
            # no more multiply-adds than 200 GRU steps of 64 columns at 1024 + 1024
            gates = 4 if case["cell"] == "lstm" else 3
            one = gates * case["hidden"] * (case["hidden"] + case["input"]) * case["batch"]
            case["steps"] = _spread(rng, 10, max(11, min(200, 200 * 64 * 3 * 1024 * 2048 // one)))
        return case
    case["rows"] = _spread(rng, 256, 6000)
    case["cols"] = _spread(rng, 256, 9216)
    most = max(1, min(1024, 4096 * 9216 * 256 // (case["rows"] * case["cols"])))
    if kind == "spmm":
        case["batch"] = _spread(rng, 1, most)
    elif kind == "tensor":
        case["batch"] = _spread(rng, 32, max(33, min(512, most)))
    else:
        case["batch"] = _spread(rng, 1, 64)
    return case


def _shape(case):
    """(rows, cols) of the weight matrix."""
    if case["kind"] in ("step", "sequence"):
        gates = 4 if case["cell"] == "lstm" else 3
        return gates * case["hidden"], case["input"] + case["hidden"]
    return case["rows"], case["cols"]


def _inputs(case, seed):
    """The numbers of a case: weights, block sizes, activations and states, from the seed alone."""
    rows, cols = _shape(case)
    gen = torch.Generator(device="cuda").manual_seed(seed)

    def normal(*shape):
        return torch.randn(*shape, generator=gen, device="cuda", dtype=torch.float32)

    dtype = torch.float32 if case["dtype"] == "f32" else torch.bfloat16
    sizes, probs = LAWS[case["law"]]
    d = {"m": np.random.default_rng(seed).choice(np.asarray(sizes, np.int32), size=rows, p=probs)}

    def weights():
        return (0.05 * normal(rows, cols) * torch.exp(0.5 * normal(rows, 1))).to(dtype)

    d["W"] = weights()
    b = case["batch"]
    if case["kind"] in ("spmm", "tensor", "retrain"):
        d["X"] = normal(cols, b)
        if case["kind"] == "retrain":
            d["W_new"] = weights()
        return d
    n, i = case["hidden"], case["input"]
    d["x"] = normal(case["steps"], i, b) if case["kind"] == "sequence" else normal(i, b)
    d["h"], d["c"] = 0.5 * normal(n, b), 0.5 * normal(n, b)
    d["bias"], d["bias_h"] = 0.1 * normal(rows), 0.1 * normal(rows)
    return d


class _State:
    """What a program has in hand before a call; releases its handle when it goes."""

    def __init__(self, case, d):
        self.case = case
        self.__dict__.update(d)
        self.handle = darb.darb_encode(self.W, self.m)
        weakref.finalize(self, darb.darb_destroy, self.handle).atexit = False
        kind, b = case["kind"], case["batch"]
        if kind != "retrain":
            self.W = None   # only the encoding is kept
        if kind in ("spmm", "tensor", "retrain"):
            self.Y = torch.empty(self.handle.rows, b, device="cuda")
            return
        n = case["hidden"]
        lead = (case["steps"],) if kind == "sequence" else ()
        self.h_out = torch.empty(*lead, n, b, device="cuda")
        self.c_out = torch.empty(n, b, device="cuda")
        if kind == "step":
            darb.darb_rnn_reserve(self.handle, b)


def prepare(case, seed):
    return _State(case, _inputs(case, seed))


def run(state):
    s, case = state, state.case
    kind = case["kind"]
    if kind == "spmm":
        return darb.darb_spmm(s.handle, s.X, s.Y)
    if kind == "tensor":
        return darb.darb_spmm_ex(s.handle, s.X, s.Y, darb.PATH_TENSOR_CORES)
    if kind == "retrain":
        darb.darb_reencode(s.handle, s.W_new)
        return darb.darb_spmm(s.handle, s.X, s.Y)
    i, n, b = case["input"], case["hidden"], case["batch"]
    if kind == "step":
        if case["cell"] == "lstm":
            darb.darb_lstm_step(s.handle, i, n, b, s.x, s.h, s.c, s.bias, s.h_out, s.c_out)
            return s.h_out, s.c_out
        darb.darb_gru_step(s.handle, i, n, b, s.x, s.h, s.bias, s.bias_h, s.h_out)
        return s.h_out
    if case["cell"] == "lstm":
        darb.darb_lstm_sequence(s.handle, case["steps"], i, n, b, s.x, s.h, s.c, s.bias, s.h_out, None, s.c_out)
        return s.h_out, s.c_out
    darb.darb_gru_sequence(s.handle, case["steps"], i, n, b, s.x, s.h, s.bias, s.bias_h, s.h_out)
    return s.h_out


def work(case):
    rows, cols = _shape(case)
    width = 4 if case["dtype"] == "f32" else 2
    kept = rows * sum(p * math.ceil(cols / m) for m, p in zip(*LAWS[case["law"]]))
    offsets = rows * sum(p * math.ceil(cols / m) * (0.5 if m <= 16 else 1) for m, p in zip(*LAWS[case["law"]]))
    encoded = kept * width + offsets + 6 * rows
    b = case["batch"]
    if case["kind"] in ("spmm", "tensor"):
        return {"bytes": encoded + 4 * (rows + cols) * b, "flops": 2 * kept * b}
    if case["kind"] == "retrain":
        # the dense weights in, the encoding out, and the product's own bytes (the encoding read again)
        return {"bytes": rows * cols * width + 2 * encoded + 4 * (rows + cols) * b, "flops": 2 * kept * b}
    t, n, i = case.get("steps", 1), case["hidden"], case["input"]
    states = 4 if case["cell"] == "lstm" else 2   # h (and c) in and out
    biases = rows if case["cell"] == "lstm" else 2 * rows
    return {"bytes": encoded + 4 * (t * i * b + (t - 1) * n * b + states * n * b + biases), "flops": 2 * kept * b * t}


def tolerance(case):
    if case["kind"] == "tensor":
        # X enters as two bf16 parts, 2^-17 of each product at most: 2.7e-6 measured against 64 bits
        return {"rel": 1.2e-5, "max": 4e-4}
    if case["kind"] == "sequence":
        # fp32 sums in another order, carried through the recurrence: up to 4e-7 measured
        return {"rel": 2e-6, "max": 1e-4}
    # fp32 sums in another order: up to 2.1e-7 measured
    return {"rel": 1e-6, "max": 2e-5}


def _pruned(W, m):
    """W in 64 bits with one weight kept per block: the largest magnitude, the lowest column on ties."""
    rows, cols = W.shape
    out = torch.zeros(rows, cols, dtype=torch.float64, device=W.device)
    for size in sorted(set(int(v) for v in m)):
        pick = torch.from_numpy(np.flatnonzero(m == size)).to(W.device)
        blocks = -(-cols // size)
        w = torch.nn.functional.pad(W[pick].float(), (0, blocks * size - cols)).view(len(pick), blocks, size)
        # the bits of a magnitude order as the magnitude does; the low bits prefer the lower column
        key = (w.abs().view(torch.int32).to(torch.int64) << 16) | (65535 - torch.arange(size, device=W.device))
        best = key.argmax(dim=2, keepdim=True)
        kept = torch.zeros_like(w).scatter_(2, best, w.gather(2, best))
        out[pick] = kept.view(len(pick), blocks * size)[:, :cols].double()
    return out


def exact(case, seed):
    d = _inputs(case, seed)
    W = _pruned(d["W_new"] if case["kind"] == "retrain" else d["W"], d["m"])
    if case["kind"] in ("spmm", "tensor", "retrain"):
        return W @ d["X"].double()
    i, n = case["input"], case["hidden"]
    wx, wh = W[:, :i], W[:, i:]
    xs = d["x"].double()
    h, c = d["h"].double(), d["c"].double()
    bias, bias_h = d["bias"].double()[:, None], d["bias_h"].double()[:, None]
    hs = []
    for x in xs if case["kind"] == "sequence" else [xs]:
        if case["cell"] == "lstm":
            gi, gf, gg, go = (wx @ x + wh @ h + bias).split(n)
            c = torch.sigmoid(gf) * c + torch.sigmoid(gi) * torch.tanh(gg)
            h = torch.sigmoid(go) * torch.tanh(c)
        else:
            ar, az, an = (wx @ x + bias).split(n)
            br, bz, bn = (wh @ h + bias_h).split(n)
            r, z = torch.sigmoid(ar + br), torch.sigmoid(az + bz)
            h = (1 - z) * torch.tanh(an + r * bn) + z * h
        hs.append(h)
    out = torch.stack(hs) if case["kind"] == "sequence" else h
    return (out, c) if case["cell"] == "lstm" else out
