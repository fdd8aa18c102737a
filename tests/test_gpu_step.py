"""One LSTM / GRU cell step (darb_lstm_step, darb_gru_step) against the CPU oracle
over the tile widths, stagings and row splits of the step kernel, and past the
widest input it stages.  Bounds as for every step (gpu_helpers), from those of
fp32 sums for either dtype."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import oracle
from paper_1911_08020_gb300 import darb, synth

from .gpu_helpers import (BATCH, ROWLANE, ROWS, dev, encode_both, gru_bound, last_kernel, lstm_bounds, sum_tol, t)

pytestmark = pytest.mark.gpu


def _buf(a, shift):
    """Device copy of `a` whose base is `shift` floats past a 16-byte boundary."""
    b = torch.empty(a.size + shift, device=dev())
    v = b[shift:].view(a.shape)
    v.copy_(torch.from_numpy(a))
    return v


# (I, H, B, block sizes, shift): tiles of 4 to 32 columns, whole, ragged and
# several; rows shorter than a chunk and longer than a lane group's run; blocks
# and chunks across I; no x; one unit; bases 4 bytes past a boundary; inputs too
# tall for the kernel (15000 rows)
SHAPES = [
    (5, 7, 1, (1, 2, 3), 0), (33, 40, 3, (3, 8, 16), 0), (64, 200, 4, (4, 30), 0), (64, 200, 4, (4, 30), 1),
    (0, 64, 8, (8, 64), 0), (100, 300, 7, (2, 10, 20), 0), (96, 160, 16, (4, 16, 40), 0), (50, 77, 13, (8, 256), 0),
    (256, 300, 32, (4, 8, 32), 0), (300, 256, 32, (4, 8, 32), 1), (40, 500, 64, (8, 16), 0), (600, 30, 96, (5, 50), 0),
    (31, 1, 33, (1, 7, 64), 0), (700, 900, 45, (10, 15, 30), 0), (15000, 4, 2, (16, 64), 0), (15000, 4, 6, (16, 64), 0),
]


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("cell", ["lstm", "gru"])
@pytest.mark.parametrize("I,H,B,mset,shift", SHAPES)
def test_step(cell, I, H, B, mset, shift, dtype):
    g = np.random.default_rng(80)
    gates = 4 if cell == "lstm" else 3
    w = (0.3 * g.standard_normal((gates * H, I + H))).astype(np.float32)
    stored = synth.f32_to_bf16_bits(w) if dtype == "bf16" else w
    m = g.choice(np.asarray(mset, np.int32), size=gates * H)
    h, ref = encode_both(stored, m, dtype)
    tol = sum_tol(-(-(I + H) // m.min()) + 4)   # and the biases, and the two parts of a GRU's sum
    try:
        x = synth.activations(max(I, 1), B, seed=1)[:I].copy()
        hp, cp = synth.state(H, B, seed=2), synth.state(H, B, seed=3)
        b1, b2 = synth.bias(gates * H, seed=4), synth.bias(gates * H, seed=5)
        xd = _buf(x, shift) if I else None
        ho, co = torch.empty((H, B), device=dev()), torch.empty((H, B), device=dev())
        Wd = t(stored.view(np.int16)).view(torch.bfloat16) if dtype == "bf16" else t(stored)
        for _ in range(2):   # with the records read early, and right after a re-encode
            if cell == "lstm":
                darb.darb_lstm_step(h, I, H, B, xd, _buf(hp, shift), _buf(cp, shift), t(b1), ho, co)
                hr, cr, ga = oracle.lstm_step(ref, I, H, x if I else None, hp, cp, b1)
                bc, bh = lstm_bounds(ga, cp, tol)
                assert np.all(np.abs(co.cpu().numpy() - cr) <= bc)
                assert np.all(np.abs(ho.cpu().numpy() - hr) <= bh)
            else:
                darb.darb_gru_step(h, I, H, B, xd, _buf(hp, shift), t(b1), t(b2), ho)
                hr, ga = oracle.gru_step(ref, I, H, x if I else None, hp, b1, b2)
                assert np.all(np.abs(ho.cpu().numpy() - hr) <= gru_bound(ga, hp, hr, tol))
            ho.fill_(float("nan"))
            co.fill_(float("nan"))
            darb.darb_reencode(h, Wd)
        darb.darb_sync_status(h)
    finally:
        darb.darb_destroy(h)


@pytest.mark.parametrize("cell,I,H,B", [("lstm", 60, 400, 8), ("gru", 90, 500, 3), ("gru", 0, 200, 40)])
def test_step_of_units_sorted_by_block_size(cell, I, H, B):
    """The CTAs' unit ranges follow the units' cost (unit_split.h)."""
    g = np.random.default_rng(81)
    gates = 4 if cell == "lstm" else 3
    w = (0.3 * g.standard_normal((gates * H, I + H))).astype(np.float32)
    m = np.tile(np.r_[np.full(H // 10, 2, np.int32), np.full(H - H // 10, 64, np.int32)], gates)
    h, ref = encode_both(w, m, "f32")
    try:
        x = synth.activations(max(I, 1), B, seed=1)[:I].copy()
        hp, cp = synth.state(H, B, seed=2), synth.state(H, B, seed=3)
        ho, co = torch.empty((H, B), device=dev()), torch.empty((H, B), device=dev())
        xd = t(x) if I else None
        if cell == "lstm":
            darb.darb_lstm_step(h, I, H, B, xd, t(hp), t(cp), None, ho, co)
            hr, cr, ga = oracle.lstm_step(ref, I, H, x if I else None, hp, cp, None)
            bc, bh = lstm_bounds(ga, cp, sum_tol((I + H + 1) // 2 + 4))
            assert np.all(np.abs(co.cpu().numpy() - cr) <= bc)
            assert np.all(np.abs(ho.cpu().numpy() - hr) <= bh)
        else:
            darb.darb_gru_step(h, I, H, B, xd, t(hp), None, None, ho)
            hr, ga = oracle.gru_step(ref, I, H, x if I else None, hp, None, None)
            assert np.all(np.abs(ho.cpu().numpy() - hr) <= gru_bound(ga, hp, hr, sum_tol((I + H + 1) // 2 + 4)))
        darb.darb_sync_status(h)
    finally:
        darb.darb_destroy(h)


# (cell, I, H, block sizes, batch, kernel): steps of large matrices whose times on
# the kernels differ by 20% or more
RULE = [
    ("lstm", 256, 1024, (4, 8, 16, 32), 32, ROWS), ("lstm", 7000, 1192, (10, 15, 20, 30), 1, ROWLANE),
    ("lstm", 4096, 4096, (16, 32, 64), 2, ROWS), ("lstm", 7000, 1192, (10, 15, 20, 30), 4, ROWS), ("lstm", 7000, 1192, (10, 15, 20, 30), 64, BATCH),
    ("lstm", 4096, 4096, (16, 32, 64), 32, BATCH), ("lstm", 4096, 4096, (16, 32, 64), 13, ROWS),
    ("gru", 2048, 2048, (8, 16, 32, 64), 32, ROWS), ("gru", 2048, 2048, (8, 16, 32, 64), 64, ROWS),
]


@pytest.mark.parametrize("cell,I,H,mset,B,kernel", RULE)
def test_large_steps_run_on_the_faster_kernel(cell, I, H, mset, B, kernel):
    """... and agree with one-column steps, which add in another order: two fp32
    sums of up to 820 products each within 820 * 2^-24 of sum |w x| (at most some
    20 here) of the exact one, through a cell that contracts."""
    gates = 4 if cell == "lstm" else 3
    gen = torch.Generator(device=dev()).manual_seed(4)
    w = (0.02 * torch.randn((gates * H, I + H), device=dev(), generator=gen)).to(torch.bfloat16)
    h = darb.darb_encode(w, np.random.default_rng(82).choice(np.asarray(mset, np.int32), gates * H))
    del w
    try:
        x, hp, cp = (torch.randn((n, B), device=dev(), generator=gen) for n in (I, H, H))

        def step(x, hp, cp):
            ho, co = torch.empty_like(hp), torch.zeros_like(hp)
            if cell == "lstm":
                darb.darb_lstm_step(h, I, H, hp.shape[1], x, hp, cp, None, ho, co)
            else:
                darb.darb_gru_step(h, I, H, hp.shape[1], x, hp, None, None, ho)
            return ho, co

        ho, co = step(x, hp, cp)
        assert last_kernel() == kernel
        for j in {0, B - 1}:
            for whole, one in zip((ho, co), step(*(v[:, j:j + 1].contiguous() for v in (x, hp, cp)))):
                assert torch.max(torch.abs(whole[:, j:j + 1] - one)).item() < 2e-3
        darb.darb_sync_status(h)
    finally:
        darb.darb_destroy(h)


def test_step_takes_scratch_only_for_the_kernels_that_use_it():
    """The local-cell kernel needs no gate sums or counters: a handle that only
    runs such steps holds no memory for them (and none is allocated in a capture
    of a first step); a step on the other kernels adds it."""
    g = np.random.default_rng(83)
    I, H, B = 40, 64, 8
    w = (0.3 * g.standard_normal((4 * H, I + H))).astype(np.float32)
    h, ref = encode_both(w, np.full(4 * H, 8, np.int32), "f32")
    try:
        x, hp, cp = synth.activations(I, B, seed=1), synth.state(H, B, seed=2), synth.state(H, B, seed=3)
        xd, hd, cd = t(x), t(hp), t(cp)
        ho, co = torch.empty((H, B), device=dev()), torch.empty((H, B), device=dev())
        held = darb.darb_info(h)["device_bytes"]
        graph = torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
        with torch.cuda.graph(graph):
            darb.darb_lstm_step(h, I, H, B, xd, hd, cd, None, ho, co)
        graph.replay()
        torch.cuda.synchronize()
        assert last_kernel() == ROWS
        assert darb.darb_info(h)["device_bytes"] == held
        hr, cr, ga = oracle.lstm_step(ref, I, H, x, hp, cp, None)
        bc, bh = lstm_bounds(ga, cp, sum_tol((I + H) // 8 + 4))
        assert np.all(np.abs(co.cpu().numpy() - cr) <= bc)
        assert np.all(np.abs(ho.cpu().numpy() - hr) <= bh)
        wide = [torch.randn((n, 1028), device=dev()) for n in (I, H, H)]
        out = [torch.empty((H, 1028), device=dev()) for _ in range(2)]
        darb.darb_lstm_step(h, I, H, 1028, *wide, None, *out)
        assert last_kernel() == BATCH
        assert darb.darb_info(h)["device_bytes"] > held
        darb.darb_sync_status(h)
    finally:
        darb.darb_destroy(h)


def test_gru_step_infinite_weight_in_a_block_across_the_boundary():
    """Block [4, 8) of a row holds x columns 4, 5 and h columns 6, 7 (I = 6); an
    infinite weight on one side must not meet the other side's zeros."""
    I, H, B = 6, 6, 3
    w = np.full((3 * H, I + H), 0.1, np.float32)
    w[:, 4] = np.inf        # every row keeps column 4 of that block
    m = np.full(3 * H, 4, np.int32)
    h = darb.darb_encode(t(w), m)
    try:
        x, hp = np.ones((I, B), np.float32), np.full((H, B), 0.5, np.float32)
        ho = torch.empty((H, B), device=dev())
        darb.darb_gru_step(h, I, H, B, t(x), t(hp), None, None, ho)
        # r = z = 1 (their sums are +inf), n = tanh(inf): h = (1 - 1) * 1 + 1 * h
        np.testing.assert_array_equal(ho.cpu().numpy(), hp)
    finally:
        darb.darb_destroy(h)
