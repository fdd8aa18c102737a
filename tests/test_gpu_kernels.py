"""Every kernel that products from batch 5 on and cell steps choose from, on the
shapes where it can go wrong, whichever the rule would take there: against the
oracle, for both dtypes, within the bound of fp32 sums (gpu_helpers.sum_tol)."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import oracle
from paper_1911_08020_gb300 import darb, synth

from .gpu_helpers import (BATCH, ROWLANE, ROWS, XRES, XRES_PLAIN, assert_product_close, dev, encode_both, gru_bound,
                          last_kernel, last_split, lstm_bounds, spmm_on, step_on, sum_tol, t)

pytestmark = pytest.mark.gpu

DTYPES = pytest.mark.parametrize("dtype", ["f32", "bf16"])


def _matrix(g, rows, cols, mset, dtype, scale=0.05):
    w = (scale * g.standard_normal((rows, cols))).astype(np.float32)
    stored = synth.f32_to_bf16_bits(w) if dtype == "bf16" else w
    m = g.choice(np.asarray(mset, np.int32), size=rows)
    h, ref = encode_both(stored, m, dtype)
    return h, ref, int(-(-cols // m.min()))


def _x(cols, B, pad, shift):
    """(host X, device view of it): rows of pitch B + pad from element `shift`, NaN around it."""
    X = synth.activations(cols, B, seed=B)
    buf = torch.full((shift + cols * (B + pad),), float("nan"), device=dev())
    Xd = buf[shift:].view(cols, B + pad)[:, :B]
    Xd.copy_(torch.from_numpy(X))
    return X, Xd


# rows, cols, block sizes: one weight; every offset width in ragged groups; wide
# matrices whose columns are split over a cluster, in slices that no block
# crosses, that fit the matrix exactly, and that need the rows past their end
MATRICES = [
    (1, 1, (1,)), (37, 91, (1, 2, 3, 8, 10, 16, 17, 32, 64, 200)), (257, 1030, (1, 2, 3, 8, 10, 16, 17, 32, 64, 200)),
    (300, 7000, (16, 32, 64)), (300, 7000, (10, 20, 40)), (260, 9000, (16, 64, 256)), (200, 6000, (3, 7, 16, 200)),
    (130, 12000, (8, 32)),
]
# (batch, extra pitch, first element): tiles whole and ragged, several of them;
# pitches and bases that are no multiples of 16 bytes
LAYOUTS = {
    ROWS: [(5, 0, 0), (8, 0, 0), (12, 4, 0), (16, 1, 0), (31, 0, 1), (32, 0, 0), (65, 3, 0), (160, 0, 0)],
    BATCH: [(5, 0, 0), (6, 2, 0), (8, 0, 0), (12, 4, 0), (13, 0, 1), (16, 0, 0), (16, 1, 0), (17, 0, 0), (33, 3, 0),
            (64, 0, 0), (64, 0, 1), (100, 0, 0)],
    XRES: [(17, 3, 0), (20, 0, 0), (32, 0, 0), (40, 0, 0), (64, 4, 0), (132, 0, 0)],
    XRES_PLAIN: [(5, 0, 0), (9, 0, 0), (13, 0, 0), (16, 1, 0), (17, 0, 0), (32, 1, 0), (36, 0, 1), (63, 0, 0),
                 (333, 0, 0)],
}


@DTYPES
@pytest.mark.parametrize("kernel", list(LAYOUTS))
@pytest.mark.parametrize("rows,cols,mset", MATRICES)
def test_product(rows, cols, mset, kernel, dtype):
    h, ref, n = _matrix(np.random.default_rng(70), rows, cols, mset, dtype)
    try:
        for B, pad, shift in LAYOUTS[kernel]:
            if kernel == ROWS and cols > 3000 and B > 16:
                continue   # tiles of 4 columns only, dozens of them: nothing new
            X, Xd = _x(cols, B, pad, shift)
            Y = torch.full((rows, B + 5), 7.0, device=dev())
            spmm_on(kernel, h, Xd, Y[:, :B])
            Yr, A = oracle.darb_spmm(ref, X, with_absdot=True)
            assert_product_close(Y[:, :B].cpu().numpy(), Yr, A, sum_tol(n))
            assert torch.all(Y[:, B:] == 7.0), "wrote outside Y's columns"
        darb.darb_sync_status(h)
    finally:
        darb.darb_destroy(h)


@DTYPES
def test_plain_copies_over_many_tiles(dtype):
    """More column tiles than clusters: a cluster changes tile and copies a new slice."""
    h, ref, n = _matrix(np.random.default_rng(71), 70, 600, (8, 16), dtype)
    try:
        X, Xd = _x(600, 2001, 0, 0)
        Y = torch.empty((70, 2001), device=dev())
        spmm_on(XRES_PLAIN, h, Xd, Y)
        Yr, A = oracle.darb_spmm(ref, X, with_absdot=True)
        assert_product_close(Y.cpu().numpy(), Yr, A, sum_tol(n))
        darb.darb_sync_status(h)
    finally:
        darb.darb_destroy(h)


# the rule's choice where the kernels are far apart: rows, cols, block sizes,
# dtype, batch, extra pitch, kernel
RULE = [
    (1024, 1024, (8, 16, 32, 64), "f32", 24, 0, ROWS), (4096, 9216, (16, 32, 64), "bf16", 13, 0, XRES_PLAIN),
    (4096, 9216, (16, 32, 64), "bf16", 16, 0, BATCH), (4096, 9216, (16, 32, 64), "bf16", 64, 0, XRES),
    (3001, 4099, (10, 15, 20, 30), "f32", 333, 0, XRES_PLAIN), (40, 30000, (200, 256), "f32", 40, 0, BATCH),
]


@pytest.mark.parametrize("rows,cols,mset,dtype,B,pad,kernel", RULE)
def test_rule(rows, cols, mset, dtype, B, pad, kernel):
    h, ref, n = _matrix(np.random.default_rng(72), rows, cols, mset, dtype)
    try:
        X, Xd = _x(cols, B, pad, 0)
        Y = darb.darb_spmm(h, Xd).cpu().numpy()
        assert last_kernel() == kernel
        Yr, A = oracle.darb_spmm(ref, X, with_absdot=True)
        assert_product_close(Y, Yr, A, sum_tol(n))
        darb.darb_sync_status(h)
    finally:
        darb.darb_destroy(h)


# rows, cols, (block size, rows) in order, batch, and the columns' splits with and
# without a finer one where clusters would have fewer than two units: a unit
# each in the finer split (faster), two that meet in one (22% slower)
@pytest.mark.parametrize("rows,cols,runs,B,finer", [
    (1000, 7000, ((10, 250), (15, 250), (20, 250), (30, 250)), 24, True),
    (739, 2652, ((16, 300), (32, 212), (64, 227)), 256, False),
])
def test_finer_split_only_where_its_longest_run_is_shorter(rows, cols, runs, B, finer):
    g = np.random.default_rng(74)
    w = (0.05 * g.standard_normal((rows, cols))).astype(np.float32)
    m = np.concatenate([np.full(n, size, np.int32) for size, n in runs])
    h, ref = encode_both(synth.f32_to_bf16_bits(w), m, "bf16")
    try:
        X, Xd = _x(cols, B, 0, 0)
        Y = torch.empty((rows, B), device=dev())
        spmm_on(XRES, h, Xd, Y)
        fewest = -(-cols * 128 // (227 * 1024 - 16384))   # slices that leave room for the partial sums
        assert last_split() > fewest + 1 if finer else last_split() <= fewest + 1
        Yr, A = oracle.darb_spmm(ref, X, with_absdot=True)
        assert_product_close(Y.cpu().numpy(), Yr, A, sum_tol(-(-cols // m.min())))
        darb.darb_sync_status(h)
    finally:
        darb.darb_destroy(h)


# ---------------------------------------------------------------------------- steps
def _state(a, shift):
    """Device copy of `a` whose base is `shift` floats past a 16-byte boundary."""
    b = torch.empty(a.size + shift, device=dev())
    v = b[shift:].view(a.shape)
    v.copy_(torch.from_numpy(a))
    return v


class _Cell:
    def __init__(self, cell, I, H, mset, dtype):
        gates = 4 if cell == "lstm" else 3
        self.cell, self.I, self.H, self.gates = cell, I, H, gates
        self.h, self.ref, n = _matrix(np.random.default_rng(73), gates * H, I + H, mset, dtype, 0.3)
        self.tol = sum_tol(n + 4)   # and the biases, and the two parts of a GRU's sum

    def check(self, B, shift, run):
        """run(x, h, c, b1, b2, h_out, c_out) against the oracle."""
        I, H = self.I, self.H
        x = synth.activations(max(I, 1), B, seed=1)[:I].copy()
        hp, cp = synth.state(H, B, seed=2), synth.state(H, B, seed=3)
        b1, b2 = synth.bias(self.gates * H, seed=4), synth.bias(self.gates * H, seed=5)
        ho, co = (torch.full((H, B), float("nan"), device=dev()) for _ in range(2))
        run(_state(x, shift) if I else None, _state(hp, shift), _state(cp, shift), t(b1), t(b2), ho, co)
        if self.cell == "lstm":
            hr, cr, ga = oracle.lstm_step(self.ref, I, H, x if I else None, hp, cp, b1)
            bc, bh = lstm_bounds(ga, cp, self.tol)
            assert np.all(np.abs(co.cpu().numpy() - cr) <= bc)
            assert np.all(np.abs(ho.cpu().numpy() - hr) <= bh)
        else:
            hr, ga = oracle.gru_step(self.ref, I, H, x if I else None, hp, b1, b2)
            assert np.all(np.abs(ho.cpu().numpy() - hr) <= gru_bound(ga, hp, hr, self.tol))

    def step(self, B, shift):
        def run(x, hp, cp, b1, b2, ho, co):
            if self.cell == "lstm":
                darb.darb_lstm_step(self.h, self.I, self.H, B, x, hp, cp, b1, ho, co)
            else:
                darb.darb_gru_step(self.h, self.I, self.H, B, x, hp, b1, b2, ho)
        self.check(B, shift, run)


CELLS = [(0, 64, (8, 64)), (33, 40, (3, 8, 16)), (64, 200, (4, 30)), (700, 300, (10, 20, 256)), (5, 7, (1, 2))]
STEPS = {ROWLANE: [(1, 0), (2, 0), (3, 0), (4, 0), (4, 1)],
         BATCH: [(5, 0), (8, 0), (8, 1), (16, 0), (20, 0), (32, 0), (33, 0), (64, 0), (64, 1), (100, 0), (132, 0)],
         ROWS: [(1, 0), (2, 0), (4, 0), (4, 1), (8, 0), (13, 0), (16, 0), (32, 0), (32, 1), (64, 0), (100, 0)]}


@DTYPES
@pytest.mark.parametrize("kernel", list(STEPS))
@pytest.mark.parametrize("cell", ["lstm", "gru"])
@pytest.mark.parametrize("I,H,mset", CELLS)
def test_step(cell, I, H, mset, kernel, dtype):
    c = _Cell(cell, I, H, mset, dtype)
    try:
        for B, shift in STEPS[kernel]:
            c.check(B, shift, lambda *a: step_on(kernel, cell, c.h, I, H, B, *a))
        darb.darb_sync_status(c.h)
    finally:
        darb.darb_destroy(c.h)


@DTYPES
@pytest.mark.parametrize("cell", ["lstm", "gru"])
def test_steps_too_tall_to_stage(cell, dtype):
    """15000 stacked rows: always the kernels that exchange their gate sums."""
    c = _Cell(cell, 15000, 4, (16, 64), dtype)
    try:
        for B, shift in ((1, 0), (2, 0), (4, 0), (4, 1), (6, 0), (8, 0), (20, 0), (33, 0), (64, 0), (64, 1)):
            c.step(B, shift)
            assert last_kernel() == (ROWLANE if B <= 4 else BATCH)
        darb.darb_sync_status(c.h)
    finally:
        darb.darb_destroy(c.h)


@pytest.mark.parametrize("cell", ["lstm", "gru"])
def test_steps_of_more_than_1024_columns(cell):
    c = _Cell(cell, 20, 30, (4, 16), "f32")
    try:
        for B, kernel in ((1024, ROWS), (1028, BATCH), (1030, BATCH)):
            c.step(B, 0)
            assert last_kernel() == kernel
        darb.darb_sync_status(c.h)
    finally:
        darb.darb_destroy(c.h)
