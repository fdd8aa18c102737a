"""Products on the kernel whose CTAs own rows (small and middling calls from batch
5 on), and around the limits of the rule that picks it, against the oracle.
Bounds: fp32 sums (gpu_helpers.sum_tol)."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import oracle
from paper_1911_08020_gb300 import darb, synth

from .gpu_helpers import assert_product_close, dev, encode_both, sum_tol, t

pytestmark = pytest.mark.gpu


# rows, cols, block sizes, batch, extra pitch of X and of Y, first element: one
# row; fewer rows than CTAs; rows of one chunk and of many; every tile width,
# whole and ragged; a pitch of whole 16-byte lines past a ragged batch; the
# streaming kernel with plain copies of X (a matrix too wide to stage)
CASES = [
    (1, 40, (3,), 5, 0, 0, 0), (70, 600, (1, 8, 16), 8, 0, 0, 0), (300, 300, (16, 32, 64), 7, 1, 3, 0),
    (1024, 1024, (8, 16, 32, 64), 24, 0, 0, 0), (500, 900, (2, 10, 100), 31, 0, 0, 1),
    (900, 333, (4, 30, 256), 32, 0, 4, 0), (200, 512, (8, 64), 65, 3, 0, 0), (129, 777, (7, 40), 160, 0, 0, 0),
    (3000, 100, (4, 8), 256, 0, 0, 0), (64, 20000, (16, 60), 9, 0, 0, 0), (4096, 9216, (16, 32, 64), 6, 0, 0, 0),
    (40, 30000, (200, 256), 6, 0, 0, 0),
]


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("rows,cols,mset,B,padx,pady,shift", CASES)
def test_product(rows, cols, mset, B, padx, pady, shift, dtype):
    g = np.random.default_rng(90)
    w = (0.05 * g.standard_normal((rows, cols))).astype(np.float32)
    stored = synth.f32_to_bf16_bits(w) if dtype == "bf16" else w
    m = g.choice(np.asarray(mset, np.int32), size=rows)
    h, ref = encode_both(stored, m, dtype)
    try:
        X = synth.activations(cols, B, seed=B)
        buf = torch.full((shift + cols * (B + padx),), float("nan"), device=dev())
        Xd = buf[shift:].view(cols, B + padx)[:, :B]
        Xd.copy_(torch.from_numpy(X))
        Yr, A = oracle.darb_spmm(ref, X, with_absdot=True)
        Wd = t(stored.view(np.int16)).view(torch.bfloat16) if dtype == "bf16" else t(stored)
        for _ in range(2):   # with the records read early, and right after a re-encode
            full = torch.full((rows, B + pady), -7.0, device=dev())
            darb.darb_spmm(h, Xd, full[:, :B])
            assert_product_close(full[:, :B].cpu().numpy(), Yr, A, sum_tol(-(-cols // m.min())))
            assert torch.all(full[:, B:] == -7.0)
            darb.darb_reencode(h, Wd)
        darb.darb_sync_status(h)
    finally:
        darb.darb_destroy(h)


@pytest.mark.parametrize("B", [6, 24])
def test_unselected_activations_do_not_matter(B):
    """Infinities and NaN in rows of X that no kept weight selects stay out of Y."""
    g = np.random.default_rng(91)
    rows, cols = 200, 640
    w = g.standard_normal((rows, cols)).astype(np.float32)
    m = np.full(rows, 8, np.int32)
    w[:, ::8] = 9.0   # every block keeps its first column
    h, ref = encode_both(w, m, "f32")
    try:
        X = synth.activations(cols, B, seed=3)
        Yr, A = oracle.darb_spmm(ref, X, with_absdot=True)
        X[1::8], X[2::8] = np.inf, np.nan
        Y = darb.darb_spmm(h, t(X)).cpu().numpy()
        assert_product_close(Y, Yr, A, sum_tol(cols // 8))
    finally:
        darb.darb_destroy(h)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("rows,cols,sizes,B", [
    (1024, 600, ((4, 102), (64, 922)), 8),       # the dense rows first: many rows for most CTAs, few for some
    (700, 900, ((256, 500), (2, 200)), 33),      # and last, on several column tiles
    (161, 400, ((1, 1), (256, 160)), 6),         # one row with most of the work; more rows than CTAs by a few
])
def test_product_of_rows_sorted_by_block_size(rows, cols, sizes, B, dtype):
    """The CTAs' row ranges follow the rows' cost (unit_split.h)."""
    g = np.random.default_rng(92)
    w = (0.05 * g.standard_normal((rows, cols))).astype(np.float32)
    stored = synth.f32_to_bf16_bits(w) if dtype == "bf16" else w
    h, ref = encode_both(stored, np.concatenate([np.full(n, m, np.int32) for m, n in sizes]), dtype)
    try:
        X = synth.activations(cols, B, seed=B)
        Y = darb.darb_spmm(h, t(X)).cpu().numpy()
        darb.darb_sync_status(h)
        Yr, A = oracle.darb_spmm(ref, X, with_absdot=True)
        assert_product_close(Y, Yr, A, sum_tol(-(-cols // min(m for m, _ in sizes))))
    finally:
        darb.darb_destroy(h)
