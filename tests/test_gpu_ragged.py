"""Products whose activations no tensor map can describe (row pitch or base not a
multiple of 16 bytes), against the oracle: the kernels then stage them with
4-byte copies.  Each on the kernel with resident column slices, for which the
shapes were chosen, and on whichever kernel the rule takes.  Bounds: fp32 sums
(gpu_helpers.sum_tol)."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import oracle
from paper_1911_08020_gb300 import darb, synth

from .gpu_helpers import XRES_PLAIN, assert_product_close, dev, encode_both, spmm_on, sum_tol

pytestmark = pytest.mark.gpu


def _stored(g, rows, cols, dtype, mset):
    w = (0.05 * g.standard_normal((rows, cols))).astype(np.float32)
    m = g.choice(np.asarray(mset, np.int32), size=rows)
    return (synth.f32_to_bf16_bits(w) if dtype == "bf16" else w), m


def _x(cols, B, ldx, shift, seed):
    """(host X, device view of it): rows of pitch ldx from element `shift`, NaN around it."""
    X = synth.activations(cols, B, seed=seed)
    buf = torch.full((shift + cols * ldx,), float("nan"), device=dev())
    Xd = buf[shift:].view(cols, ldx)[:, :B]
    Xd.copy_(torch.from_numpy(X))
    return X, Xd


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("rows,cols,mset,B,pad,shift", [
    (70, 600, (8, 16), 2001, 0, 0),        # one slice, more tiles than clusters: a cluster changes tile
    (300, 7000, (10, 20, 40), 333, 0, 0),  # several slices, tiles changed too
    (130, 9000, (3, 64, 256), 63, 0, 0),   # slices with the rows past their end, and past the matrix
    (64, 500, (8, 32), 17, 0, 0),          # half a tile and a column
    (64, 500, (8, 32), 32, 1, 0),          # a whole tile at an odd pitch
    (64, 500, (8, 32), 36, 0, 1),          # a good pitch from a base 4 bytes past a boundary
])
def test_spmm_unaligned_activations(dtype, rows, cols, mset, B, pad, shift):
    g = np.random.default_rng(70)
    stored, m = _stored(g, rows, cols, dtype, mset)
    h, ref = encode_both(stored, m, dtype)
    try:
        X, Xd = _x(cols, B, B + pad, shift, seed=B)
        Yr, A = oracle.darb_spmm(ref, X, with_absdot=True)
        tol = sum_tol(-(-cols // m.min()))
        Y = torch.empty((rows, B), device=dev())
        spmm_on(XRES_PLAIN, h, Xd, Y)
        assert_product_close(Y.cpu().numpy(), Yr, A, tol)
        assert_product_close(darb.darb_spmm(h, Xd).cpu().numpy(), Yr, A, tol)
        darb.darb_sync_status(h)
    finally:
        darb.darb_destroy(h)
