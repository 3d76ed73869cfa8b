"""The row-streaming 2D stencil kernel (MapOverlap variant 0 and the
time-blocked chains) where it can go wrong: widths around the strips' 120 and
112 output columns, rows of every alignment, grids smaller than the halo, and
segments that end at the grid's last row."""
import numpy as np
import pytest

import oracle
import synthetic as syn
from helpers import assert_elem_close, dev_empty, dev_tensor, forced, skel, to_np, wrap

pytestmark = pytest.mark.gpu

COLS = [1, 3, 4, 111, 112, 113, 119, 120, 121, 128, 225, 241, 364]


@pytest.mark.parametrize("cols", COLS)
@pytest.mark.parametrize("rows", [1, 2, 7, 40])
@pytest.mark.parametrize("boundary", ["clamp", "zero", "periodic"])
def test_single_step(rows, cols, boundary):
    import torch
    sk = skel()
    w = syn.uniform_f32(77, 9, -1.0, 1.0).reshape(3, 3)
    x = syn.uniform_f32(60 + cols, rows * cols).reshape(rows, cols)
    for pad in (0, 1):
        dout = dev_empty((rows, cols), torch.float32, pad)
        with forced("mapoverlap2d", 0):
            sk.skel_mapoverlap("stencil9", 1, w, boundary, wrap(dev_tensor(x, pad)), wrap(dout))
            # nine products of |w|, |x| < 1: each partial sum is below 9, nine roundings of at
            # most 2^-24 relative to it
            assert_elem_close(to_np(dout), oracle.mapoverlap2d_f32(x, 1, w, boundary), f"pad {pad}", atol=81 * 2.0 ** -24)
            sk.skel_mapoverlap_bwd("stencil5", 1, None, boundary, wrap(dev_tensor(x, pad)), wrap(dout))
        ref = oracle.mapoverlap2d_bwd_f32(x, 1, oracle.stencil_weights("5pt"), boundary)
        assert_elem_close(to_np(dout), ref, f"adjoint pad {pad}")


@pytest.mark.parametrize("cols", COLS)
@pytest.mark.parametrize("rows", [1, 7, 150])
@pytest.mark.parametrize("boundary", ["clamp", "zero"])
@pytest.mark.parametrize("k", [3, 5, 8])
def test_fused_steps_equal_single_calls(rows, cols, boundary, k):
    import torch
    sk = skel()
    x = syn.uniform_f32(90 + cols, rows * cols).reshape(rows, cols)
    for kind in ("stencil5", "stencil9"):
        got = {}
        for variant in (0, 1):
            tmp, out = (dev_empty((rows, cols), torch.float32) for _ in range(2))
            with forced("chain2d", variant, 0, 0, k):
                sk.skel_mapoverlap_chain(kind, None, boundary, k + 2, wrap(dev_tensor(x)), wrap(tmp), wrap(out))
            got[variant] = to_np(out)
        assert np.array_equal(got[0].view(np.uint32), got[1].view(np.uint32)), kind
