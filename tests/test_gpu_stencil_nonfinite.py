"""2D stencils and their adjoints over one infinite or NaN value: it reaches
the outputs whose taps read it (through the boundary too) and no others; a
5-point stencil has no corner taps to carry it there."""
import numpy as np
import pytest

from helpers import dev_empty, dev_tensor, forced, skel, to_np, wrap

pytestmark = pytest.mark.gpu

W = {"stencil5": [0, .125, 0, .125, .5, .125, 0, .125, 0],
     "stencil9": [.0625, .125, .0625, .125, .25, .125, .0625, .125, .0625]}
SHAPES = [(9, 130), (6, 264), (5, 7), (1, 6), (6, 1), (1, 1), (2, 128)]


def sources(k, n, boundary):
    """The element that index k of an axis of n reads, or None."""
    if 0 <= k < n:
        return k
    return {"clamp": min(max(k, 0), n - 1), "zero": None, "periodic": k % n}[boundary]


def reached(fn, boundary, shape, at, adjoint):
    """The outputs that a non-zero tap connects to element `at`."""
    hit = np.zeros(shape, bool)
    for i in range(shape[0]):
        for j in range(shape[1]):
            for k, w in enumerate(W[fn]):
                if w == 0:
                    continue
                src = sources(i + k // 3 - 1, shape[0], boundary), sources(j + k % 3 - 1, shape[1], boundary)
                if None in src:
                    continue
                if adjoint and (i, j) == at:
                    hit[src] = True
                if not adjoint and src == at:
                    hit[i, j] = True
    return hit


@pytest.mark.parametrize("shape", SHAPES, ids=str)
@pytest.mark.parametrize("boundary", ["clamp", "zero", "periodic"])
@pytest.mark.parametrize("fn", ["stencil5", "stencil9"])
def test_one_value(fn, boundary, shape):
    import torch
    sk = skel()
    rows, cols = shape
    spots = {(r, c) for r in {0, 1, rows // 2, rows - 2, rows - 1} for c in {0, 1, cols // 2, cols - 2, cols - 1}
             if 0 <= r < rows and 0 <= c < cols}
    out = dev_empty(shape, torch.float32)
    for at in sorted(spots):
        for value in (np.float32(np.inf), np.float32(np.nan)):
            x = np.ones(shape, np.float32)
            x[at] = value
            dx = wrap(dev_tensor(x))
            for adjoint in (False, True):
                hit = reached(fn, boundary, shape, at, adjoint)
                for variant in range(4):
                    try:
                        with forced("mapoverlap2d", variant):
                            (sk.skel_mapoverlap_bwd if adjoint else sk.skel_mapoverlap)(fn, 1, None, boundary, dx, wrap(out))
                    except sk.SkelError as e:
                        assert e.code == -4     # unaligned rows
                        continue
                    got = to_np(out)
                    assert np.array_equal(~np.isfinite(got), hit), (at, value, adjoint, variant)
                    assert np.all(np.isnan(got[hit]) if np.isnan(value) else got[hit] == value)
