"""The fused chain for rows of any alignment and width (compose variant 2)
where it can go wrong: widths around the strips' 120 columns, a grid that
ends inside a lane's four columns, one row, every boundary and map."""
import numpy as np
import pytest

import oracle
import synthetic as syn
from helpers import dev_tensor, forced, skel, wrap
from test_gpu_compose import check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cols", [1, 2, 3, 5, 119, 120, 121, 122, 123, 128, 241, 363])
@pytest.mark.parametrize("rows", [1, 2, 9, 70])
@pytest.mark.parametrize("boundary", ["clamp", "zero", "periodic"])
def test_any_width(rows, cols, boundary):
    sk = skel()
    x = syn.uniform_f32(70 + cols, rows * cols).reshape(rows, cols)
    w = syn.uniform_f32(71, 9, -1.0, 1.0).reshape(3, 3)
    for fn, kind, wt in (("tanh", "stencil9", None), ("copy", "stencil5", None), ("sq", "stencil9", w)):
        ref, bound = oracle.chain_map_stencil_sumsq_f32(
            fn, x, 1, oracle.stencil_weights("5pt" if kind == "stencil5" else "9pt") if wt is None else wt, boundary)
        for pad in (0, 1):
            with forced("compose", 2, 0, 0, rows % 3):
                got = sk.skel_compose_map_stencil_sumsq(fn, kind, wrap(dev_tensor(x, pad)), weights=wt, boundary=boundary)
            check(got, ref, bound, f"{fn} {kind} pad {pad}")
