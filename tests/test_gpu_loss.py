"""The composed loss as one pass each way (skel_composed_loss and its
backward) against the float64 oracle and the separate calls: one warp, one
thread and several warps of columns, rows of every alignment, grids of fewer
rows than a block's halo, both boundaries, general weights, and the shapes
that keep the separate calls."""
import numpy as np
import pytest

import oracle
import synthetic as syn
from helpers import SUM_REL, dev_tensor, skel, to_np, wrap
from test_gpu_backward import grad_tolerance, loss_value_bound

pytestmark = pytest.mark.gpu

W_GENERAL = syn.uniform_f32(77, 9, -1.0, 1.0)


def separate(sk, x, w, boundary, g):
    """The definition as single calls; returns (loss, gradient)."""
    import torch
    rows, cols = x.shape
    e = lambda: torch.empty_like(x)
    t, u, s, gu, gt, gs, gt2, gx = (e() for _ in range(8))
    r = torch.empty(2, device="cuda")
    sk.skel_map("tanh", [wrap(x)], wrap(t))
    sk.skel_mapoverlap("stencil9", 1, w, boundary, wrap(t), wrap(u))
    sk.skel_scan("add", True, wrap(t), wrap(s))
    l1 = float(sk.skel_mapreduce("sq", "add", [wrap(u)]))
    c = float(sk.skel_mapreduce("sq", "add", [wrap(s)]))
    sk.skel_mapreduce_bwd("sq", "add", [wrap(u)], None, [wrap(gu)], gr_host=g)
    sk.skel_mapoverlap_bwd("stencil9", 1, w, boundary, wrap(gu), wrap(gt))
    sk.skel_mapreduce_bwd("sq", "add", [wrap(s)], None, [wrap(gs)], gr_host=float(np.float32(g) * np.float32(1.0 / x.numel())))
    sk.skel_scan_bwd("add", True, wrap(gs), wrap(gt2))
    sk.skel_map_bwd_sum("tanh", [wrap(t)], [wrap(gt), wrap(gt2)], [wrap(gx)], [1.0])
    return l1 + c / x.numel(), to_np(gx)


@pytest.mark.parametrize("shape", [(1, 1), (1, 7), (2, 16), (3, 17), (5, 512), (7, 513), (4, 515), (11, 1000), (6, 1029),
                                   (37, 2050), (9, 8192), (3, 8191), (700, 33), (1300, 5)])
def test_fused_matches_oracle(shape):
    import torch
    from paper_1405_2915_gb300.autograd import composed_loss
    x = syn.uniform_f32(syn.SEED_GRAD + shape[1], shape[0] * shape[1]).reshape(shape)
    for pad in (0, 1):
        xt = dev_tensor(x, pad).requires_grad_(True)
        L = composed_loss(xt)
        assert L.grad_fn.fused
        (gx,) = torch.autograd.grad(L, xt)
        Lr, gr = oracle.composed_loss_f32(x, 1, oracle.stencil_weights("9pt"), "clamp")
        assert abs(float(L.item()) - Lr) <= loss_value_bound(x, Lr)
        assert np.all(np.abs(to_np(gx) - gr) <= grad_tolerance(x, gr))
    with torch.no_grad():
        assert float(composed_loss(xt)) == float(L.detach())      # no gradient wanted: the same value


@pytest.mark.parametrize("shape", [(1, 3), (2, 40), (19, 517), (64, 1024), (1000, 72)])
@pytest.mark.parametrize("boundary", ["clamp", "zero"])
def test_fused_matches_separate_calls(shape, boundary):
    import torch
    from paper_1405_2915_gb300.autograd import ComposedLossFn
    sk = skel()
    x = dev_tensor(syn.uniform_f32(5 + shape[1], shape[0] * shape[1], -2.0, 2.0).reshape(shape)).requires_grad_(True)
    L = ComposedLossFn.apply(x, W_GENERAL, boundary)
    (gx,) = torch.autograd.grad(L, x, torch.full_like(L, 1.75))
    Ls, gs = separate(sk, x.detach(), W_GENERAL, boundary, 1.75)
    # both within the reductions' bound of the same value: 2 * 2^-20 relative
    assert abs(float(L.detach()) - Ls) <= 2 * SUM_REL * abs(Ls)
    t = np.abs(np.tanh(x.detach().cpu().numpy().astype(np.float64)))
    A = float(np.abs(W_GENERAL).sum())
    # stencil branch: two stencils of nine roundings each on values below A, times 2 g, and the
    # final sum and product; scan branch: twice the reverse scan's bound (grad_tolerance)
    bound = 2 * 1.75 * A * A * 22 * 2.0 ** -24
    P = np.cumsum(t, axis=1)
    suffix = np.cumsum((2 * 1.75 * P / t.size)[:, ::-1], axis=1)[:, ::-1]
    assert np.all(np.abs(to_np(gx) - gs) <= bound + 4 * SUM_REL * suffix)


@pytest.mark.parametrize("shape", [(1, 16), (2, 32), (3, 496), (4, 512), (5, 528), (9, 1040), (300, 1024), (7, 8176),
                                   (1300, 48), (5, 8192)])
@pytest.mark.parametrize("boundary", ["clamp", "zero"])
def test_rows_by_tma_match_rows_by_copies(shape, boundary):
    """Aligned rows of a multiple of 16 columns travel as TMA boxes; the same
    grid one element off the alignment as 4-byte copies.  The arithmetic of a
    column is the same, so t and the gradient agree bit for bit; the loss sums
    its terms in another grouping (float64 above the threads' sums)."""
    import torch
    from paper_1405_2915_gb300.autograd import ComposedLossFn
    x = syn.uniform_f32(9 + shape[1], shape[0] * shape[1], -2.0, 2.0).reshape(shape)
    res = []
    for pad in (0, 1):
        xt = dev_tensor(x, pad).requires_grad_(True)
        for k in range(3):                       # ring and barriers start afresh on each call
            L = ComposedLossFn.apply(xt, W_GENERAL, boundary)
            (gx,) = torch.autograd.grad(L, xt, torch.full_like(L, 1.75))
        res.append((float(L.detach()), to_np(gx)))
    assert np.array_equal(res[0][1], res[1][1])
    assert abs(res[0][0] - res[1][0]) <= SUM_REL * abs(res[1][0])


def test_nan_and_infinite_inputs_stay_where_the_definition_puts_them():
    import torch
    from paper_1405_2915_gb300.autograd import composed_loss
    sk = skel()
    x = syn.uniform_f32(3, 12 * 1100).reshape(12, 1100)
    x[5, 700] = np.nan
    x[9, 3], x[9, 4] = np.inf, -np.inf
    xt = dev_tensor(x).requires_grad_(True)
    L = composed_loss(xt)
    (gx,) = torch.autograd.grad(L, xt)
    Ls, gs = separate(sk, xt.detach(), None, "clamp", 1.0)
    assert np.isnan(float(L.detach())) and np.isnan(Ls)
    assert np.array_equal(np.isnan(to_np(gx)), np.isnan(gs))


def test_shapes_that_keep_the_separate_calls():
    import torch
    from paper_1405_2915_gb300.autograd import ComposedLossFn, composed_loss
    x = syn.uniform_f32(9, 2 * 8200).reshape(2, 8200)
    xt = dev_tensor(x).requires_grad_(True)
    L = composed_loss(xt)
    assert not L.grad_fn.fused
    Lr, gr = oracle.composed_loss_f32(x, 1, oracle.stencil_weights("9pt"), "clamp")
    assert abs(float(L.item()) - Lr) <= loss_value_bound(x, Lr)
    (gx,) = torch.autograd.grad(L, xt)
    assert np.all(np.abs(to_np(gx) - gr) <= grad_tolerance(x, gr))
    assert not ComposedLossFn.apply(xt[:, :64].contiguous(), None, "periodic").grad_fn.fused
