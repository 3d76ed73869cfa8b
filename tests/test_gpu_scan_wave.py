"""Scan variant 9 (one wave of blocks, chunks in shared memory) where it can
go wrong: one unit, ends inside a unit, the smallest and largest chunk, every
alignment, rows that are no multiple of 4, and the bounded wait."""
import numpy as np
import pytest

import oracle
import synthetic as syn
from helpers import SUM_REL, assert_prefix_close, dev_empty, dev_tensor, forced, skel, to_np, wrap

pytestmark = pytest.mark.gpu

SIZES = [1, 3, 127, 128, 129, 2047, 2048, 2049, 4096 * 3 + 5, 152 * 2048 - 1, 152 * 2048 + 1, 1_000_003, 5_000_011]


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("inclusive", [True, False])
@pytest.mark.parametrize("pad_in,pad_out", [(0, 0), (1, 0), (0, 3), (2, 2)])
def test_1d(n, inclusive, pad_in, pad_out):
    import torch
    sk = skel()
    xi = syn.uniform_int(syn.SEED_INT + n, n, 0, 100)
    x = syn.uniform_f32(syn.SEED_X + n, n)
    val, ab = oracle.scan_f32(x, inclusive)
    outi, out = dev_empty((n,), torch.int32, pad_out), dev_empty((n,), torch.float32, pad_out)
    with forced("scan", 9):
        sk.skel_scan("add", inclusive, wrap(dev_tensor(xi, pad_in)), wrap(outi))
        assert np.array_equal(to_np(outi), oracle.scan_i32(xi, inclusive).astype(np.int32))
        sk.skel_scan("add", inclusive, wrap(dev_tensor(x, pad_in)), wrap(out))
        assert_prefix_close(to_np(out), val, ab, "forward")
        sk.skel_scan_bwd("add", inclusive, wrap(dev_tensor(x, pad_in)), wrap(out))
    # the reverse scan is the forward scan of the reversed sequence
    val, ab = oracle.scan_f32(np.ascontiguousarray(x[::-1]), inclusive)
    assert_prefix_close(to_np(out)[::-1], val, ab, "reverse")
    sk.skel_check_device()


@pytest.mark.parametrize("rows,cols", [(1, 5), (7, 1), (3, 127), (5, 129), (300, 257), (33, 1001), (4, 8192), (2, 55296)])
@pytest.mark.parametrize("inclusive", [True, False])
def test_rows(rows, cols, inclusive):
    import torch
    sk = skel()
    x = syn.uniform_f32(17 + cols, rows * cols).reshape(rows, cols)
    xi = syn.uniform_int(18 + cols, rows * cols, 0, 100).reshape(rows, cols)
    out, outi = dev_empty((rows, cols), torch.float32), dev_empty((rows, cols), torch.int32)
    with forced("scan", 9):
        sk.skel_scan("add", inclusive, wrap(dev_tensor(x)), wrap(out))
        sk.skel_scan("add", inclusive, wrap(dev_tensor(xi)), wrap(outi))
        fwd = to_np(out).copy()
        sk.skel_scan_bwd("add", inclusive, wrap(dev_tensor(x)), wrap(out))
    for r in {0, rows // 2, rows - 1}:
        val, ab = oracle.scan_f32(x[r].copy(), inclusive)
        assert_prefix_close(fwd[r], val, ab, f"row {r}")
        assert np.array_equal(to_np(outi)[r], oracle.scan_i32(xi[r].copy(), inclusive).astype(np.int32))
        val, ab = oracle.scan_f32(np.ascontiguousarray(x[r][::-1]), inclusive)
        assert_prefix_close(to_np(out)[r][::-1], val, ab, f"reverse row {r}")


def test_largest_chunk_and_refusal():
    import torch
    sk = skel()
    n = 55296 * torch.cuda.get_device_properties(0).multi_processor_count
    x = torch.randint(0, 101, (n + 4,), device="cuda", dtype=torch.int32)
    out = torch.empty_like(x)
    with forced("scan", 9):
        sk.skel_scan("add", True, wrap(x[:n]), wrap(out[:n]))
        assert torch.equal(out[:n], x[:n].cumsum(0, dtype=torch.int64).to(torch.int32))
        with pytest.raises(sk.SkelError) as e:
            sk.skel_scan("add", True, wrap(x), wrap(out))
        assert e.value.code == -4


def test_bounded_wait_reports_and_recovers():
    import torch
    sk = skel()
    n = 40 * 2048
    x = syn.uniform_int(41, n, 0, 100)
    dx, out = dev_tensor(x), dev_empty((n,), torch.int32)
    with forced("scan", 9):
        sk.skel_check_device()
        sk.skel_set_debug(2, 50_000)        # 50 ms
        sk.skel_set_debug(1, 3)             # block 3 never publishes
        try:
            sk.skel_scan("add", True, wrap(dx), wrap(out))
            with pytest.raises(sk.SkelError) as e:
                sk.skel_check_device()
            assert e.value.code == -7
        finally:
            sk.skel_set_debug(1, -1)
            sk.skel_set_debug(2, 2_000_000)
        sk.skel_scan("add", True, wrap(dx), wrap(out))
        sk.skel_check_device()
    assert np.array_equal(to_np(out), oracle.scan_i32(x, True).astype(np.int32))
