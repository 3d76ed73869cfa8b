"""Batched placement by instance and the rule for few instances: empty
instances, instances that end on tile boundaries or span many tiles, one
instance, and offsets that are rejected and then repaired (also through a
captured plan)."""
import numpy as np
import pytest

import synthetic as syn
from helpers import dev_tensor, forced, skel, to_np, wrap
from test_gpu_maparray_batched import check_batched

pytestmark = pytest.mark.gpu

CASES = [[1], [4096], [4097, 0, 4095, 0, 0], [0, 0, 5], [100_000], [4096] * 7, [1] * 700, [20_000, 3] * 300]


def layout(lens):
    off = np.zeros(len(lens) + 1, np.int64)
    off[1:] = np.cumsum(lens)
    return off, syn.uniform_f32(11 + len(lens), int(off[-1]))


@pytest.mark.parametrize("lens", CASES, ids=str)
@pytest.mark.parametrize("variant", [-1, 7])
def test_placement(lens, variant):
    import torch
    sk = skel()
    off, v = layout(lens)
    for inclusive in (True, False):
        res, sc = torch.full((len(lens),), 7.0, device="cuda"), torch.full((len(v),), 7.0, device="cuda")
        with forced("batched", variant):
            sk.skel_batched(wrap(dev_tensor(v)), wrap(dev_tensor(off)), wrap(res), wrap(sc), inclusive)
        sk.skel_check_device()
        check_batched(v, off, to_np(res), to_np(sc), inclusive)


def test_rejected_offsets_leave_the_next_call_clean():
    import torch
    sk = skel()
    lens = [3000, 5000, 1, 9000]
    off, v = layout(lens)
    bad = off.copy()
    bad[2] = -5
    dv, doff = dev_tensor(v), dev_tensor(bad)
    res, sc = torch.zeros(4, device="cuda"), torch.zeros(len(v), device="cuda")
    cv, co, cr, cs = wrap(dv), wrap(doff), wrap(res), wrap(sc)
    with forced("batched", 7):
        plan = sk.Plan(cv, co, cr, cs, True)
        for run in (lambda: sk.skel_batched(cv, co, cr, cs, True), plan.launch):
            doff.copy_(torch.from_numpy(bad))
            res.fill_(7.0)
            run()
            torch.cuda.synchronize()
            assert np.all(to_np(res) == 7.0)          # nothing computed
            doff.copy_(torch.from_numpy(off))
            run()
            check_batched(v, off, to_np(res), to_np(sc), True)
        empty = wrap(torch.zeros(3, device="cuda", dtype=torch.int64))
        r0 = torch.full((2,), 7.0, device="cuda")
        sk.skel_batched(wrap(torch.zeros(0, device="cuda")), empty, wrap(r0), None, True)
        assert np.all(to_np(r0) == 0.0)
    with pytest.raises(sk.SkelError):
        sk.skel_check_device()                        # the direct call's rejection is on record
    sk.skel_check_device()
