"""The scan's rules on top of the shipped execution-plan table: one block per
row, few long rows, one sequence past the SMs' shared memory; whole and odd row
lengths, each with the result of the 64-bit prefix sums."""
import os

import pytest

from helpers import SUM_REL, skel, wrap

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
# shape, the variants that forward and reverse scans take
CASES = [((70, 20_000), 5, 5), ((4, 300_000), 5, 5), ((75, 200_000), 8, 8), ((2, 4_000_000), 8, 8), ((20, 50_000), 4, 1),
         ((76, 20_000), 9, 9), ((5, 8192), 9, 9), ((70, 20_001), 0, 0), ((20, 50_001), 0, 1), ((9_000_004,), 8, 8),
         ((8_000_004,), 9, 9)]


@pytest.mark.parametrize("shape,forward,reverse", CASES, ids=str)
def test_rules(shape, forward, reverse):
    import torch
    sk = skel()
    sk.skel_load_dispatch_table(os.path.join(ROOT, "paper_1405_2915_gb300", "dispatch_gb300.tbl"))
    try:
        x = torch.rand(shape, device="cuda") - 0.25
        xi, out = torch.randint(0, 101, shape, device="cuda", dtype=torch.int32), torch.empty(shape, device="cuda")
        outi = torch.empty_like(xi)
        want, mag = x.double().cumsum(-1), x.double().abs().cumsum(-1)
        sk.skel_scan("add", True, wrap(xi), wrap(outi))
        assert sk.skel_last_variant("scan")[0] == forward
        assert torch.equal(outi, xi.cumsum(-1).to(torch.int32))
        sk.skel_scan("add", True, wrap(x), wrap(out))
        assert sk.skel_last_variant("scan")[0] == forward
        assert bool(((out.double() - want).abs() <= SUM_REL * mag).all())
        sk.skel_scan_bwd("add", True, wrap(x.flip(-1)), wrap(out))
        assert sk.skel_last_variant("scan")[0] == reverse
        assert bool(((out.double().flip(-1) - want).abs() <= SUM_REL * mag).all())
        sk.skel_check_device()
    finally:
        sk.skel_load_dispatch_table(None)
