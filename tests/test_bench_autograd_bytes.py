"""The benchmark knows the bytes of every call that the composed loss makes."""
import os
import re
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_every_call_of_the_composed_loss_has_its_bytes():
    sys.path.insert(0, ROOT)
    import bench
    text = open(os.path.join(ROOT, "paper_1405_2915_gb300", "autograd.py")).read()
    names = set(re.findall(r'_call\(step, "(\w+)"', text))
    assert {"fwd_fused", "bwd_fused", "fwd_map_tanh", "bwd_map_tanh_sum"} <= names
    assert names == set(bench.AUTOGRAD_BYTES)
