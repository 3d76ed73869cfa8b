"""Every kernel waits for the stream's previous kernel before anything else
(launch_kernel allows its blocks to be set up early)."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1405_2915_gb300", "csrc")


def test_every_kernel_begins_with_grid_wait():
    seen = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        assert "<<<" not in text, f"{path}: kernels are launched through launch_kernel"
        for m in re.finditer(r"__global__", text):
            body = text[text.index("{", m.end()) + 1:]
            assert body.lstrip().startswith("dev::grid_wait();"), f"{path}: {text[m.start():m.start() + 120]}"
            seen += 1
    assert seen > 40
