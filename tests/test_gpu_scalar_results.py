"""Results read on the host: from several threads and streams at once, past
the number of pinned slots, and across skel_release_cached."""
import threading

import numpy as np
import pytest

from helpers import skel, wrap

pytestmark = pytest.mark.gpu


def test_threads_and_streams_read_their_own_results():
    import torch
    sk = skel()
    errors = []

    def work(k):
        s = torch.cuda.Stream()
        x = torch.full((10_000 + k,), 1.0, device="cuda")
        xi = torch.full((10_000 + k,), k - 40, device="cuda", dtype=torch.int32)
        torch.cuda.synchronize()
        cx, cxi = wrap(x), wrap(xi)
        for _ in range(20):
            got = (sk.skel_reduce("add", cx, stream=s), sk.skel_mapreduce("sq", "add", [cx], stream=s),
                   sk.skel_reduce("max", cxi, stream=s))
            if got != (10_000 + k, 10_000 + k, k - 40):
                errors.append((k, got))

    threads = [threading.Thread(target=work, args=(k,)) for k in range(80)]   # more than the 64 slots
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors


def test_types_and_release():
    import torch
    sk = skel()
    x = wrap(torch.tensor([1.5, -2.0, float("nan")], device="cuda"))
    assert isinstance(sk.skel_reduce("add", x), np.float32) and np.isnan(sk.skel_reduce("add", x))
    sk.lib.skel_release_cached()
    xi = wrap(torch.tensor([2 ** 31 - 1, 1], device="cuda", dtype=torch.int32))
    r = sk.skel_reduce("add", xi)
    assert isinstance(r, np.int32) and r == -2 ** 31
    d = torch.zeros(1, device="cuda", dtype=torch.int32)
    assert sk.skel_reduce("add", xi, wrap(d)) == -2 ** 31 and int(d) == -2 ** 31
    g = wrap(torch.ones(4, 4, device="cuda"))
    assert sk.skel_compose_map_stencil_sumsq("copy", "stencil9", g) == np.float32(16)
