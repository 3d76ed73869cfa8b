"""Calls captured into a CUDA graph and replayed on changing data: look-back
variants, on a stream that has scratch already and on one that has none, next
to eager calls and to another graph captured on the same stream, and the
status of a wait that ran out in a replay."""
import numpy as np
import pytest

import synthetic as syn
from helpers import forced, skel, wrap

pytestmark = pytest.mark.gpu

N = 20 * 40960 + 5          # at least 20 tiles of every variant
LENS = [3, 100_000, 0, 70_001, 4096, 1, 200_000, 4095]


def zeros_and_ones(n, dtype):
    """Whole numbers, so that every order of the sums is exact in float32."""
    import torch
    return torch.randint(0, 2, (n,), device="cuda", dtype=torch.int32).to(dtype)


def captured(stream, call):
    import torch
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream):
        call()
    return g


def replay(g):
    import torch
    torch.cuda.synchronize()
    g.replay()
    torch.cuda.synchronize()


@pytest.mark.parametrize("used", [False, True])
@pytest.mark.parametrize("dtype", ["float32", "int32"])
@pytest.mark.parametrize("variant", [0, 1, 2, 3, 4, 5, 6, 7, 8, 9])
def test_scan(variant, dtype, used):
    import torch
    sk = skel()
    dt = getattr(torch, dtype)
    x, out = zeros_and_ones(N, dt), torch.empty(N, device="cuda", dtype=dt)
    s = torch.cuda.Stream()
    with forced("scan", variant):
        if used:
            torch.cuda.synchronize()
            sk.skel_scan("add", True, wrap(x), wrap(out), stream=s)
        cx, co = wrap(x), wrap(out)
        g = captured(s, lambda: sk.skel_scan("add", True, cx, co))
        for k in range(4):
            x.copy_(zeros_and_ones(N, dt))
            replay(g)
            assert torch.equal(out.to(torch.int64), x.to(torch.int64).cumsum(0)), f"replay {k}"


@pytest.mark.parametrize("used", [False, True])
@pytest.mark.parametrize("variant", [0, 1, 2, 3, 4, 5, 6, 7])
def test_batched(variant, used):
    import torch
    sk = skel()
    off = torch.from_numpy(syn.csr_offsets(np.array(LENS, np.int64))).cuda()
    n, s = int(off[-1]), torch.cuda.Stream()
    v, res, sc = torch.empty(n, device="cuda"), torch.empty(len(LENS), device="cuda"), torch.empty(n, device="cuda")
    with forced("batched", variant, 0, 4, 0):
        v.copy_(zeros_and_ones(n, torch.float32))
        if used:
            torch.cuda.synchronize()
            sk.skel_batched(wrap(v), wrap(off), wrap(res), wrap(sc), True, stream=s)
        c = [wrap(t) for t in (v, off, res, sc)]
        g = captured(s, lambda: sk.skel_batched(*c, True))
        for k in range(4):
            v.copy_(zeros_and_ones(n, torch.float32))
            replay(g)
            for b, part in enumerate(torch.split(v, LENS)):
                lo, hi = int(off[b]), int(off[b + 1])
                assert float(res[b]) == float(part.sum()), f"replay {k}, instance {b}"
                assert torch.equal(sc[lo:hi], part.cumsum(0)), f"replay {k}, instance {b}"


def test_graphs_and_eager_calls_of_one_stream_share_nothing():
    """Two graphs captured on one stream run on two others while eager calls
    run on it: scans, a two-pass sum and a composed chain, whose counters,
    partial sums and words all sit in scratch."""
    import torch
    sk = skel()
    s, streams = torch.cuda.Stream(), [torch.cuda.Stream(), torch.cuda.Stream()]
    xs = [zeros_and_ones(N, torch.float32) for _ in range(3)]
    grids = [zeros_and_ones(1 << 20, torch.float32).reshape(1024, 1024) for _ in range(3)]
    outs, sums = [torch.empty_like(x) for x in xs], [torch.zeros(2, device="cuda") for _ in xs]
    torch.cuda.synchronize()

    def call(k, cs, stream=None):
        cx, cg, co, ca, cb = cs
        sk.skel_scan("add", True, cx, co, stream=stream)
        sk.skel_reduce("add", cx, ca, host=False, stream=stream)
        sk.skel_compose_map_stencil_sumsq("copy", "stencil9", cg, result_dev=cb, host=False, stream=stream)

    def containers(k):
        return [wrap(t) for t in (xs[k], grids[k], outs[k], sums[k][0:1], sums[k][1:2])]

    cs = [containers(k) for k in range(3)]
    with forced("scan", 9), forced("compose", 1):
        call(2, cs[2], s)
        graphs = [captured(s, lambda k=k: call(k, cs[k])) for k in range(2)]
        want = [float(sk.skel_compose_map_stencil_sumsq("copy", "stencil9", wrap(g))) for g in grids]
        torch.cuda.synchronize()
        for _ in range(30):
            for k in range(2):
                with torch.cuda.stream(streams[k]):
                    graphs[k].replay()
            call(2, cs[2], s)
        torch.cuda.synchronize()
        for k in range(3):
            assert torch.equal(outs[k], xs[k].cumsum(0))
            assert float(sums[k][0]) == float(xs[k].sum()) and float(sums[k][1]) == want[k]
        del graphs                       # their scratch goes with them; the stream's own stays in use
        sk.lib.skel_release_cached()
        call(2, cs[2], s)
        torch.cuda.synchronize()
        assert torch.equal(outs[2], xs[2].cumsum(0)) and float(sums[2][1]) == want[2]


def test_a_wait_that_ran_out_in_a_replay_is_reported():
    import torch
    sk = skel()
    s = torch.cuda.Stream()
    x, out = zeros_and_ones(N, torch.int32), torch.empty(N, device="cuda", dtype=torch.int32)
    cx, co = wrap(x), wrap(out)
    sk.skel_check_device(s)
    with forced("scan", 9):
        sk.skel_set_debug(2, 50_000)     # 50 ms
        sk.skel_set_debug(1, 3)          # block 3 never publishes
        try:
            g = captured(s, lambda: sk.skel_scan("add", True, cx, co))
        finally:
            sk.skel_set_debug(1, -1)
            sk.skel_set_debug(2, 2_000_000)
        replay(g)
        with pytest.raises(sk.SkelError) as e:
            sk.skel_check_device(s)
        assert e.value.code == -7
        sk.skel_check_device(s)
        sk.skel_scan("add", True, cx, co, stream=s)
        sk.skel_check_device(s)
        assert torch.equal(out.to(torch.int64), x.to(torch.int64).cumsum(0))
