"""Calls back to back on one stream, from two streams, between torch's own
kernels and inside a captured graph: a kernel that is set up before the
previous one has drained still reads what that one wrote."""
import numpy as np
import pytest

from helpers import skel, wrap

pytestmark = pytest.mark.gpu

N = 1 << 16


def chain(sk, cs, calls):
    """x += 1 through `calls` dependent calls that alternate over the buffers."""
    for k in range(calls):
        sk.skel_map("add", [cs[k % 2], cs[2]], cs[(k + 1) % 2])


@pytest.mark.parametrize("n", [1, 1000, N, 5_000_011])
def test_dependent_calls_in_order(n):
    import torch
    sk = skel()
    a, b, one = torch.zeros(n, device="cuda"), torch.zeros(n, device="cuda"), torch.ones(n, device="cuda")
    cs = [wrap(a), wrap(b), wrap(one)]
    for _ in range(5):
        a.zero_()                       # torch's kernel before ours
        chain(sk, cs, 200)
        got = (a * 2).cpu().numpy()     # and after them
        assert np.array_equal(got, np.full(n, 400, np.float32))


def test_captured_calls_replay_in_order():
    import torch
    sk = skel()
    a, b, one = torch.zeros(N, device="cuda"), torch.zeros(N, device="cuda"), torch.ones(N, device="cuda")
    r = torch.zeros(1, device="cuda")
    cs, cr = [wrap(a), wrap(b), wrap(one)], wrap(r)
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        chain(sk, cs, 2)
        sk.skel_reduce("add", cs[0], cr, host=False)   # the stream's scratch exists before the capture
        s.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            chain(sk, cs, 20)
            sk.skel_reduce("add", cs[0], cr, host=False)
            sk.skel_map("scale", [cs[0]], cs[1], [0.5])
            chain(sk, cs, 2)
    a.zero_()
    torch.cuda.synchronize()
    for k in range(1, 6):
        # a = 20 more, then a / 2 written to b, then a + 1 + 1 through b
        before = a.clone()
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(a, before + 22)
        assert float(r) == float((before + 20).double().sum())


def test_two_streams_share_a_container():
    import torch
    sk = skel()
    a, b, one = torch.zeros(N, device="cuda"), torch.zeros(N, device="cuda"), torch.ones(N, device="cuda")
    cs = [wrap(a), wrap(b), wrap(one)]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    for k in range(200):                # each call depends on the one before, on the other stream
        sk.skel_map("add", [cs[k % 2], cs[2]], cs[(k + 1) % 2], stream=streams[k % 2])
    torch.cuda.synchronize()
    assert np.array_equal(a.cpu().numpy(), np.full(N, 200, np.float32))


def test_capture_on_a_stream_without_scratch_and_growth_afterwards():
    """The first call on a stream happens inside a capture: the graph's
    scratch is neither its own node nor freed when a later call on the stream
    needs more."""
    import torch
    sk = skel()
    s = torch.cuda.Stream()
    x = torch.rand(600, 700, device="cuda") * 2 - 1
    r = torch.zeros(2, device="cuda")
    cx, cflat, ca, cb = wrap(x), wrap(x.reshape(-1)), wrap(r[0:1]), wrap(r[1:2])
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    sk.skel_force_variant("compose", 2)
    try:
        with torch.cuda.graph(g, stream=s):
            sk.skel_compose_map_stencil_sumsq("tanh", "stencil9", cx, result_dev=ca, host=False)
            sk.skel_reduce("max", cflat, cb, host=False)
        want = sk.skel_compose_map_stencil_sumsq("tanh", "stencil9", cx)
        for k in range(3):
            r.zero_()
            torch.cuda.synchronize()
            g.replay()
            torch.cuda.synchronize()
            assert float(r[0]) == float(want) and float(r[1]) == float(x.max())
            big = torch.rand(1 << (16 + 3 * k), device="cuda")   # more scratch on the same stream
            out = torch.empty_like(big)
            with torch.cuda.stream(s):
                sk.skel_scan("add", True, wrap(big), wrap(out))
                sk.skel_reduce("add", wrap(big), cb, host=False)
            s.synchronize()
    finally:
        sk.skel_force_variant("compose", -1)
