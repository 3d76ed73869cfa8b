"""Batched variant 7 with instances of several hundred tiles (their placement is
split over warps): starts and ends on, before and after the boundary of a run
of 128 tiles of 4096 elements, alone, among short ones and among empty ones."""
import numpy as np
import pytest

from helpers import forced, skel, wrap

pytestmark = pytest.mark.gpu

RUN = 128 * 4096
CASES = {
    "one": [5 * RUN + 17],
    "one_run": [RUN],
    "short_of_a_run": [RUN - 1],
    "past_a_run": [RUN + 1],
    "runs": [RUN, 2 * RUN, RUN],
    "between_short": [100] * 50 + [3 * RUN] + [100] * 50,
    "shifted": [1, 2 * RUN - 1, 3 * RUN + 1, 4095, 2 * RUN],
    "empty_around": [0, 0, 2 * RUN, 0, 0, 0, 2 * RUN + 5, 0],
    "many": [7] * 3000 + [4 * RUN + 3] + [4096] * 40 + [2 * RUN],
    "more_than_warps": [300] * 20_000 + [0, RUN + 3, 9000] + [4096, 8192, 1, 0] * 5_000 + [2 * RUN, 5],
    "ends_in_a_part_tile": [RUN, RUN - 4096 + 1],
}


@pytest.mark.parametrize("case", CASES)
def test_long_instances(case):
    import torch
    sk = skel()
    lens = CASES[case]
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    n = int(off[-1])
    # whole numbers: every order of the sums is exact in float32
    v = torch.randint(0, 2, (n,), device="cuda", dtype=torch.int32).float()
    do = torch.from_numpy(off).cuda()
    res, out = torch.full((len(lens),), -1.0, device="cuda"), torch.full((n,), -1.0, device="cuda")
    s = v.double().cumsum(0)
    before = torch.cat([s.new_zeros(1), s])[do]                       # the sum before each instance's first element
    start = torch.repeat_interleave(before[:-1], do[1:] - do[:-1])
    for inclusive in (True, False):
        with forced("batched", 7, 0, 4, 0):
            sk.skel_batched(wrap(v), wrap(do), wrap(res), wrap(out), inclusive)
        sk.skel_check_device()
        assert torch.equal(res.double(), before[1:] - before[:-1])
        assert torch.equal(out.double(), s - start - (0 if inclusive else v.double()))
    # unsorted offsets are still rejected (instances that the bad offsets make empty may be written)
    bad = do.clone()
    bad[0] = n
    res.fill_(7.0)
    with forced("batched", 7, 0, 4, 0):
        sk.skel_batched(wrap(v), wrap(bad), wrap(res), wrap(out), True)
    with pytest.raises(sk.SkelError):
        sk.skel_check_device()
    assert bool((res[bad[1:] != bad[:-1]] == 7.0).all())


def test_a_stale_rejection_flag_is_not_the_next_calls():
    """A call whose placement rejected its offsets and whose main kernel never
    ran leaves its tag in the scratch's control block; later calls run, past the
    wrap of the tags too."""
    import torch
    sk = skel()
    s, blocks = torch.cuda.Stream(), []

    def alloc(size, stream, ctx):
        blocks.append(torch.zeros(int(size) + 256, dtype=torch.uint8, device="cuda"))
        return (blocks[-1].data_ptr() + 255) // 256 * 256

    a, f = sk._lib.ALLOC_FN(alloc), sk._lib.FREE_FN(lambda p, stream, ctx: None)
    lens = [3000, 5000, 1, 9000]
    off = torch.from_numpy(np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)).cuda()
    v = torch.ones(int(off[-1]), device="cuda")
    res, want = torch.empty(4, device="cuda"), torch.tensor(lens, device="cuda", dtype=torch.float32)
    c = [wrap(v), wrap(off), wrap(res), None]
    torch.cuda.synchronize()
    sk.check(sk.lib.skel_set_allocator(a, f, None))
    try:
        with forced("batched", 7, 0, 4, 0):
            sk.skel_batched(*c, True, stream=s)                 # the call's tag is 1
            s.synchronize()
            assert len(blocks) == 1                             # the stream's scratch
            flag = blocks[0][(-blocks[0].data_ptr()) % 256:][28:32].view(torch.int32)
            flag.fill_(1)                                       # as the failed call would leave it
            for k in range(260):
                res.zero_()
                torch.cuda.synchronize()
                sk.skel_batched(*c, True, stream=s)
                s.synchronize()
                assert torch.equal(res, want), k
            sk.skel_check_device(s)
    finally:
        sk.check(sk.lib.skel_release_cached())
        sk.use_torch_allocator(False)
