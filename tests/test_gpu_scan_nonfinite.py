"""Scans (also of batched instances) over infinities, infinities of both signs, NaN and sums that leave
float32's range: the outputs are infinite and NaN exactly where the prefix sums
in 64 bits, rounded to float32, are."""
import numpy as np
import pytest

from helpers import SUM_REL, dev_empty, dev_tensor, forced, skel, to_np, wrap

pytestmark = pytest.mark.gpu

VARIANTS = list(range(10))
SHAPES = [(300_003,), (5_000_012,), (3, 55_296), (7, 8191), (90, 257), (5, 130)]
INF, NAN = np.float32(np.inf), np.float32(np.nan)
# values at fractions of the sequence (of every second row)
PATTERNS = {
    "inf": [(0.4, INF)],
    "minus_inf_first": [(0.0, -INF)],
    "inf_last": [(1.0, INF)],
    "inf_then_minus_inf": [(0.3, INF), (0.6, -INF)],
    "both_next_to_each_other": [(0.5, -INF), (0.5, INF)],
    "nan": [(0.25, NAN)],
    "overflow": [(0.2, np.float32(3e38)), (0.7, np.float32(3e38))],
    "overflow_close": [(0.5, np.float32(-3e38)), (0.5, np.float32(-3e38))],
}


def sequence(shape, pattern):
    x = np.ones(shape, np.float32)
    n = shape[-1]
    for k, (at, v) in enumerate(PATTERNS[pattern]):
        x[(slice(None, None, 2),) * (len(shape) - 1) + (min(int(at * n) + k, n - 1),)] = v
    return x


def prefixes(x, inclusive, reverse):
    """Prefix sums in 64 bits, and those of the magnitudes."""
    with np.errstate(all="ignore"):
        y = (x[..., ::-1] if reverse else x).astype(np.float64)
        s, a = y.cumsum(-1), np.abs(y).cumsum(-1)
        if not inclusive:
            s, a = (np.concatenate([np.zeros_like(v[..., :1]), v[..., :-1]], -1) for v in (s, a))
        if reverse:
            s, a = s[..., ::-1], a[..., ::-1]
        return s, a


@pytest.mark.parametrize("variant", VARIANTS)
@pytest.mark.parametrize("shape", SHAPES, ids=str)
@pytest.mark.parametrize("pattern", PATTERNS)
def test_scan(variant, shape, pattern):
    import torch
    sk = skel()
    x = sequence(shape, pattern)
    dx, out = wrap(dev_tensor(x)), dev_empty(shape, torch.float32)
    for reverse in (False, True):
        for inclusive in (True, False):
            try:
                with forced("scan", variant):
                    (sk.skel_scan_bwd if reverse else sk.skel_scan)("add", inclusive, dx, wrap(out))
            except sk.SkelError as e:
                assert e.code == -4     # the variant is not offered for this shape
                continue
            got = to_np(out)
            want, mag = prefixes(x, inclusive, reverse)
            with np.errstate(all="ignore"):
                rounded = want.astype(np.float32)
                special = ~np.isfinite(rounded)
                assert np.array_equal(got[special], rounded[special], equal_nan=True)
                assert np.all(np.abs(got[~special] - want[~special]) <= SUM_REL * mag[~special])


LENS = [5, 300_003, 0, 4096, 130, 8191, 1, 70_000]


@pytest.mark.parametrize("variant,tile", [(0, 0), (1, 0), (2, 0), (3, 0), (4, 0), (5, 0), (6, 0), (6, 1), (7, 0), (7, 1)])
@pytest.mark.parametrize("pattern", PATTERNS)
def test_batched(variant, tile, pattern):
    """The pattern in every second instance; the others stay finite."""
    import torch
    sk = skel()
    parts = [sequence((n,), pattern) if k % 2 and n else np.ones(n, np.float32) for k, n in enumerate(LENS)]
    off = np.concatenate([[0], np.cumsum(LENS)]).astype(np.int64)
    cv, co = wrap(dev_tensor(np.concatenate(parts))), wrap(dev_tensor(off))
    res, out = dev_empty((len(LENS),), torch.float32), dev_empty((int(off[-1]),), torch.float32)
    for inclusive in (True, False):
        with forced("batched", variant, 0, 4, tile):
            sk.skel_batched(cv, co, wrap(res), wrap(out), inclusive)
        sums, got = to_np(res).copy(), to_np(out).copy()
        for k, x in enumerate(parts):
            want, mag = prefixes(x, inclusive, False)
            g = got[off[k]:off[k + 1]]
            with np.errstate(all="ignore"):
                rounded = want.astype(np.float32)
                special = ~np.isfinite(rounded)
                assert np.array_equal(g[special], rounded[special], equal_nan=True), k
                assert np.all(np.abs(g[~special] - want[~special]) <= SUM_REL * mag[~special]), k
                sq = np.float32((x.astype(np.float64) ** 2).sum())
                assert np.array_equal(sums[k], sq, equal_nan=True) if not np.isfinite(sq) else abs(sums[k] - sq) <= SUM_REL * sq, k


@pytest.mark.parametrize("shape", [s for s in SHAPES if len(s) == 1], ids=str)
@pytest.mark.parametrize("pattern", PATTERNS)
def test_noalloc(shape, pattern):
    import torch
    sk = skel()
    x = sequence(shape, pattern)
    out = dev_empty(shape, torch.float32)
    for inclusive in (True, False):
        sk.skel_scan_noalloc("add", inclusive, dev_tensor(x), out)
        got, (want, mag) = to_np(out), prefixes(x, inclusive, False)
        with np.errstate(all="ignore"):
            rounded = want.astype(np.float32)
            special = ~np.isfinite(rounded)
            assert np.array_equal(got[special], rounded[special], equal_nan=True)
            assert np.all(np.abs(got[~special] - want[~special]) <= SUM_REL * mag[~special])
