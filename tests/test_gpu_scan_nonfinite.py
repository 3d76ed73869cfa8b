"""Scans over infinities, infinities of both signs, NaN and sums that leave
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
