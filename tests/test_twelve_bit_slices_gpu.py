"""12-bit digital noise in windows of several slices, whose flagged samples share a list where the first
slice promises room, against the CPU oracle, bit for bit."""
import numpy as np
import pytest

from .parity import assert_same, gpu_run, oracle_run

pytestmark = pytest.mark.gpu


def _stream(n, W, kind, seed):
    """Noise of a few LSB with large samples: few of them, many, few in the first 8192 samples of
    every window and many after (the list overflows), or the reverse."""
    r = np.random.default_rng(seed)
    x = r.integers(-6, 7, size=n).astype(np.int16)
    at = np.arange(n) % W
    rate = {"few": np.full(n, 0.004), "many": np.full(n, 0.3), "late": np.where(at < 8192, 0.004, 0.4),
            "early": np.where(at < 8192, 0.4, 0.004)}[kind]
    hit = r.random(n) < rate
    hit[[W - 1, n - 1]] = True
    x[hit] = 900
    return x


@pytest.mark.parametrize("kind", ["few", "many", "late", "early"])
@pytest.mark.parametrize("W", [8192, 8200, 16384, 32768, 32776, 65536, 8185, 16369, 32737, 65535])
def test_lists_of_one_and_of_several_slices(cuda, rfi, W, kind):
    """One slice, a slice and a chunk, two, four, four and a chunk, eight, in the aligned form and
    (odd windows) the any-window form."""
    lens = [2 * W, W + 8191, W]
    xs = [_stream(n, W, kind, 70 + i) for i, n in enumerate(lens)]
    ref = oracle_run(xs, [W] * 3, 12, 3.0, 3, 0, 13)
    for flags in (0, rfi.RFI_PLAN_PER_STREAM, rfi.RFI_PLAN_POWER):
        got, st, totals, _ = gpu_run(rfi, xs, [W] * 3, 12, 3.0, 3, seed=13, flags=flags, calls=2)
        assert st == 0
        assert_same(got, ref, "W %d %s flags %x" % (W, kind, flags))
        assert totals.flagged == sum(int(r["counts"].sum()) for r in ref)
