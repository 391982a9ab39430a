"""The 12-bit median and MAD search over rows of 16 bins, and digital noise in slices of a window,
against the CPU oracle, bit for bit."""
import numpy as np
import pytest

from .parity import assert_same, gpu_run, oracle_run

pytestmark = pytest.mark.gpu


def _window(r, n, kind):
    if kind == 0:    # one value, at either end of the range or inside
        return np.full(n, r.choice([-2048, 2047, 0, -1, 15, 16]))
    if kind == 1:    # two far values: D is 0 or the whole span
        return np.where(r.random(n) < r.choice([0.3, 0.49, 0.51, 0.7]), -2048, 2047)
    if kind == 2:    # uniform over the range
        return r.integers(-2048, 2048, size=n)
    if kind == 3:    # narrow, around a row boundary
        return r.integers(-3, 4, size=n) + 16 * r.integers(-127, 127) + r.integers(-1, 2)
    if kind == 4:    # heavy at both ends with a thin middle
        return np.where(r.random(n) < 0.5, r.integers(-2048, -2030, size=n), r.integers(2030, 2048, size=n))
    if kind == 5:    # one-sided: M at the bottom of the range
        return np.minimum(2047, -2048 + (r.exponential(r.choice([2, 40, 900]), size=n)).astype(int))
    return np.clip(np.rint(r.normal(r.integers(-1900, 1900), r.choice([1, 7, 15, 16, 120, 700]), size=n)), -2048, 2047)


@pytest.mark.parametrize("copies", [0, 1, 2, 4])
@pytest.mark.parametrize("cw", [4, 8, 16])
def test_median_and_mad_of_every_kind_of_window(cuda, rfi, cw, copies):
    r = np.random.default_rng(77)
    wins = [1, 2, 16, 100, 1024, 2048, 829]
    xs = [np.concatenate([_window(r, W, k % 7) for k in range(28)]).astype(np.int16) for W in wins]
    shape = dict(consumer_warps=cw, hist_copies=copies)
    for k in (3.0, 0.5):
        ref = oracle_run(xs, wins, 12, k, 3, 0, 3)
        got, st, _, _ = gpu_run(rfi, xs, wins, 12, k, 3, 0, 3, flags=rfi.RFI_PLAN_NO_SPLIT, shape=shape, calls=2)
        assert st == 0
        assert_same(got, ref, "cw %d copies %d k %g" % (cw, copies, k))


@pytest.mark.parametrize("W", [8184, 8191, 8192, 8193, 16384, 20001, 65536])
def test_noise_in_slices(cuda, rfi, W):
    """Windows around a slice of 8192 (any-window form 8184) samples and of several, with few, half and
    nearly all of the samples flagged (the list holds half a slice)."""
    r = np.random.default_rng(W)
    xs = [np.clip(np.rint(r.normal(0, 120, size=2 * W + 77)), -2048, 2047).astype(np.int16) for _ in range(2)]
    xs[1][::2] = np.where(r.random(xs[1][::2].size) < 0.5, 1500, -1500)
    for k in (3.0, 0.6, 0.01):
        ref = oracle_run(xs, [W] * 2, 12, k, 3, 0, 4)
        for flags in (0, rfi.RFI_PLAN_PER_STREAM):
            got, st, totals, _ = gpu_run(rfi, xs, [W] * 2, 12, k, 3, 0, 4, flags=flags, calls=2)
            assert st == 0
            assert_same(got, ref, "W %d k %g flags %d" % (W, k, flags))
            assert totals.flagged == sum(int(x["counts"].sum()) for x in ref)
