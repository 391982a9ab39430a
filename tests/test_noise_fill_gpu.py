"""The digital-noise pass (noise_fill_kernel) at the edges of its work split, against the oracle bit
for bit: units of 256 mask words, groups of 32 nonzero words, batches of 32 flagged samples."""
import numpy as np
import pytest

from .parity import assert_same, gpu_run, oracle_run

pytestmark = pytest.mark.gpu


def _stream(bits, n, W, spots, seed):
    """Noise between -2 and 2 (D = 1 or 2) with large samples at the given positions."""
    r = np.random.default_rng(seed)
    x = r.integers(-2, 3, size=n).astype(np.int8 if bits == 8 else np.int16)
    x[spots[spots < n]] = 100
    return x


@pytest.mark.parametrize("bits", [8, 12])
@pytest.mark.parametrize("W", [31, 32, 33, 1000, 4096, 8192, 16384])
def test_flags_at_unit_group_and_batch_edges(cuda, rfi, bits, W):
    """Streams one word around a unit of 256 mask words; 31, 32, 33, 64 and 65 nonzero words; 31 to
    65 flagged samples in one word and in many; nearly every sample flagged (k small: every sample
    off the median)."""
    words = (W + 31) // 32
    per = max(1, 256 // words) * W  # samples of about one unit
    lens = [max(1, per - 1), per, per + 1, 2 * per + 33, 3 * per]
    xs = []
    for i, n in enumerate(lens):
        a = np.arange(n)
        spots = {0: a[:0], 1: a[::32][:31], 2: np.concatenate([a[::32][:32], a[-1:]]), 3: a[: 65],
                 4: np.concatenate([a[7::32][:65], a[n // 2: n // 2 + 40]])}[i]
        xs.append(_stream(bits, n, W, spots, 50 + i))
    for k in (3.0, 0.01):
        ref = oracle_run(xs, [W] * len(xs), bits, k, 3, 0, 11)
        got, st, totals, info = gpu_run(rfi, xs, [W] * len(xs), bits, k, 3, seed=11, calls=2,
                                        flags=rfi.RFI_PLAN_NOISE_PASS | rfi.RFI_PLAN_GRAPH)
        assert st == 0 and info.kernels_per_call == 2
        assert_same(got, ref, "bits %d W %d k %g" % (bits, W, k))
        assert totals.flagged == sum(int(r["counts"].sum()) for r in ref)


@pytest.mark.parametrize("bits", [8, 12])
def test_wide_spreads_and_saturation(cuda, rfi, bits):
    """Windows whose D spans the sample range, so that values round near both ends and saturate."""
    span = 255 if bits == 8 else 4095
    lo = -128 if bits == 8 else -2048
    r = np.random.default_rng(3)
    W, xs = 512, []
    for c in (0.05, 0.3, 0.5, 0.8, 1.0):
        u = lo + np.rint(span * (0.5 + c * (r.random(6 * W) - 0.5)))
        xs.append(u.astype(np.int8 if bits == 8 else np.int16))
    xs.append(np.where(np.arange(6 * W) % 3 == 0, lo, lo + span).astype(np.int8 if bits == 8 else np.int16))
    for k in (0.01, 0.4):
        ref = oracle_run(xs, [W] * len(xs), bits, k, 3, 0, (5 << 40) + 9)
        for flags in (rfi.RFI_PLAN_NOISE_PASS, 0):
            got, st, _, _ = gpu_run(rfi, xs, [W] * len(xs), bits, k, 3, seed=(5 << 40) + 9, flags=flags)
            assert st == 0
            assert_same(got, ref, "bits %d k %g flags %d" % (bits, k, flags))
