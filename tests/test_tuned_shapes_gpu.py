"""Tuned plans whose shape comes from the cache: it holds their windows and honours their constraints."""
import pytest

import synth

from .parity import assert_same, gpu_run, oracle_run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cache", ["process", "file"])
@pytest.mark.parametrize("bits", [8, 12])
def test_streams_shorter_than_their_window(cuda, rfi, bits, cache, tmp_path, monkeypatch):
    """Plans that differ only in the length of a stream shorter than its window, short ones tuned first."""
    if cache == "file":
        monkeypatch.setenv("RFI_TUNE_CACHE", str(tmp_path / "tuned"))
    W = 32768 if bits == 12 else 65536
    p = synth.params(seed=4, sigma=16.0, burst_rate=5e-3, burst_len_max=64, bits=bits)
    for n in (100 + bits, 4001, W - 9 - bits):
        xs = [synth.fill(p, 0, n)]
        for _ in range(2):  # the second takes the first one's shape
            got, st, _, info = gpu_run(rfi, xs, [W], bits, 3.0, 2, flags=rfi.RFI_PLAN_AUTOTUNE)
            assert st == 0 and info.shape.stage_bytes >= n * (bits // 8 + (bits == 12))
            assert_same(got, oracle_run(xs, [W], bits, 3.0, 2))


def test_constraints_after_a_tuned_plan_without(cuda, rfi):
    """The same layout tuned without constraints, with one, with another and without again."""
    lens, wins = [1 << 18, (1 << 18) + 77], [16384, 16384]
    free = []
    for shape in (None, dict(stages=3), dict(consumer_warps=4, dynamic_tiles=1), None, dict(stages=3)):
        plan = rfi.Plan(8, lens, wins, 3.0, 1, flags=rfi.RFI_PLAN_AUTOTUNE, shape=shape)
        try:
            got = plan.info().shape
            for field, v in (shape or {}).items():
                assert getattr(got, field) == v
            if shape is None:
                free.append([getattr(got, f) for f, _ in got._fields_])
        finally:
            plan.close()
    assert free[0] == free[1]
