"""Explicit launch shapes close to the shared memory of an SM, against the CPU oracle, bit for bit: the plans
that fit in one form of a kernel and not in another."""
import pytest

import synth

from .parity import assert_same, gpu_run, oracle_run

pytestmark = pytest.mark.gpu


def _streams(bits, lens):
    p = synth.params(seed=21, sigma=16.0 if bits == 8 else 120.0, burst_rate=5e-3, burst_len_max=64, bits=bits)
    return [synth.fill(p, s, n) for s, n in enumerate(lens)]


@pytest.mark.parametrize("bits,W,mode,flags,shape", [
    (8, 65001, 0, 0, dict(stages=3)), (8, 48500, 2, 0, dict(stages=4)), (8, 59501, 3, 0, dict(stages=3)),
    (8, 24570, 0, 0, dict(stages=8)), (12, 31613, 3, 0, dict(stages=3)),
    (8, 3200, 0, "tune", dict(stage_bytes=6400)), (8, 3200, 3, "tune", dict(stage_bytes=12800, stages=2)),
])
def test_odd_windows_in_shapes_that_only_the_aligned_form_fits(cuda, rfi, bits, W, mode, flags, shape):
    """Windows that the any-window form would serve, in shapes that it has no room or no stage size for."""
    lens = [W * 3 + 77, W * 2]
    xs = _streams(bits, lens)
    ref = oracle_run(xs, [W] * 2, bits, 3.0, mode, 0, 5)
    got, st, _, info = gpu_run(rfi, xs, [W] * 2, bits, 3.0, mode, 0, 5, flags=rfi.RFI_PLAN_AUTOTUNE if flags else 0, shape=shape)
    assert st == 0
    assert_same(got, ref)
    for field, v in shape.items():
        assert getattr(info.shape, field) == v


@pytest.mark.parametrize("bits,W,shape", [(8, 59648, dict(stages=3)), (8, 26752, dict(stages=7)), (12, 31488, dict(stages=3, hist_copies=1)),
                                          (12, 23296, dict(stages=3, hist_copies=4))])
def test_copies_in_the_largest_stages_that_fit(cuda, rfi, bits, W, shape):
    """Digital copies whose window fills the largest stage of that number: as with the default shape."""
    import torch
    variants = [(3.0, 0, 0, 0), (3.0, 3, 0, 7), (4.0, 2, 0, 0), (3.0, 1, 5, 0)]
    lens = [W * 4, W * 2 + 512]
    xs = [torch.from_numpy(x).cuda() for x in _streams(bits, lens)]
    res = []
    for s in (shape, None):
        plan = rfi.CopiesPlan(bits, lens, [W] * 2, variants, shape=s)
        try:
            outs = [[torch.empty_like(x) for x in xs] for _ in variants]
            masks = [[torch.full((plan.mask_words(i),), -1, dtype=torch.int32, device="cuda") for i in range(2)] for _ in variants]
            for _ in range(2):
                plan.excise(xs, outs, masks)
            assert plan.stats()[0] == 0 and (s is None or plan.info().shape.stages == s["stages"])
            res.append((sum(outs, []), sum(masks, [])))
        finally:
            plan.close()
    assert all(torch.equal(a, b) for k in range(2) for a, b in zip(res[0][k], res[1][k]))


@pytest.mark.parametrize("W,shape", [(32960, dict(stages=3, hist_copies=1)), (22656, dict(stages=4, hist_copies=2)),
                                     (9280, dict(stages=8, hist_copies=4)), (32953, dict(stages=3, hist_copies=1))])
def test_estimation_in_the_largest_stages_that_fit(cuda, rfi, W, shape):
    """12-bit Median of MAD whose window fills the largest stage of that number: as with the default
    shape, window for window."""
    import torch
    lens = [W * 9 + 8, W * 4, W]
    xs = [torch.from_numpy(x).cuda() for x in _streams(12, lens)]
    res = []
    for s in (shape, None):
        plan = rfi.Plan(12, lens, [W] * 3, 3.0, 2, 0, 0, 0, None, s, 4)
        try:
            outs = [torch.empty_like(x) for x in xs]
            meds, mads, moms = [[torch.full((n,), -99, dtype=torch.int32, device="cuda") for n in plan.num_windows] for _ in range(3)]
            for _ in range(2):
                plan.excise(xs, outs)
            st, _ = plan.stats(meds, mads)
            plan.stats_mom(moms)
            torch.cuda.synchronize()
            assert st == 0 and (s is None or plan.info().shape.stages == s["stages"])
            res.append(outs + meds + mads + moms)
        finally:
            plan.close()
    assert all(torch.equal(a, b) for a, b in zip(*res))
