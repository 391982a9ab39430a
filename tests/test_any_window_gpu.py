"""The any-window form (windows of any length at any alignment, staged as they lie in memory) against
the CPU oracle, bit for bit: windows that start and end anywhere in a 16-byte chunk, several to a
histogram table or one at a time, whole tiles and their remainders, and the plans that choose it."""
import numpy as np
import pytest

import oracle
import synth

from .parity import assert_same, gpu_run, oracle_run

pytestmark = pytest.mark.gpu


def _streams(bits, lens, seed, rate=8e-3):
    p = synth.params(seed=seed, sigma=16.0 if bits == 8 else 120.0, burst_rate=rate, burst_len_max=64, bits=bits)
    return [synth.fill(p, s, n) for s, n in enumerate(lens)]


@pytest.mark.parametrize("mode", [0, 1, 2, 3])
@pytest.mark.parametrize("bits", [8, 12])
def test_windows_of_every_remainder(cuda, rfi, bits, mode):
    """Windows around the chunk (16 bytes), round (31 chunks) and table (8192 samples) sizes; tiles of
    every number of windows; tails of one sample up to a window less one; every buffer alignment."""
    wins = [1, 2, 7, 15, 16, 17, 31, 33, 100, 495, 496, 497, 777, 1000, 2000, 4097, 5000, 8191, 8192, 8193, 12500, 16383, 16384]
    lens = [W * (3 + i % 9) + (0, 1, W - 1, W // 2)[i % 4] + 17 for i, W in enumerate(wins)]
    xs = _streams(bits, lens, 40 + mode)
    c = 3 if mode == 1 else 0
    ref = oracle_run(xs, wins, bits, 3.0, mode, c, 9)
    for offset in (0, 2, 6, 14) if bits == 12 else (0, 1, 7, 15):
        for in_place in (False, True):
            got, st, totals, info = gpu_run(rfi, xs, wins, bits, 3.0, mode, c, 9, flags=rfi.RFI_PLAN_NO_SPLIT, offset=offset,
                                            in_place=in_place)
            assert st == 0
            assert_same(got, ref, "bits %d mode %d offset %d in place %s" % (bits, mode, offset, in_place))
            assert totals.flagged == sum(int(r["counts"].sum()) for r in ref)


@pytest.mark.parametrize("bits", [8, 12])
def test_split_graph_noise_pass_and_autotuned_plans(cuda, rfi, bits):
    wins = [1000, 12500, 20001, 50000, 4096, 16384, 777]
    lens = [W * 5 + 123 for W in wins]
    xs = _streams(bits, lens, 7)
    ref = oracle_run(xs, wins, bits, 3.0, 3, 0, 5)
    for flags in (0, rfi.RFI_PLAN_GRAPH, rfi.RFI_PLAN_NOISE_PASS, rfi.RFI_PLAN_GRAPH | rfi.RFI_PLAN_AUTOTUNE,
                  rfi.RFI_PLAN_AUTOTUNE | rfi.RFI_PLAN_NOISE_PASS | rfi.RFI_PLAN_NO_SPLIT):
        got, st, _, _ = gpu_run(rfi, xs, wins, bits, 3.0, 3, 0, 5, flags=flags, calls=2)
        assert st == 0
        assert_same(got, ref, "bits %d flags %x" % (bits, flags))


@pytest.mark.parametrize("shape", [dict(stage_bytes=2048, stages=3, ctas_per_sm=1), dict(stage_bytes=65536, stages=1),
                                   dict(consumer_warps=4), dict(groups=2, consumer_warps=8), dict(dynamic_tiles=2)])
def test_launch_shapes(cuda, rfi, shape):
    """Stages that hold one, a few and many windows; shapes that keep the aligned form."""
    wins = [1000, 333, 5000, 16384]  # (no 2^l <= 8192: the multi-window form refuses two groups)
    lens = [W * 41 + 5 for W in wins]
    xs = _streams(8, lens, 8)
    for mode in (2, 3):
        ref = oracle_run(xs, wins, 8, 3.0, mode, 0, 5)
        got, st, _, _ = gpu_run(rfi, xs, wins, 8, 3.0, mode, 0, 5, flags=rfi.RFI_PLAN_NO_SPLIT, shape=shape, calls=2)
        assert st == 0
        assert_same(got, ref, "%s mode %d" % (shape, mode))


@pytest.mark.parametrize("bits", [8, 12])
def test_in_and_out_aligned_differently_and_out_of_range(cuda, rfi, bits):
    import torch
    wins, n = [777, 12500], [777 * 9 + 5, 12500 * 2 + 1]
    xs = _streams(bits, n, 9)
    es = xs[0].itemsize
    ref = oracle_run(xs, wins, bits, 3.0, 3, 0, 5)
    plan = rfi.Plan(bits, n, wins, 3.0, 3, 0, 5, rfi.RFI_PLAN_NO_SPLIT)
    try:
        raw = [torch.zeros(x.size * es + 64, dtype=torch.uint8, device="cuda") for x in xs]
        out = [torch.full_like(r, 0x5A) for r in raw]
        for r, x in zip(raw, xs):
            r[6:6 + x.size * es] = torch.from_numpy(x.view(np.uint8).copy())
        plan.excise([r.data_ptr() + 6 for r in raw], [o.data_ptr() + 2 for o in out])
        st, _ = plan.stats()
        assert st == 0
        for o, x, r in zip(out, xs, ref):
            z = o.cpu().numpy()
            assert np.array_equal(z[2:2 + x.size * es].view(x.dtype), r["z"])
            assert (z[:2] == 0x5A).all() and (z[2 + x.size * es:] == 0x5A).all()
        if bits == 12:  # a sample out of range anywhere in a window is reported
            for at in (0, 776, 777, n[0] - 1):
                bad = xs[0].copy()
                bad[at] = 3000
                raw[0][6:6 + bad.size * es] = torch.from_numpy(bad.view(np.uint8).copy())
                plan.excise([r.data_ptr() + 6 for r in raw], [o.data_ptr() + 2 for o in out])
                assert plan.stats()[0] == rfi.RFI_ERR_SAMPLE_RANGE
    finally:
        plan.close()


@pytest.mark.parametrize("noise_pass", [False, True])
@pytest.mark.parametrize("bits", [8, 12])
def test_median_of_mad(cuda, rfi, bits, noise_pass):
    import torch
    wins = [1000, 333, 12500, 4096]
    lens = [W * 37 + 11 for W in wins]
    xs = _streams(bits, lens, 10)
    for mode in (2, 3):
        plan = rfi.Plan(bits, lens, wins, 3.0, mode, 0, 6, rfi.RFI_PLAN_NOISE_PASS if noise_pass else 0, mom_windows=7)
        try:
            ins = [torch.from_numpy(x).cuda() for x in xs]
            outs = [torch.zeros_like(t) for t in ins]
            masks = [torch.zeros(plan.mask_words(i), dtype=torch.int32, device="cuda") for i in range(len(xs))]
            counts = [torch.zeros(v, dtype=torch.int32, device="cuda") for v in plan.num_windows]
            meds = [torch.zeros_like(c) for c in counts]
            mads = [torch.zeros_like(c) for c in counts]
            plan.excise(ins, outs, masks, counts)
            st, _ = plan.stats(meds, mads)
            assert st == 0
            for i, x in enumerate(xs):
                r = oracle.excise_mom(x, wins[i], 3.0, mode, 7, seed=6, stream_id=i, bits=bits)
                assert np.array_equal(meds[i].cpu().numpy(), r["median"]), i
                assert np.array_equal(mads[i].cpu().numpy(), r["mad"]), i
                assert np.array_equal(outs[i].cpu().numpy(), r["z"]), i
                assert np.array_equal(masks[i].cpu().numpy().view(np.uint32), r["mask"]), i
                assert np.array_equal(counts[i].cpu().numpy().view(np.uint32), r["counts"]), i
        finally:
            plan.close()


@pytest.mark.parametrize("bits,W", [(8, 1000), (8, 12500), (12, 1000), (12, 12500)])
def test_noise_of_windows_across_two_to_the_32(cuda, rfi, bits, W):
    """A stream of 2^32 samples and some, all zero but the last 100000: the noise of a window (and, in
    windows of 1000, of a tile of several) whose sample indices pass 2^32."""
    import torch
    n = (1 << 32) + 50_000
    w0 = ((1 << 32) - 50_000) // W  # first window compared
    x = torch.zeros(n, dtype=torch.int8 if bits == 8 else torch.int16, device="cuda")
    tail = _streams(bits, [n - w0 * W], 12, 2e-2)[0]
    x[w0 * W:] = torch.from_numpy(tail).cuda()
    z = torch.empty_like(x)
    plan = rfi.Plan(bits, [n], [W], 3.0, 3, 0, 99)
    try:
        plan.excise([x], [z])
        assert plan.stats()[0] == 0
    finally:
        plan.close()
    ref = oracle.excise(tail, W, 3.0, 3, seed=99, abs0=w0 * W, bits=bits)
    assert np.array_equal(z[w0 * W:].cpu().numpy(), ref["z"])
    assert not z[:w0 * W].any()


@pytest.mark.parametrize("bits", [8, 12])
def test_served_noise_across_two_to_the_32(cuda, rfi, bits):
    """Aligned windows that pass 2^32 (a served stream may start there)."""
    import torch
    W, start = 10000, ((1 << 32) // 10000 - 1) * 10000
    x = _streams(bits, [4 * W], 13, 2e-2)[0]
    sv = rfi.Server(bits, [W], 8 * W, 3.0, 3, 0, 21, memory_budget=64 << 20, stream_start=[start])
    try:
        t = torch.from_numpy(x).cuda()
        torch.cuda.synchronize()
        assert sv.push(0, t)[0] == 0
        sv.drain(10.0)
        z = torch.zeros_like(t)
        assert sv.read(0, start, x.size, z) == 0
        ref = oracle.excise(x, W, 3.0, 3, seed=21, abs0=start, bits=bits)
        assert np.array_equal(z.cpu().numpy(), ref["z"])
    finally:
        sv.close()
