"""Digital copies whose variants share threshold multiples (one pass per multiple), against the CPU
oracle, bit for bit: every replacement in a group, two noise keys of one multiple, groups that
interleave, and the buffers and windows that take one variant at a time."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

GROUPS = [
    [(3.0, 0, 0, 0), (3.0, 1, 5, 0), (3.0, 2, 0, 0), (3.0, 3, 0, 7), (3.0, 3, 0, 8)],
    [(3.0, 3, 0, 1), (5.0, 3, 0, 2), (3.0, 1, -9, 0), (5.0, 2, 0, 0), (2.0, 0, 0, 0), (3.0, 1, 77, 0), (5.0, 3, 0, 3), (0.01, 3, 0, 4)],
    [(4.0, 2, 0, 0)],
]


@pytest.mark.parametrize("variants", GROUPS)
@pytest.mark.parametrize("form", ["plain", "no mask", "odd window", "offset", "tail"])
def test_variants_of_one_multiple(cuda, rfi, variants, form):
    import torch
    wins = [512, 16384, 4096] if form != "odd window" else [520, 16000, 1000]
    lens = [W * 7 + (100 if form == "tail" else 0) for W in wins]
    p = synth.params(seed=9, sigma=16.0, burst_rate=1e-2, burst_len_max=64, bits=8)
    xs = [synth.fill(p, s, n) for s, n in enumerate(lens)]
    xs[2][4096:8192] = 3  # a window with D = 0 flags nothing
    S, V, off = len(xs), len(variants), 3 if form == "offset" else 0
    plan = rfi.CopiesPlan(8, lens, wins, variants)
    try:
        ins = [torch.from_numpy(x).cuda() for x in xs]
        raw = [[torch.full((n + 16,), 0x5A, dtype=torch.int8, device="cuda") for n in lens] for _ in range(V)]
        outs = [[t[off:off + n] for t, n in zip(r, lens)] for r in raw]
        masks = [[torch.full((plan.mask_words(s),), -1, dtype=torch.int32, device="cuda") for s in range(S)] for _ in range(V)]
        counts = [[torch.full((n,), -1, dtype=torch.int32, device="cuda") for n in plan.num_windows] for _ in range(V)]
        given = [[None if form == "no mask" and (v + s) % 3 == 0 else masks[v][s] for s in range(S)] for v in range(V)]
        for _ in range(2):
            plan.excise(ins, outs, given, counts)
        st, totals = plan.stats()
        assert st == 0
        flagged = 0
        for v, (k, mode, const, seed) in enumerate(variants):
            for s, x in enumerate(xs):
                r = oracle.excise(x, wins[s], k, mode, const=const, seed=seed, stream_id=s)
                what = "variant %d stream %d" % (v, s)
                assert np.array_equal(outs[v][s].cpu().numpy(), r["z"]), what
                if given[v][s] is not None:
                    assert np.array_equal(masks[v][s].cpu().numpy().view(np.uint32), r["mask"]), what
                assert np.array_equal(counts[v][s].cpu().numpy().view(np.uint32), r["counts"]), what
                assert (raw[v][s][:off] == 0x5A).all() and (raw[v][s][off + lens[s]:] == 0x5A).all(), what
                flagged += int(r["counts"].sum())
        assert totals.flagged == flagged
    finally:
        plan.close()
