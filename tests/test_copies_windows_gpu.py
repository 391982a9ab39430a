"""Digital copies, window by window: the counts of every variant over many windows, and the mask of a
short last window."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


def _popcounts(mask, nwin):
    """Set bits of every window of a mask of nwin windows."""
    import torch
    bits = (mask.view(nwin, -1, 1) >> torch.arange(32, device=mask.device, dtype=torch.int32)) & 1
    return bits.sum(dim=(1, 2))


def test_every_variant_counts_every_window(cuda, rfi):
    """Eight variants of two multiples on many short windows: each variant's flag count, added by a lane
    of its own, is in when the window's last warp writes it."""
    import torch
    variants = [(k, m, 5, v) for v, (k, m) in enumerate([(2.0, 0), (3.0, 1), (2.0, 2), (3.0, 3), (2.0, 1), (3.0, 0), (2.0, 3), (3.0, 2)])]
    W, n = 512, 1 << 21
    p = synth.params(seed=3, sigma=16.0, burst_rate=1e-2, burst_len_max=64, bits=8)
    x = torch.from_numpy(synth.fill(p, 0, n)).cuda()
    plan = rfi.CopiesPlan(8, [n], [W], variants)
    try:
        nwin = plan.num_windows[0]
        outs = [[torch.empty_like(x)] for _ in variants]
        masks = [[torch.full((plan.mask_words(0),), -1, dtype=torch.int32, device="cuda")] for _ in variants]
        for call in range(4):
            counts = [[torch.full((nwin,), -1, dtype=torch.int32, device="cuda")] for _ in variants]
            plan.excise([x], outs, masks, counts)
            st, totals = plan.stats()
            assert st == 0
            for v in range(len(variants)):
                assert torch.equal(counts[v][0].to(torch.int64), _popcounts(masks[v][0], nwin)), (call, v)
            assert totals.flagged == sum(int(c[0].sum()) for c in counts)
    finally:
        plan.close()


@pytest.mark.parametrize("W,tail", [(16384, 512), (16384, 15872), (4096, 2048), (1000, 512), (560, 512)])
def test_mask_ends_with_zeros_after_a_short_last_window(cuda, rfi, W, tail):
    """The last window holds a multiple of 512 samples and less than W: its mask words past the last
    sample are written as 0 for every variant, whatever the buffer held."""
    import torch
    variants = [(3.0, 0, 0, 0), (3.0, 3, 0, 7), (5.0, 2, 0, 0), (3.0, 1, 9, 0)]
    n = 3 * W + tail
    p = synth.params(seed=11, sigma=16.0, burst_rate=1e-2, burst_len_max=64, bits=8)
    x = synth.fill(p, 0, n)
    plan = rfi.CopiesPlan(8, [n], [W], variants)
    try:
        xd = torch.from_numpy(x).cuda()
        outs = [[torch.empty_like(xd)] for _ in variants]
        masks = [[torch.full((plan.mask_words(0),), -1, dtype=torch.int32, device="cuda")] for _ in variants]
        plan.excise([xd], outs, masks)
        for v, (k, mode, const, seed) in enumerate(variants):
            r = oracle.excise(x, W, k, mode, const=const, seed=seed, stream_id=0)
            assert np.array_equal(masks[v][0].cpu().numpy().view(np.uint32), r["mask"]), v
            assert np.array_equal(outs[v][0].cpu().numpy(), r["z"]), v
    finally:
        plan.close()
