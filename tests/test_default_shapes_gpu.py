"""Launch shapes that a plan takes: resident CTAs of the explicit ones, and the form that a large plan
runs by default on aligned and on unaligned buffers."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits", [8, 12])
@pytest.mark.parametrize("mode", [0, 1, 2, 3])
def test_two_ctas_of_sixteen_consumer_warps(cuda, rfi, bits, mode):
    """16 + 1 warps fit twice on an SM in every replacement mode, asked for by the caller or tuned."""
    n, W = 1 << 20, 8192
    for flags in (0, rfi.RFI_PLAN_AUTOTUNE):
        plan = rfi.Plan(bits, [n, n + 3], [W, W], 3.0, mode, flags=flags,
                        shape=dict(consumer_warps=16, ctas_per_sm=2, hist_copies=1, groups=1))
        try:
            assert plan.info().shape.consumer_warps == 16 and plan.info().shape.ctas_per_sm == 2
        finally:
            plan.close()


def _best_ms(call, reps=6):
    import torch
    best = 1e9
    for _ in range(reps):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        call()
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b))
    return best


@pytest.mark.parametrize("flags", ["", "graph", "write flagged"])
def test_large_plans_on_unaligned_buffers(cuda, rfi, flags):
    """A large int8 plan takes the split-warp form for aligned buffers; buffers one byte off run as fast
    as in the joint form (the split form takes half as long again), with the same results."""
    import torch
    n, W = 1 << 27, 16384
    bits = {"": 0, "graph": rfi.RFI_PLAN_GRAPH, "write flagged": rfi.RFI_PLAN_WRITE_FLAGGED}[flags]
    g = torch.Generator(device="cuda").manual_seed(3)
    src = torch.randn(n, device="cuda", generator=g).mul_(16.0).round_().clamp_(-128, 127).to(torch.int8)
    raw, dst = torch.zeros(n + 64, dtype=torch.int8, device="cuda"), torch.zeros(n + 64, dtype=torch.int8, device="cuda")
    plans = [rfi.Plan(8, [n], [W], 3.0, 0, flags=bits, shape=s) for s in (None, dict(warp_split=1))]
    try:
        assert [p.info().shape.warp_split for p in plans] == [2, 1]
        masks = [torch.zeros(p.mask_words(0), dtype=torch.int32, device="cuda") for p in plans]
        counts = [torch.zeros(p.num_windows[0], dtype=torch.int32, device="cuda") for p in plans]
        for off in (0, 1, 0):
            x = raw[off:off + n]
            z = x if flags == "write flagged" else dst[off:off + n]
            got, ms = [], []
            for p, m, c in zip(plans, masks, counts):
                x.copy_(src)
                p.excise([x], [z], [m], [c])
                got.append(z.clone())
                ms.append(_best_ms(lambda: p.excise([x], [z], [m], [c])))
                x.copy_(src)
                p.excise([x], [z], [m], [c])
            assert torch.equal(got[0], got[1]) and not torch.equal(got[0], src)
            assert torch.equal(masks[0], masks[1]) and torch.equal(counts[0], counts[1])
            assert ms[0] < 1.2 * ms[1], (off, ms)
    finally:
        for p in plans:
            p.close()
