"""The digital-noise pass around the size from which its warps share units through the cursor, against
the noise of the excision kernel."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits", [8, 12])
@pytest.mark.parametrize("share", [0.51, 0.999, 1.0, 1.001, 2.3])
def test_units_with_a_warp_of_their_own_and_shared_ones(cuda, rfi, bits, share):
    """From a unit less to one more than a warp each (units of 256 mask words, five CTAs of eight
    warps per SM), and the sizes below and above: the same samples as the one-pass form."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    W = 8192
    n = int(share * 256 * 8 * 5 * sms) * 32 + (W if share > 1 else 0)
    g = torch.Generator(device="cuda").manual_seed(5)
    x = torch.randn(n, device="cuda", generator=g).mul_(16.0).round_().clamp_(-100, 100).to(torch.int8 if bits == 8 else torch.int16)
    got = []
    for flags in (0, rfi.RFI_PLAN_NOISE_PASS):
        plan = rfi.Plan(bits, [n], [W], 3.0, 3, 0, 7, flags)
        try:
            z = torch.empty_like(x)
            for _ in range(2):
                plan.excise([x], [z])
            assert plan.stats()[0] == 0
            got.append(z)
        finally:
            plan.close()
    assert torch.equal(got[0], got[1]) and not torch.equal(got[0], x)
