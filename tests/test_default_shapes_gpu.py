"""Launch shapes that a plan takes: resident CTAs of the explicit ones."""
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
