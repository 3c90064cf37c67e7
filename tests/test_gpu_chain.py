"""Chained launches (csrc/lgf_internal.cuh): an apply whose passes may be set up
while their predecessors drain takes no longer than those passes one by one."""
import pytest

import lgf_inputs as li

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _times(ctx, call, reps=20):
    """us of an apply: called back to back, and the sum of its passes with
    profiling events between them (which keep the launches apart)."""
    for _ in range(3):
        call()
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    together, apart = [], []
    for _ in range(5):
        a.record()
        for _ in range(reps):
            call()
        b.record()
        b.synchronize()
        together.append(a.elapsed_time(b) * 1e3 / reps)
        ctx.profile_enable(True)
        for _ in range(reps):
            call()
        torch.cuda.synchronize()
        apart.append(sum(ms for _, ms in ctx.profile_read().values()) * 1e3 / reps)
        ctx.profile_enable(False)
    return min(together), min(apart)


# (the sums of the passes apart include a few us of event time each, so plain
# launches already meet 1.0; CTAs gathered on a few SMs took 1.3 to 2.1)
@pytest.mark.parametrize("b,extent,alpha", [(32, (2, 2, 2), 0.75), (32, (2, 2, 2), 0.25), (8, (4, 4, 4), 0.75)])
def test_chained_integrating_factor_spreads_over_the_sms(ctx64, b, extent, alpha):
    c = li.box_blocks(*extent)
    nf = 3 if b == 8 else 1
    f = torch.randn(nf * c.shape[0] * b ** 3, dtype=torch.float64, device="cuda")
    u = torch.empty_like(f)
    together, apart = _times(ctx64, lambda: ctx64.intfactor_apply(alpha, b, c, c, f, u, ncomp=nf))
    assert together < 1.2 * apart, (together, apart)


@pytest.mark.parametrize("extent,nf", [((12, 4, 4), 3), ((2, 8, 8), 1)])
def test_chained_poisson_passes_spread_over_the_sms(ctx64, extent, nf):
    b, c = 8, li.box_blocks(*extent)
    f = torch.randn(nf * c.shape[0] * b ** 3, dtype=torch.float64, device="cuda")
    u = torch.empty_like(f)
    together, apart = _times(ctx64, lambda: ctx64.poisson_apply(b, c, c, f, u, ncomp=nf))
    assert together < 1.2 * apart, (together, apart)
