"""Surrogate inference over numbers of samples at which its launch changes."""

import pytest
import torch

pytestmark = pytest.mark.gpu

H = 64
N_PARAM = 3 * H + H + H * H + H + H + 1


def inputs(n):
    gen = torch.Generator(device="cuda").manual_seed(3)
    r = torch.rand((n, 3), generator=gen, device="cuda")
    xau = torch.stack([32.0 * r[:, 0] - 16.0, 10.0 ** (-3.0 + 2.0 * r[:, 1]), 20.0 * r[:, 2] - 10.0], 1).contiguous()
    p = 0.3 * torch.randn(N_PARAM, generator=gen, device="cuda")
    return xau, p


def test_every_sample_alone():
    """Results do not depend on how many samples there are: 128 per tile, one tile per CTA up to
    304 tiles, 2 to 8 CTAs per SM, CTAs of eight tiles from 19456 tiles on."""
    from paper_2511_08498_gb300 import api
    ctx = api.Context(0)
    sizes = [1, 127, 129, 304 * 128, 305 * 128 + 1, 874 * 128, 875 * 128, 1224 * 128 + 5, 2430 * 128, 2797 * 128 - 1,
             19455 * 128, 19456 * 128, 19456 * 128 + 77]
    xau, p = inputs(max(sizes))
    ref = torch.cat([api.mlp_forward(ctx, xau[q:q + 30000].contiguous(), p) for q in range(0, max(sizes), 30000)])
    for n in sizes:
        assert torch.equal(api.mlp_forward(ctx, xau[:n].contiguous(), p), ref[:n]), n
    ctx.check()


# one tile per CTA cost 33 to 39 us here, two per CTA 29 us for 330000
@pytest.mark.parametrize("n", [260000, 290000, 310000])
def test_fewer_samples_cost_no_more(n):
    from paper_2511_08498_gb300 import api
    ctx = api.Context(0)
    xau, p = inputs(330000)
    out = torch.empty(330000, device="cuda")
    times = {}
    # in turn, twenty launches between events (their resolution is a microsecond), all queued
    # before the first starts
    for _ in range(20):
        for m in (n, 330000):
            x = xau[:m].contiguous()
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            torch.cuda._sleep(2000000)
            a.record()
            for _ in range(20):
                api.mlp_forward(ctx, x, p, out=out[:m])
            b.record()
            b.synchronize()
            times[m] = min(times.get(m, float("inf")), a.elapsed_time(b))
    ctx.check()
    assert times[n] < 1.03 * times[330000], times
