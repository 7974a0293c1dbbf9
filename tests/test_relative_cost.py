"""Costs of one call beside another's: what a path adds where it has little to do."""

import pytest
import torch

pytestmark = pytest.mark.gpu


def best_ms(f):
    best = float("inf")
    for _ in range(12):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        torch.cuda._sleep(200000)  # the launches are queued before the first starts
        a.record()
        f()
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b))
    return best


def test_voigt_at_large_damping():
    """The evaluation for a >= 0.25 inlined, not called: 1.8 times the time of small damping."""
    from paper_2511_08498_gb300 import api
    ctx = api.Context(0)
    gen = torch.Generator(device="cuda").manual_seed(1)
    a = torch.rand(1 << 22, generator=gen, device="cuda")
    x, out = 40.0 * torch.rand(1 << 22, generator=gen, device="cuda") - 20.0, torch.empty(1 << 22, device="cuda")
    thin, thick = 0.01 * a, 0.25 + a
    ratio = best_ms(lambda: api.voigt(ctx, thick, x, out)) / best_ms(lambda: api.voigt(ctx, thin, x, out))
    assert ratio < 1.9, ratio
