"""Costs of one call beside another's: what a path adds where it has little to do."""

import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


def best_ms(f):
    best = float("inf")
    for _ in range(40):
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


def test_counting_cascades():
    """Rays that cross nothing count nothing: a counting solve takes 2.7 times the other's time
    (it looks for no bound and follows rays to the block crossing of zero transmission)."""
    from paper_2511_08498_gb300 import api
    ctx = api.Context(0)
    n, L = 512, 16
    m = synth.sparse_line_atmosphere(n, n, n_lambda=L, seed=synth.SEED_BASE + 1030)
    t = {k: torch.as_tensor(m[k]).reshape(-1).contiguous().cuda()
         for k in ("chi_c", "s_c", "s_l", "ratio", "dld", "dlam")}
    eta, chi = api.synth_static_line(ctx, t["chi_c"], t["s_c"], t["s_l"], t["ratio"], t["dld"], t["dlam"])
    grid = api.grid_build(ctx, n, n, eta, chi)
    mips = api.mips_build(ctx, grid, eta, chi, 8, 3, 1e-2, 1e-2)
    J = torch.empty((L, n * n), device="cuda")
    ws = torch.empty(api.rc_workspace_floats(n, n, L, 8, 4), device="cuda")
    ratio = (best_ms(lambda: api.rc_solve(ctx, grid, mips, 4, J=J, workspace=ws, count_segments=True)) /
             best_ms(lambda: api.rc_solve(ctx, grid, mips, 4, J=J, workspace=ws)))
    ctx.check()
    assert ratio < 3.4, ratio
