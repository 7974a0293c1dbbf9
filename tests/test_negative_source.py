"""Records with a negative source function: rays end where their transmissions are zero."""

import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

N, L = 1024, 8


def best_ms(f):
    best = float("inf")
    for _ in range(4):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        a.record()
        f()
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b))
    return best


def plain(api, ctx, S, chi):
    planes = torch.full((1, N * N, 16), S, device="cuda")
    planes[..., 8:] = chi
    return lambda **kw: api.formal_solve_dense(ctx, N, N, L, 8, planes, *synth.directions(6), **kw)


def sparse(api, ctx, S, chi):
    eta = torch.full((L, N * N), 7.0 * chi, device="cuda")  # S = 7 until the records are changed
    chi = torch.full((L, N * N), chi, device="cuda")
    grid = api.grid_build(ctx, N, N, eta, chi)
    mips = api.mips_build(ctx, grid, eta, chi, 8, 0, 1.0, 1.0)
    mips.bricks[mips.bricks > 6.0] = S
    return lambda **kw: api.formal_solve_hdda(ctx, grid, mips, *synth.directions(6), **kw)


@pytest.mark.parametrize("make", [plain, sparse])
def test_thick(make):
    from paper_2511_08498_gb300 import api
    ctx = api.Context(0)
    thick, thin = make(api, ctx, -2.0, 1.0), make(api, ctx, 2.0, 1e-7)
    assert torch.equal(thick()[0], thick(count_segments=True)[0])
    # transmissions are zero after 104 cells of 400 and more on average
    assert best_ms(thick) < 0.6 * best_ms(thin)
    ctx.check()
