"""Plain solves by number of directions: how the work is split changes no bit, and fewer cost less."""

import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


def medium(nx, nz, L, seed, log_chi):
    m = synth.random_medium(nx, nz, L, seed=synth.SEED_BASE + seed, log_chi_range=log_chi, emitter_frac=0.0)
    return [torch.from_numpy(m[k].reshape(L, -1)).cuda() for k in ("eta", "chi")]


# 48 x 40: split, unsplit through a long probe list; 200 x 208, 24 wavelengths: at W = 8
# few directions go to the kernel that stages records
@pytest.mark.parametrize("n_dir", [1, 3, 7, 9, 17])
@pytest.mark.parametrize("nx,nz,L,W", [(48, 40, 3, 1), (48, 40, 3, 2), (48, 40, 7, 4), (48, 40, 13, 8), (200, 208, 24, 8)])
def test_bits(nx, nz, L, W, n_dir):
    from paper_2511_08498_gb300 import api
    ctx = api.Context(0)
    eta, chi = medium(nx, nz, L, 700 + W, (-3.0, 1.0))
    planes = api.pack_planes(ctx, eta, chi, W)
    dirs, w = synth.directions(n_dir, offset=0.0)
    full = api.formal_solve_dense(ctx, nx, nz, L, W, planes, dirs, w, i_bc=0.4, want_intensity=True,
                                  count_segments=True)
    J, I, _ = api.formal_solve_dense(ctx, nx, nz, L, W, planes, dirs, w, i_bc=0.4, want_intensity=True)
    assert torch.equal(J, full[0]) and torch.equal(I, full[1])
    probes = torch.arange(nx * nz, dtype=torch.int32, device="cuda").repeat(-(-312000 // (nx * nz)))
    Jp, _, _ = api.formal_solve_dense(ctx, nx, nz, L, W, planes, dirs, w, probes=probes, i_bc=0.4)
    assert torch.equal(Jp, J[:, probes.long()])
    ctx.check()


@pytest.mark.parametrize("nx,nz,L", [(352, 352, 16), (200, 208, 24)])
def test_half_the_directions_cost_less(nx, nz, L):
    from paper_2511_08498_gb300 import api
    ctx = api.Context(0)
    planes = api.pack_planes(ctx, *medium(nx, nz, L, 720, (-5.0, -3.0)), 8)
    J = torch.empty((L, nx * nz), device="cuda")
    times = []
    for n_dir in (4, 8):
        dirs, w = synth.directions(n_dir)
        best = float("inf")
        for _ in range(20):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            api.formal_solve_dense(ctx, nx, nz, L, 8, planes, dirs, w, J=J)
            b.record()
            b.synchronize()
            best = min(best, a.elapsed_time(b))
        times.append(best)
    ctx.check()
    assert times[0] < 0.8 * times[1], times
