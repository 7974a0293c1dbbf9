"""State words that do not describe an active block, and probes outside the grid: an error status, no J."""

import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

BAND = [6.0, 24.0, 96.0]


def fields(shape, L, seed):
    make = synth.random_medium if len(shape) == 2 else synth.random_medium3
    m = make(*shape, L, seed=synth.SEED_BASE + seed, log_chi_range=(-3.0, 1.0), emitter_frac=0.0)
    return [torch.from_numpy(m[k].reshape(L, -1)).cuda() for k in ("eta", "chi")]


def refused(ctx, J):
    from paper_2511_08498_gb300 import api
    with pytest.raises(api.DexError):
        ctx.check()
    assert not J.any()


# 64 x 48: split directions; 448 x 480, 16 wavelengths: one CTA per block; both walks, and
# pairs of batches with the same (missing) levels
@pytest.mark.parametrize("walk", ["per_batch", "paired"])
@pytest.mark.parametrize("nx,nz", [(64, 48), (448, 480)])
def test_static(walk, nx, nz):
    from paper_2511_08498_gb300 import api
    ctx = api.Context(0)
    ctx.set_traversal(api.TRAVERSAL_PAIRED if walk == "paired" else api.TRAVERSAL_PER_BATCH)
    L = 16
    eta, chi = fields((nx, nz), L, 740)
    grid = api.grid_build(ctx, nx, nz, eta, chi)
    mips = api.mips_build(ctx, grid, eta, chi, 8, 3, 1.0, 1.0)
    mips.words.zero_()
    dirs, w = synth.directions(4)
    J, _, _ = api.formal_solve_hdda(ctx, grid, mips, dirs, w, band=BAND)
    refused(ctx, J)
    d, wd = (torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda() for a in (dirs, w))
    item = api.batch_item(grid, mips, d, wd, J.fill_(1.0), band=BAND)
    api.batch_solve(ctx, [item], 8)
    refused(ctx, J)


@pytest.mark.parametrize("walk", ["per_batch", "paired"])
@pytest.mark.parametrize("shape", [(24, 16, 32), (64, 48, 40)])
def test_static_3d(walk, shape):
    from paper_2511_08498_gb300 import api
    ctx = api.Context(0)
    ctx.set_traversal(api.TRAVERSAL_PAIRED if walk == "paired" else api.TRAVERSAL_PER_BATCH)
    eta, chi = fields(shape, 16, 741)
    grid = api.grid3_build(ctx, *shape, eta, chi)
    mips = api.mips3_build(ctx, grid, eta, chi, 8, 3, 1.0, 1.0)
    mips.words.zero_()
    dirs, w = synth.directions3(4, 2)
    J, _, _ = api.formal_solve_hdda3(ctx, grid, mips, dirs, w, band=BAND)
    refused(ctx, J)


@pytest.mark.parametrize("kind", ["cav", "vel"])
def test_moving(kind):
    from paper_2511_08498_gb300 import api
    ctx = api.Context(0)
    nx, nz = 64, 48
    m = synth.dynamic_line_atmosphere(nx, nz, n_lambda=9, seed=synth.SEED_BASE + 742, empty_frac=0.2)
    f = {k: torch.from_numpy(np.ascontiguousarray(m[k]).reshape(-1)).cuda() for k in api.CAV_FIELDS}
    grid = api.cav_grid_build(ctx, nx, nz, f)
    build, solve = ((api.cav_mips_build, api.formal_solve_cav) if kind == "cav"
                    else (api.vel_mips_build, api.formal_solve_velinterp))
    mips = build(ctx, grid, f, m["dv"], m["c_kms"], 8, 3, 1.0, 1.0)
    mips.words.zero_()
    J, _, _ = solve(ctx, grid, mips, *synth.directions(4), band=BAND)
    refused(ctx, J)


def test_probe_outside_the_grid():
    from paper_2511_08498_gb300 import api
    ctx = api.Context(0)
    nx, nz, L = 512, 512, 9
    planes = api.pack_planes(ctx, *fields((nx, nz), L, 743), 8)
    probes = torch.arange(nx * nz, dtype=torch.int32, device="cuda")
    bad = torch.tensor([0, 300, 1000, nx * nz - 1], device="cuda")
    probes[bad] = torch.tensor([-1, nx * nz, 2 ** 31 - 1, -2 ** 31], dtype=torch.int32, device="cuda")
    J = torch.zeros((L, nx * nz), device="cuda")
    api.formal_solve_dense(ctx, nx, nz, L, 8, planes, *synth.directions(4), probes=probes, J=J)
    refused(ctx, J[:, bad])
    good = torch.ones(nx * nz, dtype=torch.bool, device="cuda")
    good[bad] = False
    ref, _, _ = api.formal_solve_dense(ctx, nx, nz, L, 8, planes, *synth.directions(4))
    assert torch.equal(J[:, good], ref[:, good])
