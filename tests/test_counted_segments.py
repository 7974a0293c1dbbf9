"""Segments that counting solves report: a ray is counted to the block crossing at which
all of its transmissions have become exactly zero.

In a medium so thick that they are zero after the first segment the counts along the
axes follow from the block edges alone.
"""

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

AXES = np.array([[1, 0], [-1, 0], [0, 1], [0, -1]], dtype=np.float32)


def along(n, block, before):
    """Segments of the rays from every cell of a row of n cells in the positive direction.

    ``before``: the walk looks for zero transmission before it integrates the last voxel of a
    block (where it looks up the next block first), otherwise after."""
    total = 0
    for i in range(n):
        zero = False  # all transmissions are zero
        for c in range(i, n):
            edge = (c + 1) % block == 0 and c + 1 < n
            if edge and before and zero:
                break
            total += 1
            zero = True
            if edge and not before:
                break
    return total


def uniform(n_lambda, n, value):
    return torch.full((n_lambda, n), value, device="cuda")


@pytest.mark.parametrize("walk,storage", [("per_batch", 0), ("per_batch", 1), ("paired", 0), ("paired", 2)])
def test_static(walk, storage):
    from paper_2511_08498_gb300 import api
    ctx = api.Context(0)
    ctx.set_traversal(api.TRAVERSAL_PAIRED if walk == "paired" else api.TRAVERSAL_PER_BATCH)
    nx, nz, L = 64, 48, 16
    eta, chi = uniform(L, nx * nz, 500.0), uniform(L, nx * nz, 1000.0)
    grid = api.grid_build(ctx, nx, nz, eta, chi)
    mips = api.mips_build(ctx, grid, eta, chi, 8, 0, 1.0, 1.0, storage=storage)
    _, _, seg = api.formal_solve_hdda(ctx, grid, mips, AXES, np.full(4, 0.25, np.float32), count_segments=True)
    ctx.check()
    before = walk == "paired"
    assert seg.item() == 2 * 2 * (nz * along(nx, 16, before) + nx * along(nz, 16, before))


@pytest.mark.parametrize("walk", ["per_batch", "paired"])
def test_static_3d(walk):
    from paper_2511_08498_gb300 import api
    ctx = api.Context(0)
    ctx.set_traversal(api.TRAVERSAL_PAIRED if walk == "paired" else api.TRAVERSAL_PER_BATCH)
    n, L = (24, 16, 32), 16
    cells = n[0] * n[1] * n[2]
    eta, chi = uniform(L, cells, 500.0), uniform(L, cells, 1000.0)
    grid = api.grid3_build(ctx, *n, eta, chi)
    mips = api.mips3_build(ctx, grid, eta, chi, 8, 0, 1.0, 1.0)
    dirs = np.concatenate([np.eye(3), -np.eye(3)]).astype(np.float32)
    _, _, seg = api.formal_solve_hdda3(ctx, grid, mips, dirs, np.full(6, 1 / 6, np.float32), count_segments=True)
    ctx.check()
    assert seg.item() == 2 * 2 * sum(cells // m * along(m, 8, False) for m in n)


@pytest.mark.parametrize("kind", ["cav", "vel"])
def test_moving(kind):
    from paper_2511_08498_gb300 import api
    ctx = api.Context(0)
    nx, nz, L = 64, 48, 12
    value = dict(eta_star=0.0, chi_star=0.0, damping=0.01, vth=5.0, vx=0.0, vz=0.0, eta_c=500.0, chi_c=1000.0)
    f = {k: torch.full((nx * nz,), v, device="cuda") for k, v in value.items()}
    grid = api.cav_grid_build(ctx, nx, nz, f)
    build, solve = ((api.cav_mips_build, api.formal_solve_cav) if kind == "cav"
                    else (api.vel_mips_build, api.formal_solve_velinterp))
    mips = build(ctx, grid, f, np.linspace(-20.0, 20.0, L), 299792.458, 8, 0, 1.0, 1.0)
    _, _, seg = solve(ctx, grid, mips, AXES, np.full(4, 0.25, np.float32), count_segments=True)
    ctx.check()
    assert seg.item() == 2 * 2 * (nz * along(nx, 16, True) + nx * along(nz, 16, True))


@pytest.mark.parametrize("walk", ["per_batch", "paired"])
def test_cascades(walk):
    """Rays of the upper cascades cross blocks; those of the lower ones end within theirs."""
    from paper_2511_08498_gb300 import api
    ctx = api.Context(0)
    ctx.set_traversal(api.TRAVERSAL_PAIRED if walk == "paired" else api.TRAVERSAL_PER_BATCH)
    nx, nz, L = 64, 64, 16
    eta, chi = uniform(L, nx * nz, 500.0), uniform(L, nx * nz, 1000.0)
    grid = api.grid_build(ctx, nx, nz, eta, chi)
    mips = api.mips_build(ctx, grid, eta, chi, 8, 0, 1.0, 1.0)
    _, seg = api.rc_solve(ctx, grid, mips, 4, 4, 1.5, count_segments=True)
    ctx.check()
    assert seg.item() == 723680  # counted by the walk that knew no other end than this
