"""Velocity grids: samples whose opacities are so far apart that interpolation leaves their range.

At the end of the stored velocities the interpolation weight can come out as 1 + 2^-20.  Beside
an opacity 2^20 times as large the interpolated one then nearly vanishes while the emissivity does
not, so the source function is far above both samples': rays must not end early on their bound.
"""

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


# the first makes 1024 - 2^-20 (2^30 - 1088) = 0.001 of an opacity of 1024
@pytest.mark.parametrize("other", [2.0 ** 30 - 64.0, 2.0 ** 27, 2.0 ** 24])
def test_opacities_apart(other):
    from paper_2511_08498_gb300 import api
    ctx = api.Context(0)
    nx, nz, L = 16, 64, 8
    value = dict(eta_star=0.0, chi_star=0.0, damping=0.01, vth=5.0, vx=0.0, vz=0.0, eta_c=2.0, chi_c=2.0)
    f = {k: torch.full((nx * nz,), v, device="cuda") for k, v in value.items()}
    grid = api.cav_grid_build(ctx, nx, nz, f)
    mips = api.vel_mips_build(ctx, grid, f, np.linspace(-20.0, 20.0, L), 299792.458, 8, 0, 1.0, 1.0)
    # the lowest block stays (S = 1, 2 per cell); above it the last sample has S = 1 and opacity
    # 1024, the others S = 0; speeds lie beyond the last sample, whose velocity is one of those
    # for which the weight comes out above 1
    v = mips.bricks.view(4, 256, 132)[1:]
    V = np.array(0x3fb03d61, dtype=np.uint32).view(np.float32).item()
    v[..., 0], v[..., 1], v[..., 2] = 0.0, -2.0 * V, V
    s = v[..., 4:].view(3, 256, 8, 2, 8)
    s[..., 0, :], s[..., 1, :] = 0.0, other
    s[..., 7, 0, :], s[..., 7, 1, :] = 1024.0, 1024.0
    args = (ctx, grid, mips, np.array([[0.0, 1.0]], np.float32), np.ones(1, np.float32))
    full = api.formal_solve_velinterp(*args, count_segments=True)[0]
    fast = api.formal_solve_velinterp(*args)[0]
    ctx.check()
    assert torch.equal(full, fast)
