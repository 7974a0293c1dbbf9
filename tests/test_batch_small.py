"""Batched solves of a few small atmospheres (packets of 128 probes) and of more: one by one the same bits."""

import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

BAND = [6.0, 24.0, 96.0]


def batch(api, ctx, W, n_dir, sizes):
    dirs, w = synth.directions(n_dir)
    d, wd = (torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda() for a in (dirs, w))
    items, keep = [], []
    for q, (nx, nz, L) in enumerate(sizes):
        m = synth.sparse_line_atmosphere(nx, nz, n_lambda=L, seed=synth.SEED_BASE + 990 + q)
        t = {k: torch.from_numpy(np.ascontiguousarray(m[k]).reshape(-1)).cuda()
             for k in ("chi_c", "s_c", "s_l", "ratio", "dld", "dlam")}
        eta, chi = api.synth_static_line(ctx, t["chi_c"], t["s_c"], t["s_l"], t["ratio"], t["dld"], t["dlam"])
        grid = api.grid_build(ctx, nx, nz, eta, chi)
        mips = api.mips_build(ctx, grid, eta, chi, W, 3, 1e-2, 1e-2)
        J = torch.empty((L, nx * nz), device="cuda")
        items.append(api.batch_item(grid, mips, d, wd, J, band=BAND, i_bc=0.2))
        keep.append((grid, mips, J, dirs, w, d, wd))  # items hold addresses only
    return items, keep


# below and above two packets for each of the 456 default CTAs
@pytest.mark.parametrize("walk", ["per_batch", "paired"])
@pytest.mark.parametrize("W,sizes", [(8, ((128, 128, 32), (192, 128, 24), (128, 192, 17))), (8, ((384, 320, 32), (128, 64, 9))),
                                     (4, ((64, 96, 7), (128, 48, 12)))])
def test_same_as_one_by_one(walk, W, sizes):
    from paper_2511_08498_gb300 import api
    if walk == "paired" and W != 8:
        pytest.skip("the paired walk needs W = 8")
    ctx = api.Context(0)
    ctx.set_traversal(api.TRAVERSAL_PAIRED if walk == "paired" else api.TRAVERSAL_PER_BATCH)
    items, keep = batch(api, ctx, W, 8, sizes)
    for noalloc in (False, True):
        for k in keep:
            k[2].fill_(-1.0)
        if noalloc:
            api.batch_solve_noalloc(ctx, items, W)
        else:
            api.batch_solve(ctx, items, W)
        for grid, mips, J, dirs, w, _, _ in keep:
            ref, _, _ = api.formal_solve_hdda(ctx, grid, mips, dirs, w, band=BAND, i_bc=0.2)
            assert torch.equal(J, ref)
    ctx.check()
