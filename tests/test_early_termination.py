"""Exact early termination and split directions: the bits of the full walk.

A counting solve walks every ray until its transmissions are exactly zero (the
plain solver: to the grid's edge) and one warp takes all directions of a probe.
The solves that users time stop rays as soon as the rest cannot change a bit of
I, and share a probe's directions between warps on small grids.  Both must give
the same J and I, bit for bit, so every comparison here is for equality.
"""

import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

BAND = [6.0, 24.0, 96.0]


def ctx_():
    from paper_2511_08498_gb300 import api
    return api.Context(0)


def thick_medium(nx, nz, L, seed, emitters=False, log_chi=(-3.0, 2.5)):
    """Random medium whose rays die after 1 to 100 cells, with empty cells (and blocks)."""
    m = synth.random_medium(nx, nz, L, seed=synth.SEED_BASE + seed, log_chi_range=log_chi,
                            emitter_frac=0.02 if emitters else 0.0)
    e, c = m["eta"].copy(), m["chi"].copy()
    e[:, -(nz // 4):], c[:, -(nz // 4):] = 0.0, 0.0
    return torch.from_numpy(e.reshape(L, -1)).cuda(), torch.from_numpy(c.reshape(L, -1)).cuda()


def same(a, b):
    assert (a is None) == (b is None)
    assert a is None or torch.equal(a, b)


@pytest.mark.parametrize("nx,nz,L,W", [(33, 17, 1, 1), (64, 64, 3, 2), (31, 70, 9, 4), (97, 65, 20, 8)])
@pytest.mark.parametrize("i_bc,emitters", [(0.0, False), (0.7, True)])
def test_plain(nx, nz, L, W, i_bc, emitters):
    from paper_2511_08498_gb300 import api
    ctx = ctx_()
    eta, chi = thick_medium(nx, nz, L, 800 + W, emitters)
    planes = api.pack_planes(ctx, eta, chi, W)
    dirs, w = synth.directions(12, offset=0.0)  # axis-parallel and corner rays among them
    for own in (True, False):
        ctx.set_own_cell(own)
        full = api.formal_solve_dense(ctx, nx, nz, L, W, planes, dirs, w, i_bc=i_bc, want_intensity=True,
                                      count_segments=True)
        fast = api.formal_solve_dense(ctx, nx, nz, L, W, planes, dirs, w, i_bc=i_bc, want_intensity=True)
        same(full[0], fast[0])
        same(full[1], fast[1])
    ctx.set_own_cell(True)
    # enough probes for one warp per 32 of them and all directions (unsplit)
    probes = torch.arange(nx * nz, dtype=torch.int32, device="cuda").repeat(-(-312000 // (nx * nz)))
    J, _, _ = api.formal_solve_dense(ctx, nx, nz, L, W, planes, dirs, w, probes=probes, i_bc=i_bc)
    ref, _, _ = api.formal_solve_dense(ctx, nx, nz, L, W, planes, dirs, w, i_bc=i_bc)
    same(J, ref[:, probes.long()])
    ctx.check()


@pytest.mark.parametrize("bad", [float("inf"), float("nan"), -1.0])
def test_plain_records_without_a_bound(bad):
    """Hand-made records with a non-finite source function or a negative opacity: no early end.
    Opacities near 1 per cell keep every transmission above zero, as in the counting walk."""
    from paper_2511_08498_gb300 import api
    ctx = ctx_()
    nx, nz, L, W = 40, 24, 8, 8
    eta, chi = thick_medium(nx, nz, L, 811, log_chi=(-0.2, 0.1))
    planes = api.pack_planes(ctx, eta, chi, W)
    planes[0, 500, 3 if bad != -1.0 else 8 + 3] = bad * (1e-3 if bad == -1.0 else 1.0)
    dirs, w = synth.directions(8)
    full = api.formal_solve_dense(ctx, nx, nz, L, W, planes, dirs, w, want_intensity=True, count_segments=True)
    fast = api.formal_solve_dense(ctx, nx, nz, L, W, planes, dirs, w, want_intensity=True)
    for a, b in zip(full[:2], fast[:2]):
        assert np.array_equal(a.cpu().numpy(), b.cpu().numpy(), equal_nan=True)


@pytest.mark.parametrize("walk", ["per_batch", "paired"])
@pytest.mark.parametrize("nx,nz,L,W,storage", [(64, 48, 20, 8, 0), (64, 48, 24, 8, 1), (48, 64, 17, 8, 2),
                                               (48, 48, 6, 4, 0), (512, 512, 24, 8, 0), (32, 32, 3, 1, 0)])
def test_sparse(walk, nx, nz, L, W, storage):
    from paper_2511_08498_gb300 import api
    if walk == "paired" and W != 8:
        pytest.skip("the paired walk needs W = 8")
    ctx = ctx_()
    eta, chi = thick_medium(nx, nz, L, 820 + L, emitters=storage == 0)
    grid = api.grid_build(ctx, nx, nz, eta, chi)
    dirs, w = synth.directions(10, offset=0.0)
    ctx.set_traversal(api.TRAVERSAL_PAIRED if walk == "paired" else api.TRAVERSAL_PER_BATCH)
    for iod, band, i_bc in ((1e-2, BAND, 0.0), (1e30, None, 0.4)):
        mips = api.mips_build(ctx, grid, eta, chi, W, 3, iod, iod, storage=storage)
        for own in (True, False):
            if not own and (W != 8 or storage != 0):
                continue
            ctx.set_own_cell(own)
            full = api.formal_solve_hdda(ctx, grid, mips, dirs, w, band=band, i_bc=i_bc, want_intensity=True,
                                         count_segments=True)
            fast = api.formal_solve_hdda(ctx, grid, mips, dirs, w, band=band, i_bc=i_bc, want_intensity=True)
            same(full[0], fast[0])
            same(full[1], fast[1])
        ctx.set_own_cell(True)
    ctx.check()


@pytest.mark.parametrize("walk", ["per_batch", "paired"])
@pytest.mark.parametrize("L,W,storage,n_cascades,i_bc", [(20, 8, 0, 4, 0.0), (16, 8, 1, 3, 0.6), (5, 2, 0, 4, 0.3)])
def test_cascades(walk, L, W, storage, n_cascades, i_bc):
    from paper_2511_08498_gb300 import api
    ctx = ctx_()
    nx, nz = 96, 64
    eta, chi = thick_medium(nx, nz, L, 840 + L)
    eta.view(L, nz, nx)[:, :16, :16] = 0.0  # cell 0 in an empty block
    chi.view(L, nz, nx)[:, :16, :16] = 0.0
    grid = api.grid_build(ctx, nx, nz, eta, chi)
    ctx.set_traversal(api.TRAVERSAL_PAIRED if walk == "paired" else api.TRAVERSAL_PER_BATCH)
    mips = api.mips_build(ctx, grid, eta, chi, W, 3, 1.0, 1.0, storage=storage)
    full, _ = api.rc_solve(ctx, grid, mips, n_cascades, 4, 1.5, i_bc=i_bc, count_segments=True)
    fast, _ = api.rc_solve(ctx, grid, mips, n_cascades, 4, 1.5, i_bc=i_bc)
    same(full, fast)
    assert not fast[:, 0].any()
    ctx.check()


@pytest.mark.parametrize("walk", ["per_batch", "paired"])
@pytest.mark.parametrize("L,W,storage", [(20, 8, 0), (24, 8, 1), (9, 8, 2), (3, 1, 0), (6, 4, 0)])
def test_sparse_3d(walk, L, W, storage):
    from paper_2511_08498_gb300 import api
    if walk == "paired" and W != 8:
        pytest.skip("the paired walk needs W = 8")
    ctx = ctx_()
    nx, ny, nz = 32, 24, 40
    m = synth.random_medium3(nx, ny, nz, L, seed=synth.SEED_BASE + 850 + L, log_chi_range=(-2.5, 2.5),
                             emitter_frac=0.02 if storage == 0 else 0.0)
    m["eta"][:, 32:], m["chi"][:, 32:] = 0.0, 0.0
    eta, chi = (torch.from_numpy(m[k].reshape(L, -1)).cuda() for k in ("eta", "chi"))
    grid = api.grid3_build(ctx, nx, ny, nz, eta, chi)
    dirs, w = synth.directions3(6, 2)
    ctx.set_traversal(api.TRAVERSAL_PAIRED if walk == "paired" else api.TRAVERSAL_PER_BATCH)
    for iod, band, i_bc in ((1e-2, BAND, 0.0), (1e30, None, 0.4)):
        mips = api.mips3_build(ctx, grid, eta, chi, W, 3, iod, iod, storage=storage)
        full = api.formal_solve_hdda3(ctx, grid, mips, dirs, w, band=band, i_bc=i_bc, want_intensity=True,
                                      count_segments=True)
        fast = api.formal_solve_hdda3(ctx, grid, mips, dirs, w, band=band, i_bc=i_bc, want_intensity=True)
        same(full[0], fast[0])
        same(full[1], fast[1])
    ctx.check()


@pytest.mark.parametrize("kind", ["cav", "vel"])
@pytest.mark.parametrize("L,W,i_bc", [(12, 8, 0.0), (16, 8, 0.8), (5, 2, 0.0), (9, 4, 0.2)])
def test_moving(kind, L, W, i_bc):
    from paper_2511_08498_gb300 import api
    ctx = ctx_()
    nx, nz = 96, 128
    m = synth.dynamic_line_atmosphere(nx, nz, n_lambda=L, seed=synth.SEED_BASE + 860 + L, empty_frac=0.2)
    f = {k: torch.from_numpy(np.ascontiguousarray(m[k]).reshape(-1)).cuda() for k in api.CAV_FIELDS}
    for k in ("chi_c", "eta_c"):  # a continuum that ends rays within the grid
        f[k] *= 200.0
    grid = api.cav_grid_build(ctx, nx, nz, f)
    build, solve = ((api.cav_mips_build, api.formal_solve_cav) if kind == "cav"
                    else (api.vel_mips_build, api.formal_solve_velinterp))
    mips = build(ctx, grid, f, m["dv"], m["c_kms"], W, 3, 1.0, 1.0)
    dirs, w = synth.directions(8)
    full = solve(ctx, grid, mips, dirs, w, band=BAND, i_bc=i_bc, want_intensity=True, count_segments=True)
    fast = solve(ctx, grid, mips, dirs, w, band=BAND, i_bc=i_bc, want_intensity=True)
    same(full[0], fast[0])
    same(full[1], fast[1])
    ctx.check()
