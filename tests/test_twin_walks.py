"""Solves that walk once per wavelength batch, where two batches' blocks have the same levels.

Such pairs of batches share a walk; it is each batch's own, so J and I keep every
bit.  A counting solve always walks batch by batch, so every comparison here is
for equality with it.
"""

import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

BAND = [6.0, 24.0, 96.0]


def ctx_():
    from paper_2511_08498_gb300 import api
    ctx = api.Context(0)
    ctx.set_traversal(api.TRAVERSAL_PER_BATCH)
    return ctx


def medium(nx, nz, L, seed, mirrored, log_chi=(-3.0, 2.0), ny=None):
    """Random medium with an empty corner; ``mirrored``: wavelengths l and L - 1 - l alike."""
    make = synth.random_medium if ny is None else synth.random_medium3
    m = make(*((nx, nz) if ny is None else (nx, ny, nz)), L, seed=synth.SEED_BASE + seed, log_chi_range=log_chi,
             emitter_frac=0.0)
    out = []
    for k in ("eta", "chi"):
        a = np.ascontiguousarray(m[k], dtype=np.float32).copy()
        if mirrored:
            a[L - L // 2:] = a[:L // 2][::-1]
        out.append(torch.from_numpy(a.reshape(L, -1)).cuda())
    for a in out:
        v = a.view(L, nz, -1)
        v[:, :16] = 0.0
    return out


def equal(a, b):
    assert np.array_equal(a.cpu().numpy(), b.cpu().numpy(), equal_nan=True)


def both(solve, *args, **kw):
    full = solve(*args, want_intensity=True, count_segments=True, **kw)
    fast = solve(*args, want_intensity=True, **kw)
    equal(full[0], fast[0])
    equal(full[1], fast[1])
    return fast[0]


# split and unsplit (1216 block-batches), even and odd numbers of batches (a lone middle
# batch), a ragged last batch, levels that agree and levels that do not
@pytest.mark.parametrize("storage", [0, 1, 2])
@pytest.mark.parametrize("nx,nz,L", [(96, 80, 16), (96, 80, 24), (96, 80, 20), (320, 336, 32), (448, 464, 24),
                                     (640, 336, 16), (448, 464, 40)])
def test_sparse(nx, nz, L, storage):
    from paper_2511_08498_gb300 import api
    ctx = ctx_()
    dirs, w = synth.directions(6, offset=0.0)
    for mirrored, iod, band, i_bc in ((True, 1e-2, BAND, 0.0), (False, 0.3, BAND, 0.2), (False, 1e30, None, 0.4)):
        eta, chi = medium(nx, nz, L, 900 + L, mirrored)
        grid = api.grid_build(ctx, nx, nz, eta, chi)
        mips = api.mips_build(ctx, grid, eta, chi, 8, 3, iod, iod, storage=storage)
        both(api.formal_solve_hdda, ctx, grid, mips, dirs, w, band=band, i_bc=i_bc)
    ctx.check()


@pytest.mark.parametrize("nx,nz", [(64, 64), (320, 320)])
@pytest.mark.parametrize("batch", [0, 1])
def test_records_without_a_bound(nx, nz, batch):
    """One batch holds a source function that overflowed: its partner keeps its values.
    Opacities are low enough that no ray's transmission reaches zero."""
    from paper_2511_08498_gb300 import api
    ctx = ctx_()
    L = 32
    eta, chi = medium(nx, nz, L, 950, True, log_chi=(-3.0, -2.0))
    grid = api.grid_build(ctx, nx, nz, eta, chi)
    mips = api.mips_build(ctx, grid, eta, chi, 8, 3, 1e-2, 1e-2)
    flat = mips.bricks.view(4, -1)
    flat[batch, 0] = float("inf")
    dirs, w = synth.directions(8)
    J = both(api.formal_solve_hdda, ctx, grid, mips, dirs, w, band=BAND)
    assert not torch.isfinite(J[8 * batch]).all() and torch.isfinite(J[8 * (3 - batch):8 * (4 - batch)]).all()
    ctx.check()


@pytest.mark.parametrize("nx,ny,nz,L,storage", [(64, 48, 40, 16, 0), (40, 48, 64, 32, 1), (64, 48, 40, 20, 2),
                                                (64, 64, 72, 24, 0)])
def test_3d(nx, ny, nz, L, storage):
    from paper_2511_08498_gb300 import api
    ctx = ctx_()
    dirs, w = synth.directions3(4, 2)
    for mirrored, iod, band, i_bc, bad in ((True, 1e-2, BAND, 0.0, False), (False, 0.3, BAND, 0.2, False),
                                           (False, 1e30, None, 0.4, False), (True, 1e-2, BAND, 0.3, storage == 0)):
        eta, chi = medium(nx, nz, L, 930 + L, mirrored, log_chi=(-3.0, -2.0) if bad else (-3.0, 2.0), ny=ny)
        grid = api.grid3_build(ctx, nx, ny, nz, eta, chi)
        mips = api.mips3_build(ctx, grid, eta, chi, 8, 3, iod, iod, storage=storage)
        if bad:
            mips.bricks.view((L + 7) // 8, -1)[0, 0] = float("inf")
        both(api.formal_solve_hdda3, ctx, grid, mips, dirs, w, band=band, i_bc=i_bc)
    ctx.check()


# enough blocks of pairs (3040) for the persistent launch to look for them: packets,
# packed states and one word per block, queue chunks; an atmosphere of one batch among them
@pytest.mark.parametrize("cfg", [None, dict(packet=64, staging=1, chunk=3), dict(packet=128, staging=0, occupancy=1)])
@pytest.mark.parametrize("bad", [False, True])
def test_batched(cfg, bad):
    from paper_2511_08498_gb300 import api
    ctx = ctx_()
    items, want, keep = [], [], []
    dirs, w = synth.directions(4)
    d, wd = (torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda() for a in (dirs, w))
    for q, (nx, nz, L, mirrored) in enumerate(((512, 512, 32, True), (448, 512, 24, True), (512, 256, 24, False),
                                               (128, 96, 8, False), (336, 320, 16, True))):
        eta, chi = medium(nx, nz, L, 970 + q, mirrored, log_chi=(-3.0, -2.0) if bad else (-3.0, 2.0))
        grid = api.grid_build(ctx, nx, nz, eta, chi)
        mips = api.mips_build(ctx, grid, eta, chi, 8, 3, 1e-2, 1e-2)
        if bad and L > 8:
            mips.bricks.view((L + 7) // 8, -1)[q % 2, 0] = float("inf")
        # alone, an atmosphere has too few blocks of pairs: it is walked batch by batch
        J = torch.empty((L, nx * nz), device="cuda")
        items.append(api.batch_item(grid, mips, d, wd, J, band=BAND, i_bc=0.3))
        api.batch_solve(ctx, items[-1:], 8)
        want.append(J.clone())
        if not bad:
            equal(J, api.formal_solve_hdda(ctx, grid, mips, dirs, w, band=BAND, i_bc=0.3, count_segments=True)[0])
        keep.append((grid, mips, J))
    for _ in range(2):
        if cfg is None:
            api.batch_solve(ctx, items, 8)
        else:
            api.batch_solve_config(ctx, items, 8, **cfg)
        for ref, (_, _, J) in zip(want, keep):
            equal(ref, J)
    ctx.check()
