"""Plain solves with a bound for the early termination, in every kernel: the bits of the full walk.

Counting solves walk every cell and know no bound.  The others look for one from 2^27 crossed
records on, so the grids here have 300 cells a side and more.
"""

import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


def planes_of(api, ctx, nx, nz, L, W, seed, log_chi):
    m = synth.random_medium(nx, nz, L, seed=synth.SEED_BASE + seed, log_chi_range=log_chi, emitter_frac=0.0)
    m["eta"][:, -(nz // 5):], m["chi"][:, -(nz // 5):] = 0.0, 0.0
    return api.pack_planes(ctx, *(torch.from_numpy(m[k].reshape(L, -1)).cuda() for k in ("eta", "chi")), W)


def equal(a, b):
    assert np.array_equal(a.cpu().numpy(), b.cpu().numpy(), equal_nan=True)


# whole grids of eight-wavelength batches that fill the chip (records staged in tiles of 32 x 12
# probes): neither side a multiple of the tile's, a ragged last batch, rays along the axes and
# the diagonals, thin media that rays cross and thick ones in which they end
@pytest.mark.parametrize("nx,nz,L", [(601, 437, 20), (333, 1000, 9)])
@pytest.mark.parametrize("log_chi,i_bc", [((-4.0, -1.5), 0.3), ((-3.0, 1.5), 0.0)])
def test_staged(nx, nz, L, log_chi, i_bc):
    from paper_2511_08498_gb300 import api
    ctx = api.Context(0)
    planes = planes_of(api, ctx, nx, nz, L, 8, 760, log_chi)
    dirs, w = synth.directions(16, offset=0.0)
    for own in (True, False):
        ctx.set_own_cell(own)
        full = api.formal_solve_dense(ctx, nx, nz, L, 8, planes, dirs, w, i_bc=i_bc, want_intensity=True,
                                      count_segments=True)
        fast = api.formal_solve_dense(ctx, nx, nz, L, 8, planes, dirs, w, i_bc=i_bc, want_intensity=True)
        assert torch.equal(full[0], fast[0]) and torch.equal(full[1], fast[1])
    ctx.set_own_cell(True)
    ctx.check()


@pytest.mark.parametrize("W,L", [(1, 2), (2, 3), (4, 7), (8, 9)])
@pytest.mark.parametrize("i_bc", [0.0, 0.6])
def test_split_and_listed(W, L, i_bc):
    from paper_2511_08498_gb300 import api
    ctx = api.Context(0)
    nx, nz = 300, 310
    planes = planes_of(api, ctx, nx, nz, L, W, 770 + W, (-3.0, 1.0))
    dirs, w = synth.directions(16, offset=0.0)
    probes = torch.arange(nx * nz, dtype=torch.int32, device="cuda").flip(0).repeat(4)  # unsplit
    for own in (True, False):
        ctx.set_own_cell(own)
        full = api.formal_solve_dense(ctx, nx, nz, L, W, planes, dirs, w, i_bc=i_bc, want_intensity=True,
                                      count_segments=True)
        fast = api.formal_solve_dense(ctx, nx, nz, L, W, planes, dirs, w, i_bc=i_bc, want_intensity=True)
        assert torch.equal(full[0], fast[0]) and torch.equal(full[1], fast[1])
        J, I, _ = api.formal_solve_dense(ctx, nx, nz, L, W, planes, dirs, w, probes=probes, i_bc=i_bc,
                                         want_intensity=True)
        assert torch.equal(J, full[0][:, probes.long()]) and torch.equal(I, full[1][:, :, probes.long()])
    ctx.set_own_cell(True)
    ctx.check()


# one record without a bound; transmissions stay above zero, as in the counting walk
@pytest.mark.parametrize("bad", ["inf", "nan", "negative S", "negative chi"])
@pytest.mark.parametrize("nx,nz,L,W,copies", [(300, 310, 3, 2, 0), (300, 310, 9, 8, 0), (300, 310, 9, 8, 4), (601, 437, 20, 8, 0)])
def test_records_without_a_bound(bad, nx, nz, L, W, copies):
    from paper_2511_08498_gb300 import api
    ctx = api.Context(0)
    planes = planes_of(api, ctx, nx, nz, L, W, 780, (-3.5, -1.5))
    value = {"inf": float("inf"), "nan": float("nan"), "negative S": -3.0, "negative chi": -1e-3}[bad]
    planes[0, nx * (nz // 3) + nx // 2, W if bad == "negative chi" else 0] = value
    dirs, w = synth.directions(16, offset=0.0)
    probes = torch.arange(nx * nz, dtype=torch.int32, device="cuda").repeat(copies) if copies else None
    full = api.formal_solve_dense(ctx, nx, nz, L, W, planes, dirs, w, want_intensity=True, count_segments=True)
    fast = api.formal_solve_dense(ctx, nx, nz, L, W, planes, dirs, w, probes=probes, want_intensity=True)
    sel = slice(None) if probes is None else probes.long()
    equal(full[0][:, sel], fast[0])
    equal(full[1][:, :, sel], fast[1])
