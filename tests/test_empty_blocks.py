"""Per-batch walks of grids whose blocks are mostly empty: the launches go by the active blocks.

The host knows a grid's blocks, the device how many of them are active.  Where directions are
split and where pairs of batches share a walk is decided by the latter.
"""

import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

BAND = [6.0, 24.0, 96.0]


def medium(nx, nz, L, active_rows, seed, mirrored):
    """Random medium with that many rows of active blocks; ``mirrored``: wavelengths l and L - 1 - l alike."""
    m = synth.random_medium(nx, nz, L, seed=synth.SEED_BASE + seed, log_chi_range=(-3.0, 1.0), emitter_frac=0.0)
    out = []
    for k in ("eta", "chi"):
        a = m[k].copy()
        if mirrored:
            a[L - L // 2:] = a[:L // 2][::-1]
        a[:, 16 * active_rows:] = 0.0
        out.append(torch.from_numpy(a.reshape(L, -1)).cuda())
    return out


# 600 or 1024 blocks; active (block, batch) pairs below and above 912, active blocks of pairs below
# and above what sharing a walk asks for, even and odd numbers of batches
@pytest.mark.parametrize("storage", [0, 1, 2])
@pytest.mark.parametrize("nx,nz,L,rows", [(480, 320, 32, 1), (480, 320, 32, 7), (480, 320, 32, 8), (480, 320, 20, 10),
                                          (480, 320, 24, 11), (512, 512, 16, 12), (512, 512, 24, 21), (480, 320, 32, 0)])
def test_bits(nx, nz, L, rows, storage):
    from paper_2511_08498_gb300 import api
    ctx = api.Context(0)
    dirs, w = synth.directions(5, offset=0.0)
    for mirrored, iod in ((True, 1e-2), (False, 1e30)):
        eta, chi = medium(nx, nz, L, rows, 1010 + L, mirrored)
        grid = api.grid_build(ctx, nx, nz, eta, chi)
        mips = api.mips_build(ctx, grid, eta, chi, 8, 3, iod, iod, storage=storage)
        full = api.formal_solve_hdda(ctx, grid, mips, dirs, w, band=BAND, i_bc=0.2, want_intensity=True,
                                     count_segments=True)
        fast = api.formal_solve_hdda(ctx, grid, mips, dirs, w, band=BAND, i_bc=0.2, want_intensity=True)
        assert torch.equal(full[0], fast[0]) and torch.equal(full[1], fast[1])
    ctx.check()


@pytest.mark.parametrize("W,L,storage", [(1, 2, 0), (2, 4, 0), (4, 8, 0), (4, 8, 1), (4, 7, 2)])
@pytest.mark.parametrize("rows", [10, 14, 15])
def test_bits_of_narrow_batches(W, L, storage, rows):
    """Two batches of 1024 blocks, 640, 896 and 960 active pairs."""
    from paper_2511_08498_gb300 import api
    ctx = api.Context(0)
    eta, chi = medium(512, 512, L, rows, 1050 + W, False)
    grid = api.grid_build(ctx, 512, 512, eta, chi)
    mips = api.mips_build(ctx, grid, eta, chi, W, 3, 1e-2, 1e-2, storage=storage)
    dirs, w = synth.directions(5, offset=0.0)
    full = api.formal_solve_hdda(ctx, grid, mips, dirs, w, band=BAND, i_bc=0.2, count_segments=True)
    assert torch.equal(full[0], api.formal_solve_hdda(ctx, grid, mips, dirs, w, band=BAND, i_bc=0.2)[0])
    ctx.check()


def best_ms(f):
    best = float("inf")
    for _ in range(30):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        a.record()
        f()
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b))
    return best


# split where the grid's blocks would forbid it; no shared walk where they would suggest it
@pytest.mark.parametrize("nx,nz,L,iod,storage,empty", [(480, 320, 32, 1e30, "f32", 0.7), (640, 640, 24, 1.0, "bf16", 0.7)])
def test_as_fast_as_with_the_exact_capacity(nx, nz, L, iod, storage, empty):
    from paper_2511_08498_gb300 import api
    from perf import cases
    s = cases.prepare(dict(kind="line", nx=nx, nz=nz, n_lambda=L, n_dir=24, walk="per_batch", iod=iod, band=cases.BAND,
                           storage=storage, empty=empty), 3)
    ctx = s["ctx"]
    eta, chi = api.synth_static_line(ctx, *s["fields"])
    grid = api.grid_build(ctx, nx, nz, eta, chi)
    times = []
    for capacity in (grid.n_blocks, int(grid.n_active_dev.item())):
        mips = api.mips_build(ctx, grid, eta, chi, 8, 3, iod, iod, capacity=capacity,
                              storage=api.STORE_F32 if storage == "f32" else api.STORE_BF16)
        times.append(best_ms(lambda: api.formal_solve_hdda(ctx, grid, mips, s["dirs"], s["w"], J=s["J"], band=BAND)))
    ctx.check()
    assert times[0] < 1.06 * times[1], times
