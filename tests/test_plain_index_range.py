"""Plain solves at the largest sizes that the entry point takes: indices near 2^31."""

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def room():
    torch.cuda.empty_cache()
    if torch.cuda.mem_get_info()[0] < 60e9:
        pytest.skip("needs 60 GB of device memory")
    yield
    torch.cuda.empty_cache()


def solve(nx, nz, planes, dirs, probes=None):
    from paper_2511_08498_gb300 import api
    ctx = api.Context(0)
    dirs = np.asarray(dirs, dtype=np.float32)
    J, I, _ = api.formal_solve_dense(ctx, nx, nz, 1, 1, planes, dirs, np.full(len(dirs), 1.0 / len(dirs), np.float32),
                                     probes=probes, want_intensity=len(dirs) > 1)
    ctx.check()
    return J, I


def test_whole_grid():
    """Cells so near 2^31 that the next step of a loop over them goes beyond it."""
    nx, nz = 65536, 32767
    J, _ = solve(nx, nz, torch.zeros((1, nx * nz, 2), device="cuda"), [[0.0, -1.0]])
    assert J.shape == (1, nx * nz) and J.min().item() == 0.0 and J.max().item() == 0.0


def test_probe_list():
    """2^31 - 1 probes: the number of CTAs, rounded up, is formed beyond 2^31."""
    planes = torch.empty((1, 256, 2), device="cuda")
    planes[..., 0], planes[..., 1] = 1.5, 0.25
    probes = torch.zeros(2 ** 31 - 1, dtype=torch.int32, device="cuda")
    one, _ = solve(16, 16, planes, [[0.0, 1.0]], probes[:1])
    J, _ = solve(16, 16, planes, [[0.0, 1.0]], probes)
    assert J.min().item() == one.item() == J.max().item() > 0.0


def test_rays_across_more_than_2_31_cells():
    """A ray whose records lie more than 2^31 cells behind its probe's, straight and aslant."""
    n = 65536
    planes = torch.zeros((1, n, n, 2), device="cuda")
    planes[0, 40000, :, 0], planes[0, 40000, :, 1] = 3.0, 10.0
    planes[0, n - 1, :, 0], planes[0, n - 1, :, 1] = 1e4, 1.0
    d = [[0.0, 1.0], [0.6, 0.8]]
    J, I = solve(n, n, planes.view(1, n * n, 2), d, torch.tensor([5], dtype=torch.int32, device="cuda"))
    for k, (_, dz) in enumerate(d):
        t1, t2 = 10.0 / dz, 1.0 / dz
        want = 3.0 * (1.0 - np.exp(-t1)) + np.exp(-t1) * 1e4 * (1.0 - np.exp(-t2))
        # relative errors: 4e-6 per update, and float32 path lengths and 2^x in the exponents
        assert abs(I[0, k, 0].item() - want) < 2e-5 * want
