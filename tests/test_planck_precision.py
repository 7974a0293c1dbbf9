"""Planck functions of the preconditioned rates, which stay in double, against extended precision."""

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

H, C, KB = 6.62607015e-27, 2.99792458e10, 1.380649e-16


@pytest.mark.parametrize("lam0", [121.5668, 656.2819, 1875.1])
def test_effective_mean_intensity(lam0):
    """Opaque cells without line opacity and without radiation from outside: Jeff is the mean of
    the Planck function over the samples.

    In units of 2^-53, at most: prefactor 4, exponential 3 and difference 1 with a condition of 1.6
    (arguments from 1; expm1 below), quotient 3, weights and sums 5: 20.  A double argument x
    alone would add up to 1.5 x, 45 at the largest."""
    from paper_2511_08498_gb300 import api
    ctx = api.Context(0)
    atom = api.Atom.from_dict({"energy_ev": [0.0, 1239.841984 / lam0], "g": [2.0, 8.0], "lines": [(0, 1, 1e8, lam0)],
                               "upsilon": {(0, 1): 0.5}, "mass_amu": 1.0}, 1e6, 6.652e-25)
    lam, tag = lam0 * (1.0 + 1e-9 * np.array([-1.0, 0.0, 1.0])), np.zeros(3, np.int32)
    n = 100000
    T = torch.from_numpy(np.geomspace(4e3, 2e5, n).astype(np.float32)).cuda()
    th = 2.0 * np.pi * (np.arange(8) + 0.5) / 8
    _, jeff = api.mali_rates(ctx, atom, lam, tag, T, torch.full((n,), 1e25, device="cuda"),
                             torch.zeros((2, n), dtype=torch.float64, device="cuda"), torch.zeros((3, n), device="cuda"),
                             np.stack([np.cos(th), np.sin(th)], 1).astype(np.float32), np.full(8, 0.125, np.float32))
    ctx.check()
    ld = np.longdouble
    t = T.cpu().numpy().astype(ld)
    B = [ld(2) * ld(H) * v ** 3 / ld(C) ** 2 / np.expm1(ld(H) * v / (ld(KB) * t)) for v in (C / (lam * 1e-7)).astype(ld)]
    ref = (B[0] + 2 * B[1] + B[2]) / 4  # trapezoid weights; the profile is flat to 1e-9
    assert np.abs(jeff[0].cpu().numpy() / ref - 1).max() < 20 * 2.0 ** -53
