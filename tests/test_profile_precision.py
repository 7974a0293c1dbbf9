"""The Voigt function and the lines' sums at the edges of their branches."""

import numpy as np
import pytest
import torch
from scipy.special import wofz

pytestmark = pytest.mark.gpu


# below |x| + a = 15 the float32 evaluation is good to 6e-7 with exact 2^x, cosine and quotients;
# 2^x adds 2 ulp (2.4e-7), the fast cosine 2^-21.4 of the core's term (3.6e-7), the quotient 2
# ulp: 1.5e-6.  From 15 on it is Humlicek's region I, whose own error is 5e-5 there: no claim
@pytest.mark.parametrize("a", [1e-6, 1e-4, 1e-2, 0.1, 0.2, 0.24, 0.2499999])
def test_voigt_at_small_damping(a):
    from paper_2511_08498_gb300 import api
    ctx = api.Context(0)
    a32 = np.float32(a)
    edges = [e + d for e in (6.0 - a, 15.0 - a) for d in (-1e-3, -1e-6, 0.0, 1e-6, 1e-3)]
    nodes = [(k + 0.5) / 8.0 + d for k in range(48) for d in (-1e-6, 1e-6)]  # half way between expansions
    x = np.concatenate([np.linspace(0.0, 20.0, 40001), edges, nodes]).astype(np.float32)
    x = x[x + a32 < 15.0]
    x = np.concatenate([x, -x])
    h = api.voigt(ctx, torch.full((x.size,), float(a32), device="cuda"), torch.from_numpy(x).cuda())
    ctx.check()
    ref = wofz(x.astype(np.float64) + 1j * float(a32)).real
    assert np.abs(h.cpu().numpy().astype(np.float64) / ref - 1.0).max() < 1.5e-6


# up to 45 samples of a line are kept between the two passes, the others evaluated again
@pytest.mark.parametrize("samples", [2, 45, 46, 120])
def test_line_sums(samples):
    """Rates and emissivities of a line of many samples against extended precision."""
    from paper_2511_08498_gb300 import api
    ctx = api.Context(0)
    ld = np.longdouble
    h, c, kb, amu = 6.62607015e-27, 2.99792458e10, 1.380649e-16, 1.66053906660e-24
    lam0, mass, cell, A = 656.2819, 1.00794, 1e6, 4.4101e7
    atom = api.Atom.from_dict({"energy_ev": [0.0, 1239.841984 / lam0], "g": [2.0, 8.0], "lines": [(0, 1, A, lam0)],
                               "upsilon": {(0, 1): 0.5}, "mass_amu": mass}, cell, 6.652e-25)
    lam = lam0 * (1.0 + 1.6e-4 * np.linspace(-1.0, 1.0, samples))
    tag = np.zeros(samples, np.int32)
    n = 513
    T = np.geomspace(4e3, 1e5, n).astype(np.float32)
    J = np.random.default_rng(5).random((samples, n)).astype(np.float32)
    pops = np.stack([np.full(n, 1e12), np.full(n, 3e11)])
    Tg, ne = torch.from_numpy(T).cuda(), torch.full((n,), 1e12, device="cuda")
    jbar = api.rates_accumulate(ctx, atom, lam, tag, Tg, torch.from_numpy(J).cuda())[0].cpu().numpy()
    eta, chi = (v.cpu().numpy().astype(np.float64) for v in
                api.atom_eta_chi(ctx, atom, lam, tag, Tg, ne, torch.from_numpy(pops).cuda()))
    ctx.check()
    nu, nu0 = c / (lam * 1e-7), c / (lam0 * 1e-7)
    order = np.argsort(nu)
    wq = np.zeros(samples)
    for p, q in zip(order[:-1], order[1:]):
        wq[[p, q]] += 0.5 * (nu[q] - nu[p])
    t = T.astype(ld)
    width = ld(nu0) / ld(c) * np.sqrt(2 * ld(kb) * t / (ld(mass) * ld(amu)))
    e = np.exp(-((nu.astype(ld) - ld(nu0))[:, None] / width) ** 2)
    norm = (wq[:, None] * e).sum(0)
    # double sums of positive terms: at most about 3 roundings a term
    assert np.abs(jbar / ((wq[:, None] * e * J).sum(0) / norm) - 1.0).max() < 3 * samples * 2.0 ** -53 + 2e-14
    f = ld(h) * nu[:, None] / (4 * ld(np.pi)) * e / norm * ld(cell)
    b_ul = A * c * c / (2.0 * h * nu0 ** 3)
    chi_c = 6.652e-25 * 1e12 * cell
    planck = 2 * ld(h) * (nu.astype(ld) ** 3)[:, None] / ld(c) ** 2 / np.expm1(ld(h) * nu[:, None] / (ld(kb) * t))
    assert np.abs(eta / (f * pops[1] * A + chi_c * planck) - 1.0).max() < 2.0 ** -23
    assert np.abs(chi / (f * (pops[0] * 4.0 * b_ul - pops[1] * b_ul) + chi_c) - 1.0).max() < 2.0 ** -23


def test_cold_cells():
    """Arguments beyond the exponential's table: the Planck function is zero, nothing overflows."""
    from paper_2511_08498_gb300 import api
    ctx = api.Context(0)
    atom = api.Atom.from_dict({"energy_ev": [0.0, 10.2], "g": [2.0, 8.0], "lines": [(0, 1, 4.7e8, 121.5668)],
                               "upsilon": {(0, 1): 0.5}, "mass_amu": 1.0}, 1e6, 6.652e-25)
    T = torch.tensor([1e-3, 1.0, 100.0, 169.0, 171.0, 400.0], device="cuda")
    lam, tag = np.array([121.5668, 121.567]), np.array([-1, -1], np.int32)
    eta, chi = api.atom_eta_chi(ctx, atom, lam, tag, T, torch.ones(6, device="cuda"),
                                torch.zeros((2, 6), dtype=torch.float64, device="cuda"))
    ctx.check()
    assert not eta.any() and torch.isfinite(chi).all()  # e^{-h nu / k T} < 1e-120 throughout
