"""The surrogate's activations: tails at strongly negative pre-activations."""

import pytest
import torch

pytestmark = pytest.mark.gpu

H = 64
W1, B1, W2, B2, W3, B3 = 0, 3 * H, 4 * H, 4 * H + H * H, 5 * H + H * H, 6 * H + H * H


def samples(n, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    r = torch.rand((n, 3), generator=gen, device="cuda")
    return torch.stack([32.0 * r[:, 0] - 16.0, 10.0 ** (-3.0 + 2.0 * r[:, 1]), 20.0 * r[:, 2] - 10.0], 1).contiguous()


def network(seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    p = torch.randn(B3 + 1, generator=gen, device="cuda")
    p[W1:B1] *= 0.8
    p[B1:W2] *= 0.1
    p[W2:B2] *= (2.0 / H) ** 0.5
    return p


# every second-layer unit at z: its activation lies between z 2^(1.5 z) and 0.  From -7.5 down
# that is above -1e-16, and 64 of them with weight 1 above -1e-14
@pytest.mark.parametrize("z", [-7.7, -10.0, -100.0, -1e4, -1e12])
def test_tail(z):
    from paper_2511_08498_gb300 import api
    ctx = api.Context(0)
    xau = samples(300, 1)
    p = network(2)
    p[W2:B2], p[B2:W3], p[W3:B3], p[B3] = 0.0, z, 1.0, 0.0
    y = api.mlp_forward(ctx, xau, p)
    assert y.abs().max().item() < 1e-14
    # d loss / d w3 = mean 2 (y - target) h2, target = 1
    grad, _ = api.mlp_grad(ctx, xau, torch.ones(300, device="cuda"), p)
    ctx.check()
    assert grad[W3:B3].abs().max().item() < 2e-14 and torch.isfinite(grad).all()


def test_nan_stays_nan():
    from paper_2511_08498_gb300 import api
    ctx = api.Context(0)
    p = network(3)
    p[B2 + 5] = float("nan")
    assert torch.isnan(api.mlp_forward(ctx, samples(128, 4), p)).all()
