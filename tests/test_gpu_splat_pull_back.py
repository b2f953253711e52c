"""GPU test of the FP64 splat pull-back's pixel skip: a pixel that no root of
a warp reaches is skipped on FP32 copies of the factors, and the cut is tested
in FP64 only where they cannot tell."""
from __future__ import annotations

import numpy as np
import pytest
import torch

from paper_2507_02164_gb300 import splat
from tests.gpu_common import require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    return require_gpu()


@pytest.mark.parametrize("sigma", [0.3, 0.6, 1.0, 1.5, 2.0])
@pytest.mark.parametrize("n", [1, 31, 33, 4097])
def test_pull_back_skips_only_pixels_outside(dev, sigma, n):
    """The FP64 pull-back skips a pixel that no root of a warp reaches: against
    direct FP64 sums, with roots inside, across and far outside every image
    edge, at pixel centres and corners, at huge and non-finite coordinates, and
    at ragged counts. Each root's sum has at most 169 terms |G e du| <= |G| 6:
    2^-53 times a few hundred of them."""
    W, H, win = 40, 24, (-2.0, 2.0, -1.2, 1.2)
    g = np.random.default_rng(n)
    z = g.uniform(-2.6, 2.6, n) + 1j * g.uniform(-1.7, 1.7, n)
    px, py = 4.0 / W, 2.4 / H
    z[::5] = -2.0 + px * (np.round((z[::5].real + 2.0) / px) + 0.5) + 1j * (1.2 - py * (np.round((1.2 - z[::5].imag) / py)))
    if n > 30:
        z[3], z[4], z[6], z[7], z[8] = np.nan, 1e300, -1e18j, complex(0, np.inf), 2.0**31
    G = g.standard_normal((H, W))
    z_t = torch.from_numpy(z).to(dev).requires_grad_(True)
    img = splat.splat(z_t, win, W, H, sigma, n_norm=1)
    img.backward(torch.from_numpy(G).to(dev))
    got = z_t.grad.cpu().numpy()
    u, v = (z.real - win[0]) / px - 0.5, (win[3] - z.imag) / py - 0.5
    with np.errstate(all="ignore"):
        du, dv = u[:, None, None] - np.arange(W)[None, None, :], v[:, None, None] - np.arange(H)[None, :, None]
        r2 = du * du + dv * dv
        e = np.where(r2 < 9 * sigma * sigma, np.exp(-r2 / (2 * sigma * sigma)), 0.0)
        ge = np.where(e > 0, G[None] * e, 0.0)
        ref = -(np.where(e > 0, ge * du, 0).sum((1, 2)) / px - 1j * np.where(e > 0, ge * dv, 0).sum((1, 2)) / py) / sigma**2
    # a centre within rounding of the circle may fall on either side
    edge = (np.abs(r2 - 9 * sigma * sigma) < 1e-9).any((1, 2))
    ok = ~edge
    assert ok.mean() > 0.5 or n == 1
    assert np.all(np.abs(got - ref)[ok] <= 500 * 2.0**-52 * np.abs(G).max() * 6 / (sigma**2 * min(px, py)))
