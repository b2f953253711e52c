"""GPU tests of the FP64 L2 sums (four-angle transform, radius groups): node
counts that do not fill the groups, degrees on both sides of a pass of eight
coefficients, batch sizes around the launch's steps, against FP64 sums made
here; samples near the overflow limit and non-finite ones."""
from __future__ import annotations

import math

import numpy as np
import pytest
import torch

from paper_2507_02164_gb300 import api
from tests.gpu_common import require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    return require_gpu()


def _reference(s, nr, degree):
    x, w = np.polynomial.legendre.leggauss(nr)
    r, w = 0.5 * (x + 1.0), 0.5 * w
    th = 2.0 * math.pi * np.arange(32) / 32
    m = np.stack([(2 * (j + 1) / 32) * ((w * r ** (j + 1))[:, None] * np.exp(-1j * j * th)).reshape(-1) for j in range(degree + 1)], 1)
    return s @ m


# every coefficient sums nr * 32 terms of modulus <= |s| with weights that sum
# to 2 (j + 1) / (j + 2) < 2: rounding <= (nr * 32) 2^-53 * 2 max|s|, tables included
@pytest.mark.parametrize("n", [1, 7, 151, 153, 1216, 1217, 9729])
@pytest.mark.parametrize("nr,degree", [(1, 0), (2, 3), (3, 7), (5, 8), (16, 6), (17, 12), (31, 9), (32, 12)])
def test_l2_fp64_against_direct_sums(dev, n, nr, degree):
    if n > 2000 and nr > 16:
        n //= 8
    g = np.random.default_rng(nr * 100 + degree)
    s = g.standard_normal((n, nr * 32)) + 1j * g.standard_normal((n, nr * 32))
    got = api.l2_approx(torch.from_numpy(s).to(dev), nr, 32, degree).cpu().numpy().T
    assert np.abs(got - _reference(s, nr, degree)).max() <= nr * 32 * 2.0 ** -52 * np.abs(s).max()


def test_l2_fp64_near_overflow_and_nonfinite(dev):
    g = np.random.default_rng(1)
    s = g.uniform(0.5, 1.0, (64, 512)) * np.exp(0.2j * g.uniform(size=(64, 512)))  # moduli in [0.5, 1]
    big = s * 1.7e308
    got = api.l2_approx(torch.from_numpy(big).to(dev), 16, 32, 6).cpu().numpy().T
    assert np.all(np.isfinite(got))
    assert np.abs(got / 1.7e308 - _reference(s, 16, 6)).max() <= 512 * 2.0 ** -52
    bad = s.copy()
    bad[3, 17] = np.nan
    bad[9, 300] = np.inf
    got = api.l2_approx(torch.from_numpy(bad).to(dev), 16, 32, 6).cpu().numpy().T
    fine = np.setdiff1d(np.arange(64), [3, 9])
    assert not np.isfinite(got[3]).any() and not np.isfinite(got[9]).any()
    assert np.abs(got[fine] - _reference(s[fine], 16, 6)).max() <= 512 * 2.0 ** -52
