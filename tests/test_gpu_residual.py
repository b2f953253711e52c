"""GPU test of the final residual check of RD_MIXED with the FP64 polish: the
evaluation is not made where the last Newton step proves its outcome
(residual_certain in rd_solve.cuh, for the default residual_tol and above).
A residual_tol just below the default evaluates every root; a root that the
proof lets pass has a residual below half of the default bound, so status,
roots and counters must be the same bit for bit."""
from __future__ import annotations

import numpy as np
import pytest
import torch

from paper_2507_02164_gb300 import api, workloads as WL
from tests.gpu_common import require_gpu, to_soa

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    return require_gpu()


def _batch(degree: int, n: int) -> np.ndarray:
    """Gaussian polynomials; every third has a pair of roots 10^-1 .. 10^-7
    apart, every fifth its roots scaled by 10^-6 .. 10^6, every seventh its
    coefficients by 2^-60 .. 2^60 (beyond the proof's range on both sides),
    some a root at 0, and a few are degenerate."""
    rng = np.random.default_rng(1000 + degree)
    c = WL.gaussian(300 + degree, n, degree)
    i = np.arange(n)
    if degree >= 2:
        pick = i[i % 3 == 0]
        r = rng.normal(size=(pick.size, degree)) + 1j * rng.normal(size=(pick.size, degree))
        r[:, 1] = r[:, 0] + 10.0 ** rng.uniform(-7, -1, pick.size) * np.exp(2j * np.pi * rng.uniform(size=pick.size))
        for row, rr in zip(pick, r):
            c[row] = np.poly(rr)[::-1]
    pick = i[i % 5 == 1]
    c[pick] *= (10.0 ** rng.uniform(-6, 6, (pick.size, 1))) ** np.arange(degree + 1)[None, :] if degree <= 5 else 1.0
    pick = i[i % 7 == 2]
    c[pick] *= 2.0 ** rng.integers(-60, 61, (pick.size, 1))
    c[i % 11 == 3, 0] = 0.0
    c[i % 97 == 5, degree] = 0.0
    c[i % 89 == 6, 0] = np.nan
    return c


@pytest.mark.parametrize("dtype", [torch.complex64, torch.complex128])
@pytest.mark.parametrize("degree", list(range(1, 13)))
def test_skipped_residual_changes_nothing(dev, degree, dtype):
    n = 2048 + 13
    co = to_soa(_batch(degree, n), dev, dtype)
    default = 64.0 * degree * 2.0 ** -53
    out = []
    for tol in (0.0, default * (1.0 - 1e-5)):
        for shape in ({}, dict(block=128, polish_warps=2)):
            stats = api.new_stats(dev)
            roots, status = api.roots_batched(co, "mixed", api.params("mixed", residual_tol=tol, **shape), stats=stats)
            torch.cuda.synchronize()
            out.append((torch.view_as_real(roots).view(torch.int64), status, api.stats_dict(stats)))
    assert out[0][2]["status_ok"] > n // 2 and out[0][2]["newton_steps"] > 0
    for roots, status, st in out[1:]:
        assert torch.equal(status, out[0][1])
        assert torch.equal(roots, out[0][0])
        assert st == out[0][2]
