"""The complex128 adjoint at the ends of the FP64 range: derivatives around the
singularity bound of 1e-300 and above 2^1000, and roots whose powers leave the range,
uniform and packed. Degree 1 has p'(z) = a_1 exactly, so the gradients are known:
-conj(z^k / a_1) grad_z."""
from __future__ import annotations

import numpy as np
import pytest
import torch

from paper_2507_02164_gb300 import api
from tests.gpu_common import require_gpu

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -53


@pytest.fixture(scope="module")
def dev():
    return require_gpu()


def _both(dev, coeffs, roots, grad):
    """(gradient, status) of a batch [d + 1, n], uniform and packed."""
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev)  # noqa: E731
    d, n = roots.shape
    st = torch.empty(n, dtype=torch.uint8, device=dev)
    g = api.roots_backward(t(coeffs), t(roots), t(grad), status=st)
    off = t(np.arange(n + 1, dtype=np.int64) * (d + 1))
    stu = torch.empty(n, dtype=torch.uint8, device=dev)
    gu = api.roots_backward_uneven(t(coeffs.T.reshape(-1)), torch.full((n,), d, dtype=torch.uint8, device=dev), off,
                                   t(roots.T.reshape(-1)), t(grad.T.reshape(-1)), status=stu)
    assert torch.equal(st, stu) and torch.equal(torch.view_as_real(g.T.reshape(-1).contiguous()).view(torch.int64),
                                                torch.view_as_real(gu).view(torch.int64))
    return g.cpu().numpy(), st.cpu().numpy()


def test_singularity_bound(dev):
    """|p'| between 1e-300 / sqrt 2 and 1e-300 in its larger component is decided by the modulus."""
    rng = np.random.default_rng(3)
    mod = 1e-300 * np.concatenate([rng.uniform(0.5, 2.0, 4000), 1.0 + np.array([-1e-13, 1e-13, -0.3, 0.3])])
    ang = rng.uniform(0, 2 * np.pi, mod.size)
    a1 = mod * np.cos(ang) + 1j * mod * np.sin(ang)
    a1[-2:] = [1e-300, np.nextafter(1e-300, 1.0)]  # on the real axis: at the bound and just above
    coeffs = np.stack([np.zeros_like(a1), a1])
    g, st = _both(dev, coeffs, np.full((1, a1.size), 0.5 + 0.25j), np.full((1, a1.size), 1e-5 + 0j))
    size = np.hypot(a1.real, a1.imag)
    clear = np.abs(size - 1e-300) > 1e-300 * 4 * EPS
    clear[-2:] = True
    assert np.array_equal((st == 2)[clear], (size <= 1e-300)[clear])
    assert (g[:, st == 2] == 0).all() and np.isfinite(g[:, st != 2]).all()


@pytest.mark.parametrize("exponent", [-985, -500, 0, 500, 999, 1000, 1001, 1005, 1010])
def test_derivatives_of_every_size(dev, exponent):
    """Scaling by the exponent, one reciprocal, two products: within 16 roundings."""
    rng = np.random.default_rng(abs(exponent))
    n = 2000
    a1 = (rng.standard_normal(n) + 1j * rng.standard_normal(n)) * 2.0 ** exponent
    z = rng.standard_normal(n) + 1j * rng.standard_normal(n)
    up = 2.0 ** (exponent // 2)
    gz = (rng.standard_normal(n) + 1j * rng.standard_normal(n)) * up
    g, st = _both(dev, np.stack([np.zeros_like(a1), a1]), z[None], gz[None])
    q = -np.conj(2.0 ** exponent / a1) * (gz / up) * (up / 2.0 ** exponent)
    want = np.stack([q, q * np.conj(z)])
    assert (st == 0).all()
    assert (np.abs(g - want) <= 16 * EPS * np.abs(want)).all()


def test_powers_beyond_the_range(dev):
    """z^2 overflows, u conj(z)^2 does not; a zero cotangent gives zeros, not NaN."""
    coeffs = np.array([[0.0], [1.0], [1e-10]], dtype=np.complex128).repeat(2, axis=1)
    z = np.full((2, 2), 1e200 + 0j)
    gz = np.zeros((2, 2), dtype=np.complex128)
    gz[0, 0] = 1.0
    g, st = _both(dev, coeffs, z, gz)
    dp = 1.0 + 2e-10 * 1e200
    want = [-1.0 / dp, -1e200 / dp, -1e200 / dp * 1e200]
    assert (st == 0).all() and (np.abs(g[:, 0] - want) <= 16 * EPS * np.abs(want)).all()
    assert (g[:, 1] == 0).all()
