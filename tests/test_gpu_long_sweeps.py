"""Sweep bounds far above the defaults: a task of 32 polynomials then takes
seconds, longer than the hand-off between warps waits. Such a call takes a form
without waits: no wait runs out, and every polynomial gets all its sweeps."""
from __future__ import annotations

import pytest
import torch

from paper_2507_02164_gb300 import api
from tests.gpu_common import require_gpu

pytestmark = pytest.mark.gpu

SWEEPS = 100000  # the largest bound that the parameters take: 3 to 4 s for a task of degree 12


@pytest.fixture(scope="module")
def dev():
    return require_gpu()


@pytest.mark.parametrize("packed", [False, True])
def test_every_polynomial_gets_its_sweeps(dev, packed):
    """The smallest batches that the split form takes: degree 12, uniform, and
    packed with all but 64 polynomials of degree 1 (which have nothing to sweep)."""
    sms = torch.cuda.get_device_properties(dev).multi_processor_count
    g = torch.Generator(device=dev).manual_seed(12)
    p = api.params("mixed", fixed_sweeps=SWEEPS, max_iters=SWEEPS)
    stats = api.new_stats(dev)
    n, long = (6144 * sms, 64) if packed else (224 * sms, 224 * sms)
    if packed:
        deg = torch.ones(n, dtype=torch.int64, device=dev)
        deg[:: n // long][:long] = 12
        off = torch.zeros(n + 1, dtype=torch.int64, device=dev)
        torch.cumsum(deg + 1, dim=0, out=off[1:])
        c = torch.complex(*torch.randn((2, int(off[-1])), generator=g, device=dev))
        ws = api.new_uneven_workspace(n, c.numel(), c.dtype, dev)
        api.roots_uneven(c, deg.to(torch.uint8), off, ws, "mixed", p, stats=stats)
        long = int((deg == 12).sum())
    else:
        c = torch.complex(*torch.randn((2, 13, n), generator=g, device=dev))
        api.roots_batched(c, "mixed", p, stats=stats)
    got = api.stats_dict(stats)
    assert got["wait_timeouts"] == 0
    assert got["sweeps"] == long * 11 * SWEEPS
    assert got["polys"] == n
