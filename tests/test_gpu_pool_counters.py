"""The pool solver's counters when a warp's share passes 2^32: a pool sweeps up to
160 polynomials where a warp of the one-role kernel sweeps 32, and its sums over a
round must hold all of them. With a fixed schedule they are known in advance."""
from __future__ import annotations

import pytest
import torch

from paper_2507_02164_gb300 import api
from tests.gpu_common import require_gpu

pytestmark = pytest.mark.gpu


def test_counters_of_a_long_schedule():
    """256 polynomials per SM on four warps: 64 per pool, 4.5e9 flops of each round."""
    dev = require_gpu()
    degree, sweeps = 7, 18000
    n = 256 * torch.cuda.get_device_properties(dev).multi_processor_count
    g = torch.Generator(device=dev).manual_seed(7)
    c = torch.complex(*torch.randn((2, degree + 1, n), generator=g, device=dev, dtype=torch.float64))
    stats = api.new_stats(dev)
    api.roots_batched(c, "plain", api.params("plain", fixed_sweeps=sweeps, max_iters=sweeps), stats=stats)
    got = api.stats_dict(stats)
    sizes = range(2, degree + 1)
    assert 64 * sweeps * sum(20 * (m * (m + 1) - 2) + 24 * (m - 1) + 60 for m in sizes) > 2 ** 32
    assert got["polys"] == n and got["sweeps"] == n * sweeps * (degree - 1)
    assert got["pair_updates"] == n * sweeps * sum(m * (m + 1) - 2 for m in sizes)
    assert got["rotations"] == n * sweeps * sum(m - 1 for m in sizes)
    assert got["flops_fp64"] == n * (sweeps * sum(20 * (m * (m + 1) - 2) + 24 * (m - 1) + 60 for m in sizes) + 4 * degree)
