"""GPU test of the launch shape the library picks when the caller leaves it
open: on either side of every line of the rule (polynomials per SM, degree,
polish) roots, status, histogram and counters are those of an explicit
one-role shape bit for bit, with the coefficients on the device and in
page-locked host memory, and under capture."""
from __future__ import annotations

import pytest
import torch

from paper_2507_02164_gb300 import api
from tests.gpu_common import require_gpu

pytestmark = pytest.mark.gpu

WIN = api.Window(-2.0, 2.0, -1.125, 1.125)


@pytest.fixture(scope="module")
def dev():
    return require_gpu()


def _run(co, degree, dev, kw):
    n = co.shape[1]
    hist, stats = api.new_hist(640, 360, dev), api.new_stats(dev)
    roots = torch.empty((degree, n), dtype=torch.complex128, device=dev)
    status = torch.empty(n, dtype=torch.uint8, device=dev)
    api.roots_density(co, WIN, hist, "mixed", api.params("mixed", **kw), roots=roots, status=status, stats=stats)
    torch.cuda.synchronize()
    return torch.view_as_real(roots).view(torch.int64), status, hist, api.stats_dict(stats)


def _same(a, b):
    assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1]) and torch.equal(a[2], b[2]) and a[3] == b[3]
    assert a[3]["wait_timeouts"] == 0


@pytest.mark.parametrize("degree,per_sm,polish", [(4, 640, "fp64"), (6, 576, "fp64"), (8, 352, "fp64"),
                                                  (9, 224, "fp64"), (7, 1536, "df"), (5, 1536, "df"),
                                                  (8, 1536, "df")])
def test_open_shape_is_one_role_bit_for_bit(dev, degree, per_sm, polish):
    sms = torch.cuda.get_device_properties(dev).multi_processor_count
    g = torch.Generator(device=dev).manual_seed(degree)
    for n in (per_sm * sms - 1, per_sm * sms + 1):
        for dt in (torch.float32, torch.float64):
            co = torch.complex(*torch.randn((2, degree + 1, n), generator=g, device=dev, dtype=dt))
            _same(_run(co, degree, dev, {"polish_mode": polish}), _run(co, degree, dev, {"polish_mode": polish, "block": 128}))


def test_open_shape_zero_copy_and_capture(dev):
    n = 800 * torch.cuda.get_device_properties(dev).multi_processor_count
    co = torch.randn((7, n), dtype=torch.complex64, generator=torch.Generator().manual_seed(1))
    ref = _run(co.to(dev), 6, dev, {"block": 128})
    _same(_run(co.pin_memory(), 6, dev, {}), ref)
    c_t, hist = co.to(dev), api.new_hist(640, 360, dev)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        api.roots_density(c_t, WIN, hist, "mixed", api.params("mixed"))
    for _ in range(2):
        api.hist_clear(hist)
        graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(hist, ref[2])
