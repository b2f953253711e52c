"""GPU tests of the pool solver (rd_pool.cu): RD_PLAIN_FP64, degrees 3 to 7,
taken by large uniform batches whose launch shape is open. Roots, status,
histogram and counters must be the one-role kernel's bit for bit, from the line
of the dispatch rule on, for both storage types, at sizes that leave pools
ragged, full, in two rounds and (for whole warps) empty, with degenerate,
clustered and non-convergent polynomials, every parameter of the sweeps, the
tile clip, zero-copy input and capture."""
from __future__ import annotations

import pytest
import torch

from paper_2507_02164_gb300 import api
from tests.gpu_common import require_gpu
from tests.test_gpu_split import WIN, _coeffs, _same

pytestmark = pytest.mark.gpu

PER_SM = {3: 448, 4: 256, 5: 256, 6: 256, 7: 256}
KW = [{"max_iters": 1}, {"max_iters": 3}, {"shift": "rayleigh", "exc_period": 5}, {"fixed_sweeps": 4}, {"tol": 1e-6}]


@pytest.fixture(scope="module")
def dev():
    return require_gpu()


def _run(co, dev, clip=None, window=WIN, hist=True, **kw):
    d, n = co.shape[0] - 1, co.shape[1]
    h, st = api.new_hist(640, 360, dev), api.new_stats(dev)
    roots = torch.full((d, n), 3.0, dtype=torch.complex128, device=dev)
    status = torch.full((n,), 9, dtype=torch.uint8, device=dev)
    p = api.params("plain", **kw)
    if hist:
        api.roots_density(co, window, h, "plain", p, clip=clip, roots=roots, status=status, stats=st)
    else:
        api.roots_batched(co, "plain", p, roots=roots, status=status, stats=st)
    torch.cuda.synchronize()
    return torch.view_as_real(roots).view(torch.int64), status, h, api.stats_dict(st)


@pytest.mark.parametrize("dtype", [torch.complex64, torch.complex128])
@pytest.mark.parametrize("degree", sorted(PER_SM))
def test_bit_identical_to_one_role(dev, degree, dtype):
    sms = torch.cuda.get_device_properties(dev).multi_processor_count
    for n in (PER_SM[degree] * sms, PER_SM[degree] * sms + 1, 640 * sms, 640 * sms + 1, 1000 * sms + 12345):
        co = _coeffs(dev, degree, n, dtype)
        _same(_run(co, dev), _run(co, dev, block=64))


@pytest.mark.parametrize("kw", KW)
@pytest.mark.parametrize("degree", [3, 6, 7])
def test_parameters(dev, degree, kw):
    n = 500 * torch.cuda.get_device_properties(dev).multi_processor_count + 77
    for dtype in (torch.complex64, torch.complex128):
        co = _coeffs(dev, degree, n, dtype, 1)
        for hist in (True, False):
            _same(_run(co, dev, hist=hist, **kw), _run(co, dev, hist=hist, block=64, **kw))


def test_clip_zero_copy_and_capture(dev):
    nx, ny = 360, 250
    tiles = api.Window(-1.0, 1.0, -0.5, 0.5)
    ix, iy = torch.arange(nx, device=dev, dtype=torch.float64), torch.arange(ny, device=dev, dtype=torch.float64)
    cen = torch.complex((-1 + (ix + 0.5) * 2 / nx).expand(ny, nx), (0.5 - (iy + 0.5) / ny)[:, None].expand(ny, nx)).reshape(-1).contiguous()
    co = _coeffs(dev, 6, nx * ny, torch.complex128, 2)
    clip = api.make_clip(cen, 0.01, nx, ny, tiles)
    a, b = _run(co, dev, clip=clip, window=tiles), _run(co, dev, clip=clip, window=tiles, block=64)
    _same(a, b)
    assert a[3]["binned"] > 0 and a[3]["clipped"] > 0
    co = _coeffs(dev, 5, 90001, torch.complex64, 3)
    ref = _run(co, dev, block=64)
    _same(_run(co.cpu().pin_memory(), dev), ref)
    hist = api.new_hist(640, 360, dev)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        api.roots_density(co, WIN, hist, "plain", api.params("plain"))
    for _ in range(2):
        api.hist_clear(hist)
        graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(hist, ref[2])
