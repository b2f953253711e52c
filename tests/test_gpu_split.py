"""GPU tests of the split-register warp-specialised solver (rd_solve_split.cuh):
taken by large FP64-polish batches whose launch shape is open. Roots, status,
histogram and counters must be the one-role kernel's bit for bit, from the
line of the dispatch rule on, for every degree and storage type, at ragged
sizes, with degenerate, ill-conditioned, rejected and non-convergent
polynomials, every parameter the path takes, the tile clip, packed batches,
zero-copy input and capture."""
from __future__ import annotations

import numpy as np
import pytest
import torch

from paper_2507_02164_gb300 import api
from tests.gpu_common import require_gpu

pytestmark = pytest.mark.gpu

WIN = api.Window(-3.0, 3.0, -1.6875, 1.6875)
PER_SM = {4: 640, 5: 576, 6: 576, 7: 352, 8: 352, 9: 224, 10: 224, 11: 224, 12: 224}
KW = [{}, {"polish_steps": 0, "polish_extra": 0}, {"polish_steps": 0, "polish_extra": 4}, {"polish_steps": 1, "collapse_tol": 0.3},
      {"max_iters": 2}, {"shift": "rayleigh", "exc_period": 5}, {"residual_tol": 1e-17}, {"fixed_sweeps": 6}]


@pytest.fixture(scope="module")
def dev():
    return require_gpu()


def _coeffs(dev, degree, n, dtype, seed=0):
    """Complex-Gaussian, with pairs of roots 10^-1 .. 10^-7 apart (every 16th),
    real +-1 coefficients, zeros at 0, a_d = 0, infinities and small scales."""
    g = torch.Generator(device=dev).manual_seed(100 * degree + seed)
    real = torch.float32 if dtype == torch.complex64 else torch.float64
    c = torch.complex(*torch.randn((2, degree + 1, n), generator=g, device=dev, dtype=real))
    m = (n + 15) // 16
    z = torch.complex(*torch.randn((2, degree, m), generator=g, device=dev, dtype=torch.float64))
    z[1] = z[0] + 10.0 ** (-7.0 + 6.0 * torch.rand(m, generator=g, device=dev, dtype=torch.float64))
    p = torch.zeros((degree + 1, m), dtype=torch.complex128, device=dev)
    p[0] = 1.0
    for k in range(degree):
        up = torch.zeros_like(p)
        up[1:] = p[:-1]
        p = up - z[k] * p
    c[:, ::16] = p.to(dtype)
    c[:, 5::257] = torch.sign(c[:, 5::257].real).to(dtype)
    c[0, 7::263] = 0
    c[degree, 11::1009] = 0
    c[1, 13::1013] = float("inf")
    c[:, 17::271] *= 2.0 ** -40
    return c.contiguous()


def _run(co, dev, clip=None, window=WIN, hist=True, **kw):
    d, n = co.shape[0] - 1, co.shape[1]
    h, st = api.new_hist(640, 360, dev), api.new_stats(dev)
    roots = torch.full((d, n), 3.0, dtype=torch.complex128, device=dev)
    status = torch.full((n,), 9, dtype=torch.uint8, device=dev)
    p = api.params("mixed", **kw)
    if hist:
        api.roots_density(co, window, h, "mixed", p, clip=clip, roots=roots, status=status, stats=st)
    else:
        api.roots_batched(co, "mixed", p, roots=roots, status=status, stats=st)
    torch.cuda.synchronize()
    return torch.view_as_real(roots).view(torch.int64), status, h, api.stats_dict(st)


def _same(a, b):
    assert a[3] == b[3], {k: (a[3][k], b[3][k]) for k in a[3] if a[3][k] != b[3][k]}
    assert torch.equal(a[1], b[1]) and torch.equal(a[0], b[0]) and torch.equal(a[2], b[2])
    assert a[3]["wait_timeouts"] == 0


@pytest.mark.parametrize("dtype", [torch.complex64, torch.complex128])
@pytest.mark.parametrize("degree", sorted(PER_SM))
def test_bit_identical_to_one_role(dev, degree, dtype):
    sms = torch.cuda.get_device_properties(dev).multi_processor_count
    for n in (PER_SM[degree] * sms, PER_SM[degree] * sms + 12345, 1000 * sms + 1):
        co = _coeffs(dev, degree, n, dtype)
        _same(_run(co, dev), _run(co, dev, block=128))


@pytest.mark.parametrize("kw", KW)
@pytest.mark.parametrize("degree", [6, 9, 12])
def test_parameters(dev, degree, kw):
    n = 620 * torch.cuda.get_device_properties(dev).multi_processor_count + 7
    for dtype in (torch.complex64, torch.complex128):
        co = _coeffs(dev, degree, n, dtype, 1)
        _same(_run(co, dev, **kw), _run(co, dev, block=64, **kw))
        _same(_run(co, dev, hist=False, **kw), _run(co, dev, hist=False, block=64, **kw))


def test_clip_zero_copy_and_capture(dev):
    nx, ny = 360, 250
    tiles = api.Window(-1.0, 1.0, -0.5, 0.5)
    ix, iy = torch.arange(nx, device=dev, dtype=torch.float64), torch.arange(ny, device=dev, dtype=torch.float64)
    cen = torch.complex((-1 + (ix + 0.5) * 2 / nx).expand(ny, nx), (0.5 - (iy + 0.5) / ny)[:, None].expand(ny, nx)).reshape(-1).contiguous()
    co = _coeffs(dev, 6, nx * ny, torch.complex128, 2)
    order = torch.randperm(nx * ny, generator=torch.Generator(device=dev).manual_seed(1), device=dev)
    for index in (None, order):
        clip = api.make_clip(cen if index is None else cen[index].contiguous(), 0.01, nx, ny, tiles, tile_index=index)
        a, b = _run(co, dev, clip=clip, window=tiles), _run(co, dev, clip=clip, window=tiles, block=128)
        _same(a, b)
        assert a[3]["binned"] > 0 and a[3]["clipped"] > 0
    co = _coeffs(dev, 6, 90001, torch.complex64, 3)
    ref = _run(co, dev, block=128)
    _same(_run(co.cpu().pin_memory(), dev), ref)
    hist = api.new_hist(640, 360, dev)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        api.roots_density(co, WIN, hist, "mixed", api.params("mixed"))
    for _ in range(2):
        api.hist_clear(hist)
        graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(hist, ref[2])


@pytest.mark.parametrize("dtype", [torch.complex64, torch.complex128])
@pytest.mark.parametrize("n_per_sm,lo,hi", [(6144, 0, 14), (6200, 9, 13), (6150, 4, 5)])
def test_packed_bit_identical(dev, n_per_sm, lo, hi, dtype):
    """All degrees (0, 13 and 14 unsolved), the high ones, and one bin alone."""
    n = n_per_sm * torch.cuda.get_device_properties(dev).multi_processor_count + 3
    g = torch.Generator(device=dev).manual_seed(n)
    deg = torch.randint(lo, hi + 1, (n,), generator=g, device=dev)
    off = torch.zeros(n + 1, dtype=torch.int64, device=dev)
    torch.cumsum(deg + 1, dim=0, out=off[1:])
    real = torch.float32 if dtype == torch.complex64 else torch.float64
    c = torch.complex(*torch.randn((2, int(off[-1])), generator=g, device=dev, dtype=real))
    ws = api.new_uneven_workspace(n, c.numel(), dtype, dev)
    out = []
    # every shape open; explicit; open but for three degrees
    for tuning, kw in ((None, {}), (None, {"block": 128}), (api.uneven_tuning(block={5: 64, 10: 128, 12: 32}), {})):
        h, st = api.new_hist(640, 360, dev), api.new_stats(dev)
        roots, status = api.roots_uneven(c, deg.to(torch.uint8), off, ws, "mixed", api.params("mixed", **kw), tuning=tuning,
                                         window=WIN, hist=h, stats=st)
        torch.cuda.synchronize()
        out.append((torch.view_as_real(roots).view(torch.int64), status, h, api.stats_dict(st)))
    _same(out[0], out[1])
    _same(out[2], out[1])
    assert np.array_equal(np.bincount(status.cpu().numpy(), minlength=4)[3], int(((deg < 1) | (deg > 12)).sum()))
