"""GPU tests of the split-register solver (rd_solve_split.cuh) with the
compensated polish, degrees 7 to 11: taken by large batches whose launch shape
is open. Roots, status, histogram and counters must be the one-role kernel's
bit for bit, from the line of the dispatch rule on, for both storage types (the
complex128 one keeps the coefficients' FP32 remainders), at ragged sizes, over
the hard polynomials and parameters of the FP64 polish's tests, and for packed
batches."""
from __future__ import annotations

import pytest
import torch

from paper_2507_02164_gb300 import api
from tests.gpu_common import require_gpu
from tests.test_gpu_split import KW, WIN, _coeffs, _run, _same

pytestmark = pytest.mark.gpu

PER_SM = {7: 1536, 8: 640, 9: 256, 10: 256, 11: 256}
UNEVEN_PER_SM = 9216


@pytest.fixture(scope="module")
def dev():
    return require_gpu()


@pytest.mark.parametrize("dtype", [torch.complex64, torch.complex128])
@pytest.mark.parametrize("degree", sorted(PER_SM))
def test_bit_identical_to_one_role(dev, degree, dtype):
    sms = torch.cuda.get_device_properties(dev).multi_processor_count
    for n in (PER_SM[degree] * sms, PER_SM[degree] * sms + 12345, 1700 * sms + 1):
        co = _coeffs(dev, degree, n, dtype)
        _same(_run(co, dev, polish_mode="df"), _run(co, dev, polish_mode="df", block=128))


@pytest.mark.parametrize("kw", KW)
@pytest.mark.parametrize("degree", [8, 11])
def test_parameters(dev, degree, kw):
    n = 700 * torch.cuda.get_device_properties(dev).multi_processor_count + 7
    for dtype in (torch.complex64, torch.complex128):
        co = _coeffs(dev, degree, n, dtype, 1)
        for hist in (True, False):
            _same(_run(co, dev, hist=hist, polish_mode="df", **kw), _run(co, dev, hist=hist, polish_mode="df", block=64, **kw))


@pytest.mark.parametrize("dtype", [torch.complex64, torch.complex128])
@pytest.mark.parametrize("lo,hi", [(0, 14), (9, 12)])
def test_packed_bit_identical(dev, lo, hi, dtype):
    n = UNEVEN_PER_SM * torch.cuda.get_device_properties(dev).multi_processor_count + 3
    g = torch.Generator(device=dev).manual_seed(n)
    deg = torch.randint(lo, hi + 1, (n,), generator=g, device=dev)
    off = torch.zeros(n + 1, dtype=torch.int64, device=dev)
    torch.cumsum(deg + 1, dim=0, out=off[1:])
    real = torch.float32 if dtype == torch.complex64 else torch.float64
    c = torch.complex(*torch.randn((2, int(off[-1])), generator=g, device=dev, dtype=real))
    ws = api.new_uneven_workspace(n, c.numel(), dtype, dev)
    out = []
    for kw in ({}, {"block": 128}):
        h, st = api.new_hist(640, 360, dev), api.new_stats(dev)
        roots, status = api.roots_uneven(c, deg.to(torch.uint8), off, ws, "mixed", api.params("mixed", polish_mode="df", **kw),
                                         window=WIN, hist=h, stats=st)
        torch.cuda.synchronize()
        out.append((torch.view_as_real(roots).view(torch.int64), status, h, api.stats_dict(st)))
    _same(out[0], out[1])
