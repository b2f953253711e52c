"""Packed batches between the sizes that always take the group solver and those
that always take the degree bins: the degrees counted on the device decide.
Which form ran is read off the workspace (the bins' permutation); the results are
those of the bins bit for bit either way."""
from __future__ import annotations

import ctypes

import pytest
import torch

from paper_2507_02164_gb300 import _native as N
from paper_2507_02164_gb300 import api
from tests.gpu_common import require_gpu
from tests.test_gpu_split import WIN, _same

pytestmark = pytest.mark.gpu

SURE = {("mixed", "fp64"): 88, ("mixed", "df"): 56, ("plain", "fp64"): 16}  # polynomials per SM: groups up to here
HIGH = {("mixed", "fp64"): 104, ("mixed", "df"): 80, ("plain", "fp64"): 16}  # degrees 5 and 6 may have a bin from here on
MOST = {("mixed", "fp64"): 144, ("mixed", "df"): 128, ("plain", "fp64"): 24}  # bins from here on


@pytest.fixture(scope="module")
def dev():
    return require_gpu()


def _batch(dev, degrees, dtype):
    off = torch.zeros(degrees.numel() + 1, dtype=torch.int64, device=dev)
    torch.cumsum(degrees + 1, dim=0, out=off[1:])
    g = torch.Generator(device=dev).manual_seed(degrees.numel())
    real = torch.float32 if dtype == torch.complex64 else torch.float64
    return torch.complex(*torch.randn((2, int(off[-1])), generator=g, device=dev, dtype=real)), off


def _run(dev, c, degrees, off, mode, ws, **kw):
    n = degrees.numel()
    h, st = api.new_hist(640, 360, dev), api.new_stats(dev)
    roots = torch.full((c.numel() - n,), 3.0, dtype=torch.complex128, device=dev)
    status = torch.full((n,), 9, dtype=torch.uint8, device=dev)
    api.roots_uneven(c, degrees.to(torch.uint8), off, ws, mode, api.params(mode, **kw), window=WIN, hist=h, stats=st, roots=roots,
                     status=status)
    torch.cuda.synchronize()
    return torch.view_as_real(roots).view(torch.int64), status, h, api.stats_dict(st)


def _permuted(ws, n):
    """Whether the call has written the bins' permutation (the workspace held -1)."""
    perm = ws.view(torch.uint8)[512:512 + 4 * n].view(torch.int32)
    return bool((perm != -1).any())


def _degrees(kind, n, dev):
    i = torch.arange(n, device=dev)
    if kind == "one":
        return torch.full((n,), 9, device=dev)
    if kind == "two":
        return 7 + i % 2
    if kind == "spread":
        return 2 + i % 11
    if kind in ("low", "six"):  # never and (above HIGH polynomials per SM) sometimes with a bin
        return torch.full((n,), 4 if kind == "low" else 6, device=dev)
    # exactly a third of degree 8 ("third") or one polynomial more ("above"), the rest below that share
    return torch.where(i < n // 3 + (kind == "above"), 8, 1 + i % 4 + 8 * (i % 2))


@pytest.mark.parametrize("dtype", [torch.complex64, torch.complex128])
@pytest.mark.parametrize("mode,polish", sorted(SURE))
@pytest.mark.parametrize("kind", ["one", "two", "spread", "low", "six", "third", "above"])
def test_the_degrees_decide(dev, kind, mode, polish, dtype):
    sms = torch.cuda.get_device_properties(dev).multi_processor_count
    kw = {"polish_mode": polish} if mode == "mixed" else {}
    sure, high, most = (line[mode, polish] * sms for line in (SURE, HIGH, MOST))
    for line, extra in ((sure, 0), (sure, 3), (high, 0), (high, 3), (most, 0), (most, 3)):
        n = 3 * ((line + extra) // 3)
        degrees = _degrees(kind, n, dev)
        c, off = _batch(dev, degrees, dtype)
        ws = api.new_uneven_workspace(n, c.numel(), dtype, dev)
        ws.fill_(255)
        a = _run(dev, c, degrees, off, mode, ws, **kw)
        bins = n > most or (sure < n and kind in ("one", "two", "above")) or (high < n and kind == "six")
        assert _permuted(ws, n) == bins, (n, line, extra)
        _same(a, _run(dev, c, degrees, off, mode, ws, block=128, **kw))


def test_unsolvable_overlapping_and_captured(dev):
    sms = torch.cuda.get_device_properties(dev).multi_processor_count
    n = 100 * sms + 5
    degrees = torch.arange(n, device=dev) % 15  # 0, 13 and 14 are not solved
    c, off = _batch(dev, degrees, torch.complex64)
    ws = api.new_uneven_workspace(n, c.numel(), c.dtype, dev)
    ref = _run(dev, c, degrees, off, "mixed", ws, block=128)
    _same(_run(dev, c, degrees, off, "mixed", ws), ref)
    # no helper streams: all on one stream
    hist, stats = api.new_hist(640, 360, dev), api.new_stats(dev)
    roots, status = torch.full((c.numel() - n,), 3.0, dtype=torch.complex128, device=dev), torch.full((n,), 9, dtype=torch.uint8, device=dev)
    win, prm = WIN.c(), api.params("mixed")
    p = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    d8 = degrees.to(torch.uint8)
    assert N.load().rd_roots_uneven_static(p(c), N.C64, p(d8), p(off), n, c.numel(), N.MIXED, ctypes.byref(prm), None, ctypes.byref(win),
                                           640, 360, p(hist), p(roots), p(status), p(stats), None) == 0
    torch.cuda.synchronize()
    _same((torch.view_as_real(roots).view(torch.int64), status, hist, api.stats_dict(stats)), ref)
    # ranges that overlap: the second half's start over at offset n / 2, so that the
    # solvable polynomials need more coefficients than there are
    h = n // 2
    deg2 = 3 + torch.arange(n, device=dev) % 4
    step = deg2 + 1
    off2 = torch.zeros(n + 1, dtype=torch.int64, device=dev)
    torch.cumsum(step[:h], dim=0, out=off2[1:h + 1])
    off2[h + 1:] = h + torch.cumsum(step, dim=0)[h:] - int(step[:h].sum())
    c2 = c[: int(6.5 * h) + 32]
    a = _run(dev, c2, deg2, off2, "mixed", ws)
    _same(a, _run(dev, c2, deg2, off2, "mixed", ws, block=128))
    assert bool((a[1] == 3).all())
    stats = api.new_stats(dev)
    roots = torch.empty(c.numel() - n, dtype=torch.complex128, device=dev)
    status = torch.empty(n, dtype=torch.uint8, device=dev)
    hist = api.new_hist(640, 360, dev)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        api.roots_uneven(c, d8, off, ws, "mixed", api.params("mixed"), window=WIN, hist=hist, stats=stats, roots=roots, status=status)
    for solved in (degrees, torch.full_like(degrees, 9)):  # the same graph: spread, then one degree in every range that fits it
        d8.copy_(solved.to(torch.uint8))
        for t in (hist, stats):
            api.hist_clear(t)
        roots.fill_(3.0)
        status.fill_(9)
        graph.replay()
        torch.cuda.synchronize()
        _same((torch.view_as_real(roots).view(torch.int64), status, hist, api.stats_dict(stats)),
              _run(dev, c, solved, off, "mixed", ws, block=128))
