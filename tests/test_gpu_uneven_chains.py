"""GPU tests of the uneven call's chains: a host thread whose first call was a
small batch can capture a large one; captured and eager calls with twelve and
with four chains give the same bits, also from several threads at once."""
from __future__ import annotations

import threading

import pytest
import torch

from paper_2507_02164_gb300 import api
from tests.gpu_common import require_gpu

pytestmark = pytest.mark.gpu

WIN = api.Window(-3.0, 3.0, -1.6875, 1.6875)


@pytest.fixture(scope="module")
def dev():
    return require_gpu()


def _batch(dev, n, seed):
    g = torch.Generator(device=dev).manual_seed(seed)
    deg = torch.randint(1, 13, (n,), generator=g, device=dev)
    off = torch.zeros(n + 1, dtype=torch.int64, device=dev)
    torch.cumsum(deg + 1, dim=0, out=off[1:])
    c = torch.complex(*torch.randn((2, int(off[-1])), generator=g, device=dev))
    return c, deg.to(torch.uint8), off, api.new_uneven_workspace(n, c.numel(), c.dtype, dev)


def _call(b, hist, **kw):
    return api.roots_uneven(*b, "mixed", api.params("mixed", **kw), window=WIN, hist=hist)


def _work(dev, per_sm, seed, fail):
    try:
        torch.cuda.set_device(dev)
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            sms = torch.cuda.get_device_properties(dev).multi_processor_count
            small, large = _batch(dev, 100, seed), _batch(dev, per_sm * sms + 5, seed + 1)
            _call(small, api.new_hist(320, 180, dev))
            graph, hist = torch.cuda.CUDAGraph(), api.new_hist(320, 180, dev)
            stream.synchronize()
            with torch.cuda.graph(graph, stream=stream, capture_error_mode="thread_local"):
                roots, status = _call(large, hist)
            for _ in range(3):
                api.hist_clear(hist)
                graph.replay()
                h2 = api.new_hist(320, 180, dev)
                r2, s2 = _call(large, h2, block=128)
                stream.synchronize()
                assert torch.equal(hist, h2) and torch.equal(status, s2)
                assert torch.equal(torch.view_as_real(roots).view(torch.int64), torch.view_as_real(r2).view(torch.int64))
    except BaseException as e:  # noqa: BLE001
        fail.append(e)


@pytest.mark.parametrize("per_sm", [300, 1536, 1600, 6200])
def test_small_call_then_capture_of_a_large_one(dev, per_sm):
    fail = []
    t = threading.Thread(target=_work, args=(dev, per_sm, per_sm, fail))  # a thread of its own: its first call
    t.start()
    t.join()
    assert not fail, fail


def _eager(dev, per_sm, seed, fail):
    try:
        torch.cuda.set_device(dev)
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            b = _batch(dev, per_sm * torch.cuda.get_device_properties(dev).multi_processor_count + 3, seed)
            h1, h2 = api.new_hist(320, 180, dev), api.new_hist(320, 180, dev)
            r1, s1 = _call(b, h1)
            r2, s2 = _call(b, h2, block=64)
            stream.synchronize()
            assert torch.equal(h1, h2) and torch.equal(s1, s2)
            assert torch.equal(torch.view_as_real(r1).view(torch.int64), torch.view_as_real(r2).view(torch.int64))
    except BaseException as e:  # noqa: BLE001
        fail.append(e)


def test_threads(dev):
    """Each thread has helper streams of its own (torch captures one graph at a time, so these calls are eager)."""
    fail = []
    ts = [threading.Thread(target=_eager, args=(dev, p, p + 7, fail)) for p in (20, 280, 900, 2000)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not fail, fail
