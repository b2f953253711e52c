"""GPU tests of the small-batch solver (rd_group.cuh: a group of lanes per
polynomial, the matrix in shared memory), which small batches take when the
caller leaves the launch shape open: roots, status, histogram and counters
must be those of the one-thread-per-polynomial kernel bit for bit, for every
degree, storage type, mode and shift, at ragged sizes, with degenerate, ill-
conditioned and non-convergent polynomials, and for packed batches whose
offsets are wrong or overlap."""
from __future__ import annotations

import numpy as np
import pytest
import torch

from paper_2507_02164_gb300 import api, workloads as WL
from tests.gpu_common import require_gpu, to_soa

pytestmark = pytest.mark.gpu

W, H = 640, 360
WIN = api.Window(-3.0, 3.0, -1.6875, 1.6875)
MODES = [("plain", {}), ("mixed", {}), ("mixed", {"polish_mode": "df"}),
         ("mixed", {"shift": "rayleigh", "exc_period": 4}), ("mixed", {"polish_steps": 0, "polish_extra": 0}),
         ("mixed", {"fixed_sweeps": 5, "max_iters": 5}), ("plain", {"max_iters": 2}), ("mixed", {"max_iters": 1}),
         ("mixed", {"polish_steps": 1, "polish_extra": 16, "collapse_tol": 0.3})]


@pytest.fixture(scope="module")
def dev():
    return require_gpu()


def _batch(degree: int, n: int) -> np.ndarray:
    rng = np.random.default_rng(40 + degree)
    c = WL.gaussian(60 + degree, n, degree)
    i = np.arange(n)
    if degree >= 2:  # a pair of roots 10^-1 .. 10^-7 apart
        for row in i[i % 4 == 1]:
            r = rng.normal(size=degree) + 1j * rng.normal(size=degree)
            r[1] = r[0] + 10.0 ** rng.uniform(-7, -1)
            c[row] = np.poly(r)[::-1]
    c[i % 13 == 2, 0] = 0.0
    c[i % 17 == 3] = np.sign(c[i % 17 == 3].real)  # real +-1 coefficients
    c[i % 19 == 4, degree] = 0.0
    c[i % 23 == 5, degree // 2] = np.inf
    c[i % 29 == 6] *= 1e-12
    return c


def _bits(r):
    return torch.view_as_real(r).view(torch.int64)


@pytest.mark.parametrize("mode,kw", MODES)
@pytest.mark.parametrize("dtype", [torch.complex64, torch.complex128])
@pytest.mark.parametrize("degree", list(range(1, 13)))
def test_uniform_bit_identical(dev, degree, dtype, mode, kw):
    # mixed below degree 3 and plain below 6 keep the one-thread kernel; the
    # largest sizes lie on either side of the line (40 and 8 per SM)
    sms = torch.cuda.get_device_properties(dev).multi_processor_count
    edge = (40 if mode == "mixed" else 8) * sms
    for n in (1, 3, 1021, edge, edge + 1):
        co = to_soa(_batch(degree, n), dev, dtype)
        out = []
        for shape in ({}, {"block": 128}):
            p = api.params(mode, **kw, **shape)
            hist, stats = api.new_hist(W, H, dev), api.new_stats(dev)
            roots = torch.empty((degree, n), dtype=torch.complex128, device=dev)
            status = torch.empty(n, dtype=torch.uint8, device=dev)
            api.roots_density(co, WIN, hist, mode, p, roots=roots, status=status, stats=stats)
            torch.cuda.synchronize()
            out.append((_bits(roots), status, hist, api.stats_dict(stats)))
        (ra, sa, ha, ta), (rb, sb, hb, tb) = out
        assert torch.equal(sa, sb)
        assert torch.equal(ra, rb)
        assert torch.equal(ha, hb)
        assert ta == tb, {k: (ta[k], tb[k]) for k in ta if ta[k] != tb[k]}


def test_clip_bit_identical(dev):
    """The own-tile clip, with and without a tile index."""
    tiles = api.Window(-1.0, 1.0, -0.5, 0.5)
    centres, rho, _, _ = WL.tiles(*tiles.tuple(), 40, 20)
    n = centres.size
    co = to_soa(WL.gaussian(3, n, 6), dev)
    c_t = torch.from_numpy(centres).to(dev)
    index = torch.arange(n, device=dev)
    for idx in (None, index):
        out = []
        for shape in ({}, {"block": 64}):
            hist, stats = api.new_hist(W, H, dev), api.new_stats(dev)
            clip = api.make_clip(c_t, 40.0 * rho, 40, 20, tiles, tile_index=idx)
            api.roots_density(co, tiles, hist, "mixed", api.params("mixed", **shape), clip=clip, stats=stats)
            torch.cuda.synchronize()
            out.append((hist, api.stats_dict(stats)))
        assert torch.equal(out[0][0], out[1][0]) and out[0][1] == out[1][1]
        assert out[0][1]["binned"] > 0 and out[0][1]["clipped"] > 0


@pytest.mark.parametrize("mode,kw", MODES[:3])
@pytest.mark.parametrize("dtype", [torch.complex64, torch.complex128])
@pytest.mark.parametrize("n,fault", [(1, None), (2, None), (777, None), (3001, None), (777, "offset"), (777, "overlap")])
def test_uneven_bit_identical(dev, n, fault, dtype, mode, kw):
    rng = np.random.default_rng(n)
    deg = rng.integers(0, 15, n).astype(np.uint8)  # degrees 0, 13 and 14 are not solved
    if n > 3:
        deg[3] = 12
    off = np.zeros(n + 1, dtype=np.int64)
    np.cumsum(deg.astype(np.int64) + 1, out=off[1:])
    packed = rng.normal(size=int(off[-1])) + 1j * rng.normal(size=int(off[-1]))
    if fault == "offset":  # one polynomial's range disagrees with its degree
        deg[5] = (int(deg[5]) + 1) % 12
    if fault == "overlap":  # the same range over and over: more coefficients than there are
        deg[:], size = 6, 7 * 300
        off = np.zeros(n + 1, dtype=np.int64)
        off[:] = np.minimum(7 * np.arange(n + 1), size)
        off[n // 3:] = n  # not monotone
        off[n // 3 + 1::2] = n + 7
        packed = packed[:n * 2] if packed.size >= n * 2 else packed
    c_t = torch.from_numpy(packed).to(dev, dtype)
    d_t, o_t = torch.from_numpy(deg).to(dev), torch.from_numpy(off).to(dev)
    ws = api.new_uneven_workspace(n, c_t.numel(), dtype, dev)
    out = []
    for shape in ({}, {"block": 128}):
        hist, stats = api.new_hist(W, H, dev), api.new_stats(dev)
        roots = torch.full((max(c_t.numel() - n, 1),), 7.0, dtype=torch.complex128, device=dev)
        status = torch.full((n,), 9, dtype=torch.uint8, device=dev)
        api.roots_uneven(c_t, d_t, o_t, ws, mode=mode, params_=api.params(mode, **kw, **shape), window=WIN, hist=hist,
                         roots=roots, status=status, stats=stats)
        torch.cuda.synchronize()
        out.append((_bits(roots), status, hist, api.stats_dict(stats)))
    (ra, sa, ha, ta), (rb, sb, hb, tb) = out
    assert torch.equal(sa, sb)
    assert torch.equal(ra, rb)
    assert torch.equal(ha, hb)
    assert ta == tb, {k: (ta[k], tb[k]) for k in ta if ta[k] != tb[k]}
