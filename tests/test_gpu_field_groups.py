"""GPU test of the one-launch field path's tile groups: the number of tiles a
warp fits before it solves them depends on the grid (params.ctas_per_sm) and
on the number of tiles; coefficients, roots, status, histogram and counters
must not."""
from __future__ import annotations

import pytest
import torch

from paper_2507_02164_gb300 import api
from tests.gpu_common import require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    return require_gpu()


@pytest.mark.parametrize("mode", ["mixed", "plain"])
@pytest.mark.parametrize("nx,ny", [(1, 1), (3, 2), (31, 1), (33, 1), (64, 38), (97, 51), (152, 17)])
def test_groups_do_not_change_the_result(dev, nx, ny, mode):
    tiles = api.Window(-2.03, 1.91, -1.07, 1.13)
    out = []
    for cps in (0, 1):
        n = nx * ny
        hist, stats = api.new_hist(320, 180, dev), api.new_stats(dev)
        co = torch.empty((7, n), dtype=torch.complex128, device=dev)
        roots = torch.empty((6, n), dtype=torch.complex128, device=dev)
        status = torch.empty(n, dtype=torch.uint8, device=dev)
        api.field_density(api.field_spec(tiles, nx, ny), tiles, hist, mode=mode, params_=api.params(mode, ctas_per_sm=cps),
                          coeffs=co, roots=roots, status=status, stats=stats)
        torch.cuda.synchronize()
        bits = lambda t: torch.view_as_real(t).view(torch.int64)  # noqa: E731
        out.append((bits(co), bits(roots), status, hist, api.stats_dict(stats)))
    a, b = out
    assert a[4] == b[4] and a[4]["polys"] == nx * ny
    assert all(torch.equal(x, y) for x, y in zip(a[:4], b[:4]))
    # and the tiles of a larger grid's corner are those of the same tiles alone
    half = api.Window(tiles.xmin, tiles.xmin + (tiles.xmax - tiles.xmin) / nx, tiles.ymax - (tiles.ymax - tiles.ymin) / ny, tiles.ymax)
    co = torch.empty((7, 1), dtype=torch.complex128, device=dev)
    api.field_density(api.field_spec(half, 1, 1), tiles, api.new_hist(320, 180, dev), mode=mode, params_=api.params(mode), coeffs=co)
    torch.cuda.synchronize()
    ref = torch.view_as_complex(a[0].view(torch.float64))[:, 0]
    assert (co[:, 0] - ref).abs().max() <= 1e-13 * ref.abs().max()
