"""Packed complex128 batches whose roots go over their coefficients: each
polynomial's coefficients are read before any roots are written, for small
batches as for large ones."""
from __future__ import annotations

import pytest
import torch

from paper_2507_02164_gb300 import api
from tests.gpu_common import require_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["mixed", "plain"])
@pytest.mark.parametrize("n", [2, 501, 2400, 8001, 20003])
def test_roots_over_the_coefficients(n, mode):
    dev = require_gpu()
    g = torch.Generator(device=dev).manual_seed(n)
    deg = torch.randint(1, 13, (n,), generator=g, device=dev)
    off = torch.zeros(n + 1, dtype=torch.int64, device=dev)
    torch.cumsum(deg + 1, dim=0, out=off[1:])
    m = int(off[-1])
    c = torch.complex(*torch.randn((2, m), generator=g, device=dev, dtype=torch.float64))
    ws = api.new_uneven_workspace(n, m, c.dtype, dev)
    d8 = deg.to(torch.uint8)
    want, want_st = api.roots_uneven(c, d8, off, ws, mode)
    want = torch.view_as_real(want).view(torch.int64).clone()
    got, st = api.roots_uneven(c, d8, off, ws, mode, roots=c[:m - n])
    assert torch.equal(torch.view_as_real(got).view(torch.int64), want) and torch.equal(st, want_st)
