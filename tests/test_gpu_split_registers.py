"""A compiler that gives a split kernel another register count than its roles'
shares were added up for: the kernel is not launched (a share above what the
launch holds would wait forever), and the call takes the one-role kernel, whose
results are the same bits. The count is faked on the host: a shim in front of
the CUDA runtime's query reports eight registers more."""
from __future__ import annotations

import os
import shutil
import subprocess
import sys

import pytest

from tests.gpu_common import require_gpu

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SHIM = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
#include <stdio.h>
#include <cuda_runtime_api.h>
cudaError_t cudaFuncGetAttributes(struct cudaFuncAttributes *attr, const void *func)
{
    static cudaError_t (*real)(struct cudaFuncAttributes *, const void *);
    if (!real) real = (cudaError_t(*)(struct cudaFuncAttributes *, const void *))dlsym(RTLD_NEXT, "cudaFuncGetAttributes");
    cudaError_t e = real(attr, func);
    if (e == cudaSuccess) {
        attr->numRegs += 8;
        fputs("asked\n", stderr);
    }
    return e;
}
"""

CHILD = r"""
import torch
from paper_2507_02164_gb300 import api

dev = torch.device("cuda:0")
sms = torch.cuda.get_device_properties(dev).multi_processor_count
bits = lambda z: torch.view_as_real(z).view(torch.int64)
for degree, n, kw in ((6, 600 * sms + 5, {}), (9, 300 * sms, {"polish_mode": "df"})):
    c = torch.complex(*torch.randn((2, degree + 1, n), device=dev))
    a, b = (api.roots_batched(c, "mixed", api.params("mixed", **kw, **shape)) for shape in ({}, {"block": 128}))
    assert torch.equal(bits(a[0]), bits(b[0])) and torch.equal(a[1], b[1])
n = 6200 * sms
deg = 2 + torch.arange(n, device=dev) % 11
off = torch.zeros(n + 1, dtype=torch.int64, device=dev)
torch.cumsum(deg + 1, dim=0, out=off[1:])
c = torch.complex(*torch.randn((2, int(off[-1])), device=dev))
ws = api.new_uneven_workspace(n, c.numel(), c.dtype, dev)
a, b = (api.roots_uneven(c, deg.to(torch.uint8), off, ws, "mixed", api.params("mixed", **kw)) for kw in ({}, {"block": 128}))
assert torch.equal(bits(a[0]), bits(b[0])) and torch.equal(a[1], b[1])
print("served")
"""


def test_another_register_count_is_served_by_the_one_role_kernel(tmp_path):
    require_gpu()
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    home = os.path.dirname(os.path.dirname(os.path.realpath(nvcc)))
    src, lib = tmp_path / "shim.c", tmp_path / "shim.so"
    src.write_text(SHIM)
    subprocess.run(["gcc", "-shared", "-fPIC", "-O1", "-I", os.path.join(home, "include"), "-o", str(lib), str(src), "-ldl"],
                   check=True)
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, capture_output=True, text=True, timeout=300,
                       env=dict(os.environ, LD_PRELOAD=str(lib)))
    assert r.returncode == 0 and "served" in r.stdout, r.stdout + r.stderr
    assert "asked" in r.stderr  # the shim was in the way
