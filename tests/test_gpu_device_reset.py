"""Calls after a cudaDeviceReset, which ends the process's own context: kernel
attributes, streams and events made before it are gone. A child process without
other users of the context solves, resets, and solves again."""
from __future__ import annotations

import os
import subprocess
import sys

import pytest

from tests.gpu_common import require_gpu

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import ctypes as C, sys
import numpy as np
from paper_2507_02164_gb300 import _native as N

L = N.load()
R = C.CDLL("libcudart.so.13")  # the one that libroots.so is linked against
P = C.c_void_p


def ok(rc):
    assert rc == 0, (rc, L.rd_last_error().decode())


def dev(host=None, nbytes=0):
    p = P()
    ok(R.cudaMalloc(C.byref(p), C.c_size_t(host.nbytes if host is not None else nbytes)))
    if host is not None:
        ok(R.cudaMemcpy(p, P(host.ctypes.data), C.c_size_t(host.nbytes), 1))
    return p


def back(p, shape, dtype):
    out = np.empty(shape, dtype)
    ok(R.cudaMemcpy(P(out.ctypes.data), p, C.c_size_t(out.nbytes), 2))
    return out


def uniform(degree, n, **kw):
    rng = np.random.default_rng(degree)
    c = (rng.standard_normal((degree + 1, n)) + 1j * rng.standard_normal((degree + 1, n))).astype(np.complex64)
    prm = N.default_params(N.MIXED)
    for k, v in kw.items():
        setattr(prm, k, v)
    z, st = dev(nbytes=16 * degree * n), dev(nbytes=n)
    ok(L.rd_roots_batched(dev(c), N.C64, degree, n, N.MIXED, C.byref(prm), z, st, None, None))
    ok(R.cudaDeviceSynchronize())
    return back(z, (degree, 2 * n), np.int64), back(st, (n,), np.uint8)


def packed(n, stream=None, tuning=None):
    rng = np.random.default_rng(n)
    deg = rng.integers(2, 13, n)
    off = np.concatenate([[0], np.cumsum(deg + 1)]).astype(np.int64)
    m = int(off[-1])
    c = (rng.standard_normal(m) + 1j * rng.standard_normal(m)).astype(np.complex64)
    b = L.rd_uneven_workspace_bytes(n, m, N.C64)
    args = [dev(c), N.C64, dev(deg.astype(np.uint8)), dev(off), n, m, N.MIXED, None, tuning, None, 0, 0, None,
            dev(nbytes=16 * (m - n)), dev(nbytes=n), None, dev(nbytes=b), b]
    return args, m - n


def packed_roots(n, tuning=None):
    args, m = packed(n, tuning=tuning)
    ok(L.rd_roots_uneven(*args, None))
    ok(R.cudaDeviceSynchronize())
    return back(args[13], (m, 2), np.int64), back(args[14], (n,), np.uint8)


def captured(n):
    # the whole call in a graph, replayed once
    st, graph, ex = P(), P(), P()
    ok(R.cudaStreamCreate(C.byref(st)))
    args, m = packed(n)
    ok(R.cudaStreamBeginCapture(st, 2))
    rc = L.rd_roots_uneven(*args, st)
    ok(R.cudaStreamEndCapture(st, C.byref(graph)))
    ok(rc)
    ok(R.cudaGraphInstantiate(C.byref(ex), graph, C.c_ulonglong(0)))
    ok(R.cudaGraphLaunch(ex, st))
    ok(R.cudaStreamSynchronize(st))
    return back(args[13], (m, 2), np.int64), back(args[14], (n,), np.uint8)


sms = L.rd_device_sm_count()
tuning = N.UnevenTuning()
for d in range(1, 9):
    tuning.block[d], tuning.polish_warps[d] = (512, 10) if d <= 6 else (256, 4)
CALLS = {
    "open": [lambda: uniform(6, 600 * sms), lambda: uniform(12, 240 * sms), lambda: uniform(9, 300 * sms, polish_mode=1)],
    "packed": [lambda: packed_roots(6200 * sms)],
    "explicit": [lambda: uniform(6, 5000, block=512, polish_warps=10), lambda: packed_roots(40000, C.byref(tuning))],
    # a small call first, as every host thread's first call on a device is to be outside capture
    "captured": [lambda: packed_roots(500), lambda: captured(200 * sms)],
}[sys.argv[1]]
before = [f() for f in CALLS]
ok(R.cudaDeviceReset())
for f, want in zip(CALLS, before):
    got = f()
    assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])
print("same after the reset")
"""


@pytest.mark.parametrize("calls", ["open", "packed", "explicit", "captured"])
def test_the_same_results_after_a_reset(calls):
    require_gpu()
    r = subprocess.run([sys.executable, "-c", CHILD, calls], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "same after the reset" in r.stdout, r.stdout + r.stderr
