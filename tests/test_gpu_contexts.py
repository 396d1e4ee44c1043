"""The library in more than one context of a device.  What a launch needs of the driver (a kernel's grant of more
than 48 KB of shared memory, how many clusters are resident) is asked for in every context anew: a context made after
the first call, and the primary context after a reset.  In a child process of its own, through the driver's API."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import ctypes
import sys

import numpy as np

import paper_2410_15704_b200 as rvq                    # (torch stays without a context here)

cu = ctypes.CDLL("libcuda.so.1")


def ask(name, *args):
    rc = getattr(cu, name)(*args)
    assert rc == 0, (name, rc)


def upload(a):
    p = ctypes.c_uint64()
    ask("cuMemAlloc_v2", ctypes.byref(p), ctypes.c_size_t(a.nbytes))
    ask("cuMemcpyHtoD_v2", p, a.ctypes.data_as(ctypes.c_void_p), ctypes.c_size_t(a.nbytes))
    return p.value


def download(p, nbytes):
    a = np.empty(nbytes, dtype=np.uint8)
    ask("cuMemcpyDtoH_v2", a.ctypes.data_as(ctypes.c_void_p), ctypes.c_uint64(p), ctypes.c_size_t(nbytes))
    return a


def run():
    # one call of each encoder and of the table decoder: all of them take more than 48 KB of shared memory
    out = []
    g = np.random.default_rng(3)
    for n, K, R in ((8, 1024, 8), (2000, 512, 2), (20000, 256, 1), (30000, 512, 8)):
        cfg = rvq.make_config(128, 32, 0, R, K, 16, rvq.F32, 0)
        c = ctypes.byref(cfg)
        cb = upload(g.normal(size=(R, K, 32)).astype(np.float32))
        x = upload(g.normal(size=(n, 128)).astype(np.float32))
        prepared = upload(np.zeros(rvq.rvq_prepared_bytes(cfg), dtype=np.uint8))
        codes, std = upload(np.zeros(n * rvq.rvq_code_bytes(cfg), dtype=np.uint8)), upload(np.zeros(n, dtype=np.uint16))
        assert rvq.lib.rvq_prepare_codebooks(c, cb, prepared, None) == 0
        rc = rvq.lib.rvq_encode(c, x, n, 128, cb, prepared, codes, std, None, None, 0, None, None)
        assert rc == 0, (n, K, rc)
        ask("cuCtxSynchronize")
        out.append(download(codes, n * rvq.rvq_code_bytes(cfg)))
        if R == 8 and n > 28672:
            half = rvq.make_config(128, 32, 0, R, K, 16, rvq.BF16, 0)
            back = upload(np.zeros(n * 128, dtype=np.uint16))
            rc = rvq.lib.rvq_decode(ctypes.byref(half), codes, std, n, cb, prepared, back, 128, None, None)
            assert rc == 0, ("decode", rc)
            ask("cuCtxSynchronize")
            out.append(download(back, n * 256))
    # the update whose scratch is an array of the library, one to a context (whole numbers: exact sums in any order)
    cfg = rvq.make_config(128, 32, 0, 1, 64, 16, rvq.F32, 0)
    x, codes = upload(np.tile(np.repeat(np.float32([1, -1]), 64), (500, 1))), upload((np.arange(2000) % 64).astype(np.uint16))
    cb, count, total = upload(np.ones((64, 32), np.float32)), upload(np.ones(64, np.float32)), upload(np.ones((64, 32), np.float32))
    for _ in range(2):
        rc = rvq.lib.rvq_ema_update_static(ctypes.byref(cfg), x, 500, 128, codes, cb, count, total, None, 0.5, 0.0, None, None)
        assert rc == 0, ("update", rc)
    ask("cuCtxSynchronize")
    return out + [download(cb, 64 * 32 * 4), download(count, 64 * 4), download(total, 64 * 32 * 4)]


device, primary, second = ctypes.c_int(), ctypes.c_void_p(), ctypes.c_void_p()
ask("cuInit", 0)
ask("cuDeviceGet", ctypes.byref(device), 0)
ask("cuDevicePrimaryCtxRetain", ctypes.byref(primary), device)
ask("cuCtxSetCurrent", primary)
want = run()


def check():
    for a, b in zip(want, run()):
        assert np.array_equal(a, b)


if sys.argv[1] == "second":
    ask("cuCtxCreate_v2", ctypes.byref(second), 0, device)
    check()
    ask("cuCtxSetCurrent", primary)
    check()
else:
    ask("cuCtxSetCurrent", None)
    ask("cuDevicePrimaryCtxReset_v2", device)
    ask("cuDevicePrimaryCtxRetain", ctypes.byref(primary), device)
    ask("cuCtxSetCurrent", primary)
    check()
print("same in both")
"""


@pytest.mark.parametrize("how", ["second", "reset"])
def test_calls_in_a_new_context(how):
    env = dict(os.environ, PYTHONPATH=ROOT)
    p = subprocess.run([sys.executable, "-c", CHILD, how], cwd=ROOT, env=env, capture_output=True, text=True, timeout=300)
    assert p.returncode == 0 and "same in both" in p.stdout, p.stderr[-2000:]
