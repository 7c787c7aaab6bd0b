"""What the library keeps in the process between uploads, against what a process may do in between (needs
a B200): trim, contexts of the driver API, a reset of the device's primary context.  Own processes,
without torch: they call the C ABI and the driver."""
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

PROGRAM = r'''
import ctypes, sys, threading
import numpy as np
from paper_2607_08786_b200 import tl3, workloads as wl
cu = ctypes.CDLL("libcuda.so.1")
vp, u64 = ctypes.c_void_p, ctypes.c_uint64
def ck(rc, what):
    assert rc == 0, (what, rc)
ck(cu.cuInit(0), "init")
def primary():
    ctx = vp()
    ck(cu.cuDevicePrimaryCtxRetain(ctypes.byref(ctx), 0), "retain")
    ck(cu.cuCtxSetCurrent(ctx), "current")
def upload(data, want):
    m = tl3.Matrix.deserialize(data)
    d = u64()
    L = tl3.lib()
    assert L.tl3_plan_device(m._h, None) == 0, L.tl3_last_cuda_error()
    ck(cu.cuMemAlloc_v2(ctypes.byref(d), ctypes.c_size_t(m.device_bytes())), "alloc")
    rc = L.tl3_upload_device(m._h, vp(d.value), None)
    assert rc == 0, (rc, L.tl3_last_cuda_error())
    got = np.empty(want.size, dtype=np.uint8)
    ck(cu.cuMemcpyDtoH_v2(got.ctypes.data_as(vp), d, ctypes.c_size_t(got.size)), "copy")
    ck(cu.cuMemFree_v2(d), "free")
    assert np.array_equal(got, want)
def download(data, want):
    d, h = u64(), vp()
    ck(cu.cuMemAlloc_v2(ctypes.byref(d), ctypes.c_size_t(W.nbytes)), "alloc")
    ck(cu.cuMemcpyHtoD_v2(d, W.ctypes.data_as(vp), ctypes.c_size_t(W.nbytes)), "copy")
    rc = tl3.lib().tl3_encode_device(vp(d.value), 4096, 2048, 2048, None, ctypes.byref(h))
    assert rc == 0, (rc, tl3.lib().tl3_last_cuda_error())
    ck(cu.cuMemFree_v2(d), "free")
    assert tl3.Matrix(h.value).serialize() == data
W = wl.Case(0, "state", 4096, 2048, 8, 5, 0.5, "bernoulli").make_W()
m = tl3.encode(W)
data, want = m.serialize(), m.pack()
if sys.argv[2] == "down":
    upload = download
assert len(data) > 9 << 20                                   # beyond the size from which the pinned memory is used
primary()
upload(data, want)
what = sys.argv[1]
if what == "trim":
    for _ in range(3):
        tl3.trim()
        upload(data, want)
    tl3.trim()
    tl3.trim()
    stop = threading.Event()
    def trimmer():
        while not stop.is_set():
            tl3.trim()
    t = threading.Thread(target=trimmer)
    t.start()
    try:
        for _ in range(10):
            upload(data, want)
    finally:
        stop.set()
        t.join()
elif what == "context":
    ctx = vp()
    ck(cu.cuCtxCreate_v2(ctypes.byref(ctx), 0, 0), "create")
    upload(data, want)
    ck(cu.cuCtxPopCurrent_v2(ctypes.byref(vp())), "pop")
    upload(data, want)
elif what == "reset":
    ck(cu.cuDevicePrimaryCtxReset_v2(0), "reset")
    primary()
    upload(data, want)
print("done")
'''


@pytest.mark.parametrize("what", ["trim", "context", "reset"])
def test_uploads_around(what):
    res = subprocess.run([sys.executable, "-c", PROGRAM, what, "up"], capture_output=True, text=True, timeout=300)
    assert res.returncode == 0 and res.stdout.endswith("done\n"), res.stdout + res.stderr[-2000:]


@pytest.mark.parametrize("what", ["trim", "context", "reset"])
def test_downloads_around(what):
    """The same for containers that come from the device."""
    res = subprocess.run([sys.executable, "-c", PROGRAM, what, "down"], capture_output=True, text=True, timeout=300)
    assert res.returncode == 0 and res.stdout.endswith("done\n"), res.stdout + res.stderr[-2000:]
