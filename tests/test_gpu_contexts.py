"""The library in a second context of a device and in the context behind a reset: in a process of its own, on the
driver API alone, without another library's runtime."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import ctypes as C
import sys

import numpy as np

from paper_2609_15810_b200.binding import Params
import paper_2609_15810_b200 as vc

cu, lib = C.CDLL("libcuda.so.1"), vc.load_library()


def ck(r):
    assert r == 0, r


def attn(bits):
    # one call on buffers of the current context; its output
    N, H, d = 1024, 2, 128
    rng = np.random.default_rng(1)
    p = Params.make(1, H, N, d, (4, 16, 16), bits=bits)

    def alloc(n):
        a = C.c_uint64()
        ck(cu.cuMemAlloc_v2(C.byref(a), C.c_size_t(n)))
        return a.value
    host = [(rng.standard_normal(H * N * d).astype(np.float32).view(np.uint32) >> 16).astype(np.uint16) for _ in range(3)]
    dev = [alloc(x.nbytes) for x in host]
    for a, x in zip(dev, host):
        ck(cu.cuMemcpyHtoD_v2(C.c_uint64(a), x.ctypes.data_as(C.c_void_p), C.c_size_t(x.nbytes)))
    o, quant, work = alloc(host[0].nbytes), alloc(vc.vc_quant_bytes(p)), alloc(vc.vc_workspace_bytes(p))
    ck(lib.vc_attn(C.byref(p), *dev, None, o, quant, work, None))
    ck(lib.vc_poll_status(work, None))
    out = np.empty_like(host[0])
    ck(cu.cuMemcpyDtoH_v2(out.ctypes.data_as(C.c_void_p), C.c_uint64(o), C.c_size_t(out.nbytes)))
    for a in dev + [o, quant, work]:
        ck(cu.cuMemFree_v2(C.c_uint64(a)))
    return out


ck(cu.cuInit(0))
dev, primary, second = C.c_int(), C.c_void_p(), C.c_void_p()
ck(cu.cuDeviceGet(C.byref(dev), 0))
ck(cu.cuDevicePrimaryCtxRetain(C.byref(primary), dev))
ck(cu.cuCtxSetCurrent(primary))
first = [attn(8), attn(4)]
if sys.argv[1] == "second":
    ck(cu.cuCtxCreate_v2(C.byref(second), 0, dev))
    assert all(np.array_equal(a, b) for a, b in zip(first, [attn(8), attn(4)]))
    ck(cu.cuCtxSetCurrent(primary))
else:
    ck(cu.cuDevicePrimaryCtxReset_v2(dev))
    ck(cu.cuDevicePrimaryCtxRetain(C.byref(primary), dev))
    ck(cu.cuCtxSetCurrent(primary))
assert all(np.array_equal(a, b) for a, b in zip(first, [attn(8), attn(4)]))
print("CONTEXTS OK")
"""


@pytest.mark.gpu
@pytest.mark.parametrize("what", ["second", "reset"])
def test_library_in_another_context(what):
    r = subprocess.run([sys.executable, "-c", CHILD, what], cwd=ROOT, env=dict(os.environ, PYTHONPATH=ROOT), capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "CONTEXTS OK" in r.stdout, r.stdout + r.stderr
