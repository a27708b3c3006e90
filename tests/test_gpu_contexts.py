"""Plans of several CUDA contexts on one device: what the library keeps between plans (device blocks, a stream, the kernels'
shared-memory opt-in) belongs to the context it was made in.  The contexts are made through the driver in a process of its
own, without torch, which knows the primary context only."""
import os
import subprocess
import sys

import pytest

from paper_2602_21788_b200 import build

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import ctypes as C
import numpy as np
from paper_2602_21788_b200 import fcp
cu = C.CDLL("libcuda.so.1")
def ok(r):
    assert r == 0, r
ok(cu.cuInit(0))
dev = C.c_int()
ok(cu.cuDeviceGet(C.byref(dev), 0))
def context():
    ctx = C.c_void_p()
    ok(cu.cuCtxCreate_v2(C.byref(ctx), 0, dev))          # becomes current
    return ctx
def to_dev(a):
    p = C.c_uint64()
    ok(cu.cuMemAlloc_v2(C.byref(p), C.c_size_t(a.nbytes)))
    ok(cu.cuMemcpyHtoD_v2(p, a.ctypes.data_as(C.c_void_p), C.c_size_t(a.nbytes)))
    return p
def one_plan(lens):
    rng = np.random.default_rng(3)
    T, hq, hkv, D = sum(lens), 4, 2, 64
    bits = lambda h: (rng.standard_normal((T, h, D), dtype=np.float32).view(np.uint32) >> 16).astype(np.uint16)
    q, k, v = to_dev(bits(hq)), to_dev(bits(hkv)), to_dev(bits(hkv))
    o, lse = np.zeros((T, hq, D), np.uint16), np.zeros((T, hq), np.float32)
    od, ld = to_dev(o), to_dev(lse)
    plan = fcp.Plan(lens, [1] * len(lens), hq, hkv, D).upload()
    fcp.fcp_attn_fwd_fused(plan, q.value, k.value, v.value, od.value, ld.value)
    ok(cu.cuCtxSynchronize())
    assert plan.device_status()[0] == 0
    ok(cu.cuMemcpyDtoH_v2(o.ctypes.data_as(C.c_void_p), od, C.c_size_t(o.nbytes)))
    ok(cu.cuMemcpyDtoH_v2(lse.ctypes.data_as(C.c_void_p), ld, C.c_size_t(lse.nbytes)))
    assert np.isfinite(lse).all() and o.any()
    return o, lse                                        # the plan goes: its block stays with this context
lens = [700, 130, 1]
a = context()
first = one_plan(lens)
b = context()
second = one_plan(lens)                                  # must not get a block or a stream of the first context
ok(cu.cuCtxSetCurrent(a))
third = one_plan(lens)                                   # back again
ok(cu.cuCtxSetCurrent(b))
ok(cu.cuCtxDestroy_v2(b))
c = context()
fourth = one_plan(lens)                                  # what the destroyed context held is not used
fcp.fcp_release_cached()
for x in (second, third, fourth):
    assert np.array_equal(x[0], first[0]) and np.array_equal(x[1], first[1])
print("contexts ok")
"""


def test_plans_in_several_contexts_of_one_device():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and "contexts ok" in r.stdout, r.stdout + r.stderr
