"""What a call needs to find in place, in processes of their own: the first call under stream capture, calls in a second
context of the device, and after the first one was reset."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

COMMON = """
import sys
sys.path[:0] = [{root!r}, {root!r} + "/tests"]
import numpy as np
"""

CAPTURED = """
import torch
from test_attention_gpu import Case
from paper_2304_01089_b200 import binding
c = Case(80, H=2, hd=64, gh=4, Tq={tq}, Tk=64)
out = torch.full((c.Tq, 128), float("nan"), dtype=torch.float16, device="cuda")
q16 = torch.randn((c.Tq, 128), device="cuda").half()
def call():
    if {kv}:
        binding.attention_kv(c.LK, c.LV, 2, q16, c.dk, c.dv, out, c.qk_scale, True)
    else:
        binding.attention(c.LQ, c.LK, c.LV, 2, c.dq, c.dk, c.dv, out, c.s_P, c.qk_scale, True)
g = torch.cuda.CUDAGraph()
with torch.cuda.graph(g):
    call()
g.replay()
first = out.clone()
out.fill_(float("nan"))
call()
torch.cuda.synchronize()
assert not torch.isnan(first).any() and torch.equal(first, out)
assert binding.get_device_status() == 0
print("done")
"""


def _run(script, **fields):
    r = subprocess.run([sys.executable, "-c", (COMMON + script).format(root=ROOT, **fields)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "done" in r.stdout, r.stdout[-1000:] + r.stderr[-3000:]


@pytest.mark.parametrize("kv,tq", [(False, 64), (True, 64), (True, 1)])
def test_first_attention_call_of_a_process_can_be_captured(kv, tq):
    _run(CAPTURED, kv=kv, tq=tq)


# Every kind of kernel that asks for more shared memory than the default, through plain ctypes: no tensor library, whose memory
# belongs to the device's primary context.
CONTEXTS = """
import ctypes as C
import oracle
from helpers import random_layout_params
from paper_2304_01089_b200 import binding
cu, lib = C.CDLL("libcuda.so.1"), binding._lib
def ck(status):
    assert status == 0, status
def once():
    rng = np.random.default_rng(0)
    M, N = 200, 512
    perm, size, scale, zero = random_layout_params(rng, 256, 2, 4, allow_empty=False)
    perm, size = np.arange(256, dtype=np.int32), np.array([128, 128], np.int32)          # two heads of 128 channels
    L = binding.Layout(perm, size, scale, zero, 4)
    bufs = []
    def up(a):
        a, p = np.ascontiguousarray(a), C.c_void_p()
        ck(cu.cuMemAlloc_v2(C.byref(p), C.c_size_t(a.nbytes)))
        ck(cu.cuMemcpyHtoD_v2(p, a.ctypes.data_as(C.c_void_p), C.c_size_t(a.nbytes)))
        bufs.append((p, a.shape, a.dtype))
        return p
    def down(p):
        shape, dtype = [(s, d) for q, s, d in bufs if q is p][0]
        a = np.empty(shape, dtype)
        ck(cu.cuCtxSynchronize())
        ck(cu.cuMemcpyDtoH_v2(a.ctypes.data_as(C.c_void_p), p, C.c_size_t(a.nbytes)))
        return a
    x, ln = up(rng.normal(size=(M, 256)).astype(np.float16)), up(np.ones(256, np.float16))
    codes, codes8 = up(np.zeros((M, L.row_bytes), np.uint8)), up(np.zeros((8, L.row_bytes), np.uint8))
    w, s_w, wsum = binding.weight_pack(L, rng.normal(size=(N, 256)).astype(np.float32))
    dw, ds, dws = up(w), up(s_w), up(wsum)
    y, y8 = up(np.zeros((M, N), np.float32)), up(np.zeros((8, N), np.float32))
    ck(lib.rptq_ln_reorder_quant(L.handle, x, 256, ln, ln, 1e-5, M, codes, None, None))
    ck(lib.rptq_ln_reorder_quant(L.handle, x, 256, ln, ln, 1e-5, 8, codes8, None, None))
    ck(lib.rptq_cluster_gemm(L.handle, codes, M, dw, ds, dws, wsum.shape[1], None, N, 0, None, y, 0, N, None))
    ck(lib.rptq_cluster_gemm(L.handle, codes8, 8, dw, ds, dws, wsum.shape[1], None, N, 0, None, y8, 0, N, None))
    y_na = up(np.zeros((M, N), np.float32))
    ck(lib.rptq_cluster_gemm_noalloc(L.handle, codes, M, dw, ds, dws, wsum.shape[1], None, N, 0, None, y_na, 0, N, None))
    status = C.c_int(1)
    ck(lib.rptq_get_device_status(C.byref(status)))
    assert status.value == 0
    o, o8 = up(np.zeros((M, 256), np.float16)), up(np.zeros((4, 256), np.float16))
    ck(lib.rptq_attention(L.handle, L.handle, L.handle, 2, codes, M, codes, codes, M, 1, 1 / 256, 0, 0.05, 1, o, 256, None, None))
    ck(lib.rptq_attention(L.handle, L.handle, L.handle, 2, codes8, 4, codes, codes, M, 1, 1 / 256, 0, 0.05, 1, o8, 256, None, None))
    return [down(p) for p in (codes, y, y8, y_na, o, o8)]
ck(cu.cuInit(0))
dev, ctx = C.c_int(), C.c_void_p()
ck(cu.cuDeviceGet(C.byref(dev), 0))
results = []
if {reset}:
    for i in range(2):
        ck(cu.cuDevicePrimaryCtxRetain(C.byref(ctx), dev))
        ck(cu.cuCtxSetCurrent(ctx))
        results.append(once())
        if i == 0:
            ck(cu.cuDevicePrimaryCtxReset_v2(dev))           # ends this process's own context of the device
else:
    for i in range(2):
        ck(cu.cuCtxCreate_v2(C.byref(ctx), 0, dev))          # current from here on
        results.append(once())
for a, b in zip(*results):
    assert np.array_equal(a, b) and a.any()
print("done")
"""


@pytest.mark.parametrize("reset", [False, True])
def test_every_context_of_a_device_can_call(reset):
    _run(CONTEXTS, reset=reset)
