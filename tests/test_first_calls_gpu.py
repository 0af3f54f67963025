"""What a call needs to find in place, in processes of their own: the first call under stream capture."""
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
