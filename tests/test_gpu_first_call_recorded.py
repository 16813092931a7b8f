"""The first attention call of a process, recorded into a graph: it draws its items from a counter like any later call."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CHILD = r"""
import ctypes
import torch
from paper_2410_23608_b200 import binding as L

class KernelParams(ctypes.Structure):
    _fields_ = [("func", ctypes.c_void_p), ("grid", ctypes.c_uint * 3), ("block", ctypes.c_uint * 3), ("smem", ctypes.c_uint),
                ("args", ctypes.POINTER(ctypes.c_void_p)), ("extra", ctypes.c_void_p), ("kern", ctypes.c_void_p), ("ctx", ctypes.c_void_p)]

B, N, H, d = 16, 1024, 8, 32                       # 128 row tiles x 8 heads: several items for every CTA
C, cap = H * d, B * N
p = L.make_params(B, N, C, H, "bf16", cap)
qkv = torch.randn(cap, 3 * C, device="cuda").bfloat16()
seg = torch.arange(0, cap + 1, N, dtype=torch.int32, device="cuda")
ao, lse = torch.empty(cap, C, device="cuda").bfloat16(), torch.empty(H, cap, device="cuda")
g = torch.cuda.CUDAGraph(keep_graph=True)
torch.cuda.synchronize()
with torch.cuda.graph(g):
    L.spa_packed_attention_fwd(p, qkv, seg, B, ao, lse)
cu = ctypes.CDLL("libcuda.so.1")          # the driver knows kernels of every runtime in the process
n = ctypes.c_size_t(0)
graph = ctypes.c_void_p(g.raw_cuda_graph())
assert cu.cuGraphGetNodes(graph, None, ctypes.byref(n)) == 0 and n.value == 1
node = (ctypes.c_void_p * 1)()
assert cu.cuGraphGetNodes(graph, node, ctypes.byref(n)) == 0
kp = KernelParams()
assert cu.cuGraphKernelNodeGetParams_v2(ctypes.c_void_p(node[0]), ctypes.byref(kp)) == 0
assert kp.block[0] == 288
pointer = lambda i: ctypes.cast(kp.args[i], ctypes.POINTER(ctypes.c_void_p))[0]
assert pointer(7) == ao.data_ptr()                 # tm, seg, n_seg, capacity, C, H, scale, ao, lse, counter
print("counter", "there" if pointer(9) else "missing")
g.instantiate()
g.replay()
torch.cuda.synchronize()
first = ao.clone()
L.spa_packed_attention_fwd(p, qkv, seg, B, ao, lse)
torch.cuda.synchronize()
assert torch.equal(ao, first)
"""


def test_first_call_recorded():
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    assert "counter there" in r.stdout
