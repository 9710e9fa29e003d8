"""The first tensor-copy launches of a process, made by several host threads at once:
every one finds the driver's encoder (a process of its own per attempt, since only its
first calls look it up)."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

pytestmark = pytest.mark.gpu

CHILD = r"""
import ctypes as C, sys, threading
import torch
from paper_2010_00409_gb300 import psatd
L = psatd.lib()
A = torch.randn((128, 64), device="cuda").to(torch.bfloat16)
B = torch.randn((256, 64), device="cuda").to(torch.bfloat16)
out = [torch.empty((128, 256), device="cuda") for _ in range(8)]
torch.cuda.synchronize()
sys.setswitchinterval(1e-6)
status, go = [None] * 8, threading.Barrier(8)
args = [(128, 256, 64, C.c_void_p(A.data_ptr()), C.c_void_p(B.data_ptr()), C.c_void_p(o.data_ptr()), None) for o in out]

def body(i):
    go.wait()
    status[i] = L.psatd_gemm_bf16_tma(*args[i])

threads = [threading.Thread(target=body, args=(i,)) for i in range(8)]
for t in threads:
    t.start()
for t in threads:
    t.join()
torch.cuda.synchronize()
ref = A.float() @ B.float().t()
assert status == [0] * 8, status
assert all(torch.allclose(o, ref, rtol=1e-3, atol=1e-3) for o in out)
"""


@pytest.mark.parametrize("attempt", range(3))
def test_first_tensor_copy_launches(lib, attempt):
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
