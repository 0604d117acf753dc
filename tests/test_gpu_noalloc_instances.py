"""sg_direct_noalloc allocates nothing after its first call in a context, whatever
grid or dtype the later calls have: the first call loads the kernels of all of
them (CUDA loads a kernel at its first use, into device memory).  In a process of its
own, which has launched none of them before."""
import os
import subprocess
import sys

import pytest

from paper_2506_10812_gb300 import build as B

pytestmark = pytest.mark.gpu
ROOT = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..")

CHILD = """
import ctypes, torch
from paper_2506_10812_gb300 import _native as N
lib, dev = N.load(), torch.device("cuda:0")
f, d = torch.float32, torch.float64
grids = [(16, 32, f), (16, 4, f), (45, 521, f), (162, 326, f), (16, 4, d), (64, 64, d), (8, 326, d)]
bufs = [(torch.ones(g[:2], dtype=g[2], device=dev), torch.zeros(g[:2], dtype=g[2], device=dev)) for g in grids]
def call(k):
    nr, nphi, dt = grids[k]
    p = N.SgParams()
    p.nr, p.nphi, p.r_in, p.r_out, p.h_g, p.h_d, p.G = nr, nphi, 0.2, 2.5, 0.05, 0.0, 1.0
    p.dtype, p.method = N.SG_F64 if dt == d else N.SG_F32, N.SG_METHOD_DIRECT
    x, o = bufs[k]
    st = lib.sg_direct_noalloc(ctypes.byref(p), x.data_ptr(), None, o.data_ptr(), None, None, None, None, None, None)
    torch.cuda.synchronize()
    assert st == N.SG_OK and bool(torch.isfinite(o).all()) and float(o.abs().min()) > 0
torch.cuda.synchronize()
call(0)
free = torch.cuda.mem_get_info(dev)[0]
for k in range(1, len(grids)):
    call(k)
    print(grids[k], torch.cuda.mem_get_info(dev)[0] - free)
assert torch.cuda.mem_get_info(dev)[0] == free
"""


def test_later_calls_allocate_nothing(cuda_device):
    B.build()
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
