"""The allocation-free entry point does its one-time work, for every D, in the
first call on a device: in a fresh process, after a call at D = 1 and after
each kernel has been loaded, a first call at another D allocates no host
memory either, and it can be captured."""
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CHILD = r"""
import ctypes, sys
import torch
sys.path.insert(0, {root!r})
from paper_1905_04582_gb300 import capi
lib = capi.lib()
libc = ctypes.CDLL(None)

class Mall(ctypes.Structure):
    _fields_ = [(k, ctypes.c_size_t) for k in
                ("arena", "ordblks", "smblks", "hblks", "hblkhd", "usmblks", "fsmblks", "uordblks", "fordblks",
                 "keepcost")]

libc.mallinfo2.restype = Mall
n = 90
data = {{}}
for d in range(1, 9):
    x = torch.randn(n, d, dtype=torch.float64, device="cuda")
    y = torch.cdist(x, x).float().contiguous()
    data[d] = (x, y, torch.empty_like(x), torch.empty_like(x))
torch.cuda.synchronize()
stream = torch.cuda.Stream()

def call(d, k, s):
    x, y, *g = data[d]
    capi.check(lib.mds_loglik_grad_noalloc(n, d, y.data_ptr(), n, x.data_ptr(), 0.5, g[k].data_ptr(), None, None, s))

call(1, 0, None)
torch.cuda.synchronize()
used = []
for d in (1, 1, 3, 7, 8):
    args = (n, d, data[d][1].data_ptr(), n, data[d][0].data_ptr(), 0.5, data[d][2].data_ptr(), None, None, None)
    before = libc.mallinfo2()
    st = lib.mds_loglik_grad_noalloc(*args)
    after = libc.mallinfo2()
    assert st == 0
    used.append((d, after.uordblks - before.uordblks))
torch.cuda.synchronize()
print("host bytes", used)
assert all(grown == 0 for _, grown in used), used
g = torch.cuda.CUDAGraph()
with torch.cuda.graph(g, stream=stream):
    for d in (2, 4, 5, 6):
        call(d, 0, stream.cuda_stream)
g.replay()
torch.cuda.synchronize()
for d in (2, 4, 5, 6):
    call(d, 1, None)
    torch.cuda.synchronize()
    assert torch.equal(data[d][2], data[d][3]) and bool(torch.isfinite(data[d][2]).all())
print("captured ok")
"""


def test_first_call_does_the_one_time_work():
    import os
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", CHILD.format(root=root)], capture_output=True, text=True, timeout=300)
    print(r.stdout)
    assert r.returncode == 0, r.stdout + r.stderr
    assert "captured ok" in r.stdout
