"""The first decompressions of a process, many threads at once on streams of their own: each
launch finds the shared memory its kernel needs allowed, whichever thread came first."""
import subprocess
import sys

import pytest
import torch

pytestmark = pytest.mark.gpu

CHILD = r"""
import ctypes as C, sys, threading
import torch
from paper_2105_12912_gb300 import _lib, api
sys.setswitchinterval(1e-5)
x = torch.cumsum(torch.randn((48, 48, 48), generator=torch.Generator().manual_seed(1)), -1)
x[:16] = 0
x = x.cuda()
# (run books: more shared memory than a kernel gets without asking)
ar, nb, _ = api.compress(x, 1e-2, select="rle_huff")
n = 24
go = threading.Barrier(n)
outs = [torch.empty_like(x) for _ in range(n)]
wss = [torch.empty(api.workspace_bytes(tuple(x.shape)), dtype=torch.uint8, device="cuda") for _ in range(n)]
streams = [torch.cuda.Stream() for _ in range(n)]
res = [None] * n
torch.cuda.synchronize()
fn = _lib.lib().csz_decompress
args = [(C.c_void_p(ar.data_ptr()), nb, C.c_void_p(o.data_ptr()), o.numel(), C.c_void_p(w.data_ptr()), w.numel(),
         C.c_void_p(s.cuda_stream)) for o, w, s in zip(outs, wss, streams)]
def work(i):
    a = args[i]
    go.wait()
    res[i] = fn(*a)
ts = [threading.Thread(target=work, args=(i,)) for i in range(n)]
[t.start() for t in ts]
[t.join() for t in ts]
torch.cuda.synchronize()
assert res == [0] * n, res
want, _ = api.decompress(ar, nb)
assert all(torch.equal(o, want) for o in outs)
"""


@pytest.mark.parametrize("turn", range(4))
def test_first_calls_of_many_threads(turn):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    r = subprocess.run([sys.executable, "-c", CHILD], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
