"""The entry points in contexts other than the device's primary one, in processes of their own."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SECOND_CONTEXT = r"""
import ctypes as C
import numpy as np, torch
from paper_2604_03260_b200 import binding as fb
H, n, D, K = 8, 2000, 128, 4
x = torch.randn((1, H, n, D), device="cuda").to(torch.bfloat16)
c = torch.randn((H, K, D), device="cuda")
m = torch.empty((H, n), dtype=torch.int32, device="cuda")
shape = fb.make_shape(H, H, n, D, K, 2, 16)
fb.focus_assign(shape, x, H, c, m)                     # the kernel's attributes are set in the primary context
torch.cuda.synchronize()
xh, ch, want = x.view(torch.int16).cpu().numpy(), c.cpu().numpy(), m.cpu().numpy()
cu = C.CDLL("libcuda.so.1")
def ok(r):
    assert r == 0, r
primary, dev = C.c_void_p(), C.c_int()
ok(cu.cuCtxGetCurrent(C.byref(primary)))
ok(cu.cuDeviceGet(C.byref(dev), 0))
def up(a):
    p = C.c_uint64()
    ok(cu.cuMemAlloc_v2(C.byref(p), C.c_size_t(a.nbytes)))
    ok(cu.cuMemcpyHtoD_v2(p, a.ctypes.data_as(C.c_void_p), C.c_size_t(a.nbytes)))
    return p
for _ in range(2):                                     # a context, and another after it is gone
    ctx = C.c_void_p()
    ok(cu.cuCtxCreate_v2(C.byref(ctx), 0, dev))
    got = np.zeros_like(want)
    px, pc, pm = up(xh), up(ch), up(got)
    rc = fb.lib().focus_assign(C.byref(shape), fb.focus_tensor(px.value, H * n * D, n * D, D), H, pc.value, pm.value, None, 1e-5, None)
    assert rc == 0, fb.lib().focus_last_error()
    ok(cu.cuCtxSynchronize())
    ok(cu.cuMemcpyDtoH_v2(got.ctypes.data_as(C.c_void_p), pm, C.c_size_t(got.nbytes)))
    assert (got == want).all()
    ok(cu.cuCtxDestroy_v2(ctx))
ok(cu.cuCtxSetCurrent(primary))
m.zero_()
fb.focus_assign(shape, x, H, c, m)
assert (m.cpu().numpy() == want).all()
print("done")
"""


PARTITION = r"""
import torch
from paper_2604_03260_b200 import binding as fb
from torch.cuda import green_contexts
n, K, iters = 131072, 8, 5
S, dg = 0.3 * torch.randn((1, n, K), device="cuda"), torch.randn((1, n, K), device="cuda")
shape = fb.make_shape(4, 2, n, 128, K, 1, 16)
ws = torch.empty(fb.focus_sinkhorn_workspace_bytes(shape, iters), dtype=torch.uint8, device="cuda")
wb = torch.empty(fb.focus_sinkhorn_bwd_workspace_bytes(shape, iters), dtype=torch.uint8, device="cuda")
def both():
    g, ds = torch.empty_like(S), torch.empty_like(S)
    fb.focus_sinkhorn(shape, S, 0.1, iters, ws, g)
    fb.focus_sinkhorn_bwd(shape, S, 0.1, iters, wb, dg, ds)
    torch.cuda.synchronize()
    return g, ds
want = both()
part = green_contexts.GreenContext.create(num_sms=24, device_id=0)
part.set_context()
got = both()
graph, replayed = torch.cuda.CUDAGraph(), torch.zeros_like(S)
with torch.cuda.graph(graph, stream=torch.cuda.Stream()):
    fb.focus_sinkhorn(shape, S, 0.1, iters, ws, replayed)
graph.replay()
torch.cuda.synchronize()
part.pop_context()
for a, b in zip(got + (replayed,), want + want[:1]):
    assert (a - b).abs().max() <= 2e-4 * b.abs().max(), (a - b).abs().max()
again = both()                                         # no error is left behind
assert torch.equal(again[0], want[0]) and torch.equal(again[1], want[1])
print("done")
"""


def run(code):
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True, timeout=240)
    assert r.returncode == 0 and "done" in r.stdout, r.stdout[-1000:] + r.stderr[-2000:]


def test_second_context_on_the_device():
    run(SECOND_CONTEXT)


def test_partition_of_the_multiprocessors():
    """24 multiprocessors do not hold the blocks of a long Sinkhorn call at once: a launch per iteration instead"""
    pytest.importorskip("torch.cuda.green_contexts")
    run(PARTITION)
