"""The short calls through csrc/marshal.cpp and through ctypes: the same results, the same errors."""
import os
import shutil
import subprocess
import sys

import pytest
import torch

from paper_2604_03260_b200 import binding as fb
from paper_2604_03260_b200 import inputs as fi

pytestmark = pytest.mark.gpu


class NotRead:
    """in the place of the module: no argument is of the usual kind"""
    def __getattr__(self, name):
        return lambda *args: None


@pytest.fixture(autouse=True)
def loaded():
    """Loading puts the module in its place: before a test puts another there, and so that it is put back afterwards."""
    fb.lib()
    assert fb._marshal is not fb._Ctypes


class Sub(torch.Tensor):
    pass


def run(wl, wrap, batch, stream=None, eps=1e-5):
    """assign -> build_tiles -> attn_fwd, a decode step, and the router, with tensors passed through `wrap`"""
    dev = "cuda"
    shape = fb.make_shape(wl.Hq, wl.Hkv, wl.n, wl.D, wl.K, wl.topk, wl.window, batch=batch)
    Q, K, V, C = fi.make_inputs(wl, dev)
    if batch > 1:
        Q, K, V = (torch.stack([x] + [x.flip(1)] * (batch - 1)) for x in (Q, K, V))
    K = torch.cat([K, K], dim=-2)[..., :wl.n, :]                # head stride other than n * D
    mq, mk = (torch.zeros((batch * h, wl.n), dtype=torch.int32, device=dev) for h in (wl.Hq, wl.Hkv))
    near = torch.zeros(1, dtype=torch.int64, device=dev)
    fb.focus_assign(shape, wrap(Q), wl.Hq, wrap(C), wrap(mq), wrap(near), eps, stream)
    fb.focus_assign(shape, wrap(K), wl.Hkv, C, mk, stream=stream)
    ws = fb.alloc_workspace(shape, 0)
    fb.focus_build_tiles(shape, wrap(mq), mk, 0, wrap(ws), stream)
    O, lse, status = torch.zeros_like(Q), torch.zeros((batch * wl.Hq, wl.n), device=dev), torch.zeros(4, dtype=torch.int32, device=dev)
    fb.focus_attn_fwd(shape, wrap(Q), wrap(K), wrap(V), mq, mk, ws, 0, wrap(O), lse, status, stream)
    q1 = Q[..., -1, :]
    o1, l1 = torch.zeros(q1.shape, dtype=torch.bfloat16, device=dev), torch.zeros(batch * wl.Hq, device=dev)
    wd = torch.zeros(fb.focus_decode_workspace_bytes(shape), dtype=torch.uint8, device=dev)
    fb.focus_decode_step(shape, wrap(q1), K, V, mq[:, -1].contiguous(), mk, wrap(o1), l1, wd, stream)
    h = torch.sin(torch.arange(batch * wl.n * 64, device=dev)).to(torch.bfloat16).view(batch, wl.n, 64)
    h = h[0] if batch == 1 else h
    Wg, Cg = (torch.cos(torch.arange(m * 16, device=dev)).float().view(m, 16) for m in (64, wl.K))
    f, hq, hk = torch.zeros((wl.K, 64), device=dev), torch.zeros_like(mq), torch.zeros_like(mk)
    fb.focus_assign_hidden(shape, wrap(h), Wg, Cg, None, f, hq, hk, stream=stream)
    torch.cuda.synchronize()
    return mq, mk, near, O, lse, status, o1, l1, f, hq, hk


@pytest.mark.parametrize("batch", [1, 3])
def test_same_results_both_ways(monkeypatch, batch):
    wl = fi.Workload("marshal", 4, 2, 64, 300, 4, 2, 32, seed=3)
    got = run(wl, lambda t: t, batch)
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    others = [run(wl, lambda t: t, batch, stream=torch.cuda.current_stream()), run(wl, lambda t: t.as_subclass(Sub), batch)]
    with torch.cuda.stream(side):
        others.append(run(wl, lambda t: t, batch))
    monkeypatch.setattr(fb, "_marshal", NotRead())
    others.append(run(wl, lambda t: t, batch))
    for other in others:
        for a, b in zip(got, other):
            assert torch.equal(a, b)


@pytest.mark.parametrize("direct", [True, False])
def test_same_errors_both_ways(monkeypatch, direct):
    if not direct:
        monkeypatch.setattr(fb, "_marshal", NotRead())
    wl = fi.Workload("marshal", 4, 2, 64, 40, 4, 2, 32, seed=3)
    shape = fb.shape_of(wl)
    Q, K, V, C = fi.make_inputs(wl, "cuda")
    m = torch.zeros((4, 40), dtype=torch.int32, device="cuda")
    for bad in (Q.float(), Q.cpu(), Q.transpose(1, 2), Q[0]):
        with pytest.raises(AssertionError):
            fb.focus_assign(shape, bad, 4, C, m)
    with pytest.raises(fb.FocusError, match="focus status"):
        fb.focus_assign(fb.make_shape(4, 2, 40, 63, 4, 2, 32), Q, 4, C, m)
    with pytest.raises(fb.FocusError):
        fb.focus_build_tiles(shape, m, m, 0, torch.zeros(16, dtype=torch.uint8, device="cuda"))
    with pytest.raises((AttributeError, TypeError)):
        fb.focus_attn_fwd(shape, Q, K, 7, None, None, None, 0, torch.empty_like(Q), m)
    fb.focus_assign(shape, Q, 4, C, m, None, 0)                  # a whole number for a float
    torch.cuda.synchronize()


class Calls:
    """In the place of the module: counts how often it was asked and how often it answered.  Without `behind`, no argument is of the
    usual kind."""
    def __init__(self, behind=None):
        self.asked = self.answered = 0
        self.behind = behind

    def __getattr__(self, name):
        def call(*args):
            self.asked += 1
            rc = getattr(self.behind, name)(*args) if self.behind else None
            self.answered += rc is not None
            return rc
        return call


@pytest.fixture
def through(monkeypatch):
    """through(direct) -> Calls: from here on the calls go through the module (with `direct`), or through ctypes"""
    module, put = fb._marshal, []

    def through(direct):
        put.append(Calls(module if direct else None))
        monkeypatch.setattr(fb, "_marshal", put[-1])
        return put[-1]
    yield through
    assert fb._marshal is put[-1]


def test_which_way_a_call_took(through):
    wl = fi.Workload("marshal", 4, 2, 64, 300, 4, 2, 32, seed=3)
    same, sub = lambda t: t, lambda t: t.as_subclass(Sub)
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    for direct, wrap, stream, current, answered in (
            (True, same, None, None, 6), (True, same, None, side, 6),
            (True, same, torch.cuda.current_stream(), None, 0), (True, sub, None, None, 0),    # a stream object, a tensor subclass: through ctypes
            (False, same, None, None, 0)):
        calls = through(direct)
        with torch.cuda.stream(current):
            run(wl, wrap, 1, stream=stream)
        assert calls.asked == 6 and calls.answered == answered


@pytest.mark.parametrize("direct", [True, False])
def test_same_errors_of_a_decode_step_and_of_the_router(through, direct):
    calls = through(direct)
    wl = fi.Workload("marshal", 4, 2, 64, 40, 4, 2, 32, seed=3)
    shape = fb.shape_of(wl)
    Q, K, V, C = fi.make_inputs(wl, "cuda")
    mq, mk = torch.zeros(4, dtype=torch.int32, device="cuda"), torch.zeros((2, 40), dtype=torch.int32, device="cuda")
    q, o, lse = Q[:, 0].contiguous(), torch.zeros((4, 64), dtype=torch.bfloat16, device="cuda"), torch.zeros(4, device="cuda")
    ws = torch.zeros(fb.focus_decode_workspace_bytes(shape), dtype=torch.uint8, device="cuda")
    step = lambda q=q, k=K, o=o, ws=ws: fb.focus_decode_step(shape, q, k, V, mq, mk, o, lse, ws)
    for bad in (q.float(), q.cpu(), torch.zeros((4, 128), dtype=torch.bfloat16, device="cuda")[:, ::2]):
        with pytest.raises(AssertionError):
            step(q=bad)
        with pytest.raises(AssertionError):
            step(o=bad)
    with pytest.raises(IndexError):
        step(q=q[0])                                             # [D]
    with pytest.raises(AssertionError):
        step(k=K[0])                                             # [n, D]
    with pytest.raises(fb.FocusError):
        step(ws=ws[:16])
    with pytest.raises(AttributeError):
        step(ws=None)
    h = torch.zeros((40, 128), dtype=torch.bfloat16, device="cuda")
    Wg, Cg, f = torch.zeros((64, 16), device="cuda"), torch.zeros((4, 16), device="cuda"), torch.zeros((4, 64), device="cuda")
    hq, hk = torch.zeros((4, 40), dtype=torch.int32, device="cuda"), torch.zeros((2, 40), dtype=torch.int32, device="cuda")
    route = lambda h=h[:, :64].contiguous(), Wg=Wg: fb.focus_assign_hidden(shape, h, Wg, Cg, None, f, hq, hk)
    for bad in (h[:, ::2], h[:, :64].float(), h[:, :64].cpu()):  # the first: a stride along d_model
        with pytest.raises(AssertionError):
            route(h=bad)
    with pytest.raises(IndexError):
        route(Wg=Wg[0])
    answered = calls.answered
    step()
    route()
    torch.cuda.synchronize()
    assert calls.answered == answered + (2 if direct else 0)


@pytest.mark.parametrize("direct", [True, False])
def test_a_tensor_without_storage_is_refused_both_ways(through, direct):
    """under torch.func.vmap a tensor is of the usual class and says its strides, but has no address"""
    calls = through(direct)
    wl = fi.Workload("marshal", 4, 2, 64, 40, 4, 2, 32, seed=3)
    Q, K, V, C = fi.make_inputs(wl, "cuda")
    m = torch.zeros((4, 40), dtype=torch.int32, device="cuda")
    with pytest.raises(RuntimeError):
        torch.func.vmap(lambda q: fb.focus_assign(fb.shape_of(wl), q, 4, C, m))(torch.stack([Q, Q]))
    assert calls.asked == 1 and calls.answered == 0


def test_the_library_loaded_is_the_one_called(tmp_path):
    """LIB_PATH names a copy of the library: the short calls go to it too, and their errors are found there"""
    copy = tmp_path / "libfocus_b200.so"
    shutil.copy(fb.LIB_PATH, copy)
    code = f"""
import torch
from paper_2604_03260_b200 import binding as fb
fb.LIB_PATH = {str(copy)!r}
m = torch.zeros((4, 40), dtype=torch.int32, device="cuda")
try:
    fb.focus_build_tiles(fb.make_shape(4, 2, 40, 64, 4, 2, 32), m, m, 0, torch.zeros(16, dtype=torch.uint8, device="cuda"))
except fb.FocusError as e:
    assert len(str(e)) > len(f"focus status {{e.status}}: "), str(e)
    assert fb._marshal is not fb._Ctypes
    print("refused")
"""
    out = subprocess.run([sys.executable, "-c", code], cwd=os.path.dirname(os.path.dirname(fb.LIB_PATH)), capture_output=True, text=True)
    assert out.stdout.strip() == "refused", out.stderr
