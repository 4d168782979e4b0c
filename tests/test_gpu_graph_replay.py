"""The path captured into a CUDA graph (launches that depend on their predecessor's end, the attention kernel's queue of blocks,
clusters of routing blocks): a replay over changed inputs gives what direct calls on them give, bit for bit."""
import pytest
import torch

from paper_2604_03260_b200 import binding as fb

pytestmark = pytest.mark.gpu


def replayed(call, change, outputs):
    call()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=torch.cuda.Stream()):
        call()
    change()
    for t in outputs:
        t.zero_()
    graph.replay()
    graph.replay()
    torch.cuda.synchronize()
    got = [t.clone() for t in outputs]
    for t in outputs:
        t.zero_()
    call()
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(got, outputs))


@pytest.mark.parametrize("D,n,layout", [(64, 1000, 0), (128, 3001, 0), (128, 3001, 1), (256, 2500, 3), (128, 2500, 4)])
def test_tiles_and_attention(D, n, layout):
    g = torch.Generator(device="cuda"); g.manual_seed(n + D)
    Hq, Hkv, K = 8, 4, 4
    shape = fb.make_shape(Hq, Hkv, n, D, K, 1, 200, batch=2)
    q, k, v = (torch.randn((2, H, n, D), generator=g, device="cuda").to(torch.bfloat16) for H in (Hq, Hkv, Hkv))
    mq, mk = ((1 << torch.randint(0, K, (2 * H, n), generator=g, device="cuda")).to(torch.int32) for H in (Hq, Hkv))
    ws = fb.alloc_workspace(shape, layout)
    o, lse = torch.empty_like(q), torch.empty((2 * Hq, n), device="cuda")
    status = torch.zeros(4, dtype=torch.int32, device="cuda")

    def call():
        fb.focus_build_tiles(shape, mq, mk, layout, ws)
        fb.focus_attn_fwd(shape, q, k, v, mq, mk, ws, layout, o, lse, status)

    def change():
        q.neg_()
        mq.copy_(mq.roll(1, 1))

    replayed(call, change, [o, lse])
    assert status.tolist()[0] == 0 and o.isfinite().all()


def test_routing_gate_and_decode():
    g = torch.Generator(device="cuda"); g.manual_seed(3)
    n, d, K, D, Hq, Hkv = 700, 1024, 8, 128, 8, 2
    shape = fb.make_shape(Hq, Hkv, n, D, K, 2, 64)
    h = torch.randn((n, d), generator=g, device="cuda").to(torch.bfloat16)
    Wg, C = torch.randn((d, 16), generator=g, device="cuda") / d ** 0.5, torch.randn((K, 16), generator=g, device="cuda")
    folded = torch.empty((K, d), device="cuda")
    mq, mk = (torch.zeros((H, n), dtype=torch.int32, device="cuda") for H in (Hq, Hkv))
    q, k, v = (torch.randn((H, n, D), generator=g, device="cuda").to(torch.bfloat16) for H in (Hq, Hkv, Hkv))
    soft = torch.softmax(torch.randn((1, n, K), generator=g, device="cuda"), -1)
    o, lse = torch.empty_like(q), torch.empty((Hq, n), device="cuda")
    od, ld = torch.empty((Hq, D), dtype=torch.bfloat16, device="cuda"), torch.empty(Hq, device="cuda")
    status = torch.zeros(4, dtype=torch.int32, device="cuda")
    ws = torch.empty(fb.focus_decode_workspace_bytes(shape), dtype=torch.uint8, device="cuda")
    mq_new = torch.zeros(Hq, dtype=torch.int32, device="cuda")

    def call():
        fb.focus_assign_hidden(shape, h, Wg, C, None, folded, mq, mk)
        mq_new.copy_(mq[:, -1])
        fb.focus_decode_step(shape, q[:, -1], k, v, mq_new, mk, od, ld, ws)
        fb.focus_gate_attn_fwd(shape, q, k, v, soft, 10.0, o, lse, status)

    def change():
        h.copy_(h.roll(1, 0))
        k.neg_()

    replayed(call, change, [mq, mk, od, ld, o, lse])
    assert status.tolist()[0] == 0 and o.isfinite().all()
