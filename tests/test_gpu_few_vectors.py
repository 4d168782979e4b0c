"""focus_assign's warp-per-vector form against the tile form and fp64: the sizes on both sides of the line between them."""
import pytest
import torch

from paper_2604_03260_b200 import binding as fb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D,H,Hkv,n,K,topk,batch", [(128, 32, 8, 1, 4, 2, 1), (128, 8, 8, 1, 4, 1, 3), (64, 12, 12, 341, 4, 2, 1), (64, 12, 12, 342, 4, 2, 1),
                                                    (256, 16, 8, 127, 7, 2, 1), (256, 16, 8, 129, 7, 7, 1), (128, 4, 2, 511, 1, 1, 1), (128, 4, 2, 33, 8, 3, 2)])
def test_few_vectors(D, H, Hkv, n, K, topk, batch):
    g = torch.Generator(device="cuda"); g.manual_seed(n + D + K)
    # rows further apart than D, and a zero vector
    x = torch.randn((batch, H, n, D + 8), generator=g, device="cuda").to(torch.bfloat16)[..., :D]
    x[0, 0, 0] = 0
    C = torch.randn((Hkv, K, D), generator=g, device="cuda")
    shape = fb.make_shape(H, Hkv, n, D, K, topk, 16, batch=batch)
    m = torch.full((batch * H, n), -1, dtype=torch.int32, device="cuda")
    near = torch.zeros(1, dtype=torch.int64, device="cuda")
    fb.focus_assign(shape, x, H, C, m, near)
    c64 = (C.double() / C.double().norm(dim=-1, keepdim=True)).repeat_interleave(H // Hkv, 0)
    v = x.double()
    cos = torch.einsum("bhnd,hkd->bhnk", v / v.norm(dim=-1, keepdim=True).clamp_min(1e-30), c64)
    top = cos.sort(dim=-1, descending=True, stable=True)
    ref = (1 << top.indices[..., :topk]).sum(-1).to(torch.int32).view(batch * H, n)
    margin = top.values[..., topk - 1] - top.values[..., topk] if topk < K else torch.ones_like(cos[..., 0])
    margin[0, 0, 0] = 1.0                                   # all scores of the zero vector tie: the first groups
    sure = (margin >= 1e-5).reshape(batch * H, n)
    assert (m == ref)[sure].all() and near.item() <= (~sure).sum().item() + (1 if topk < K else 0) and (~sure).sum().item() < 3 + 1e-3 * m.numel()


@pytest.mark.parametrize("D,n", [(64, 3), (128, 1), (256, 40)])
def test_centroids_at_an_odd_float(D, n):
    """a contiguous set of centroids that starts on the 4-byte grid only, as a slice of a parameter buffer can"""
    H, Hkv, K = 8, 4, 5
    g = torch.Generator(device="cuda"); g.manual_seed(n + D)
    x = torch.randn((1, H, n, D), generator=g, device="cuda").to(torch.bfloat16)
    buf = torch.randn(Hkv * K * D + 1, generator=g, device="cuda")
    odd = buf[1:].view(Hkv, K, D)
    assert odd.data_ptr() % 8 == 4
    shape = fb.make_shape(H, Hkv, n, D, K, 2, 16)
    got, want = (torch.full((H, n), -1, dtype=torch.int32, device="cuda") for _ in range(2))
    fb.focus_assign(shape, x, H, odd, got)
    fb.focus_assign(shape, x, H, odd.clone(), want)
    assert torch.equal(got, want) and (want > 0).all()
