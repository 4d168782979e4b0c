"""focus_assign of few vectors (generation, short prompts) against fp64, and against the same vectors in a long call."""
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


@pytest.mark.parametrize("D,K,topk", [(64, 4, 2), (128, 4, 1), (128, 8, 2), (256, 7, 3), (256, 4, 2), (64, 3, 3)])
def test_masks_do_not_depend_on_the_size_of_the_call(D, K, topk):
    """the vectors of one long call in short calls of every size: the same masks and near-ties, bit for bit, with pairs of
    centroids a rounding apart, a zero one, one with a vanishing norm, and vectors that are zero, huge, tiny, infinite or not numbers"""
    H, Hkv, n = 8, 4, 3000
    g = torch.Generator(device="cuda"); g.manual_seed(D + K)
    x = torch.randn((1, H, n, D), generator=g, device="cuda").to(torch.bfloat16)
    x[:, :, 5], x[:, :, 6], x[:, :, 7], x[:, :, 8] = 0, x[:, :, 6] * 1e30, x[:, :, 7] * 1e-25, x[:, :, 8] * 1e18
    x[:, :, 9, 3], x[:, :, 10, 0] = float("inf"), float("nan")
    C = torch.randn((Hkv, K, D), generator=g, device="cuda")
    C[:, 1] = C[:, 0] * (1 + 2e-7 * torch.randn((Hkv, D), generator=g, device="cuda"))
    C[1, K - 1], C[2, K - 1] = 0, 1e-24 * C[2, K - 1]
    C[3] *= 1e-6

    def assign(x):
        m = torch.full((H, x.shape[2]), -1, dtype=torch.int32, device="cuda")
        near = torch.zeros(1, dtype=torch.int64, device="cuda")
        fb.focus_assign(fb.make_shape(H, Hkv, x.shape[2], D, K, topk, 16), x, H, C, m, near)
        return m, near.item()
    want, near = assign(x)
    assert topk == K or 0.02 < ((want ^ (want >> 1)) & 1).float().mean()          # some vectors take one of the pair alone
    for sizes in ((1, 2, 3, 127), (128, 129, 200), (256,)):
        at, i, total, parts = 0, 0, 0, []
        while at < n:
            c = min(sizes[i % len(sizes)], n - at)
            if sizes[0] == 1 and at >= 700:                  # the shortest calls over the first part only
                c = min(256, n - at)
            m, t = assign(x[:, :, at:at + c])
            parts.append(m); total += t; at += c; i += 1
        assert torch.equal(torch.cat(parts, 1), want) and total == near
