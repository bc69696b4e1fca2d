"""Kernels at the sizes where they can go wrong: edges of tiles, remainders, the smallest and the largest
of a range, against plain fp64 arithmetic on the identical bf16 inputs."""
import pytest
import torch

pytestmark = pytest.mark.gpu

def _randn(g, *shape):
    return torch.randn(*shape, generator=g).to(torch.bfloat16)


@pytest.mark.parametrize("n0,n,H,relu", [
    (0, 1, 2, 0), (0, 63, 2, 0), (0, 64, 3, 0), (0, 65, 2, 1), (1, 62, 2, 0), (1, 63, 2, 0), (63, 2, 2, 0), (64, 640, 2, 1),
    (100, 1000, 16, 0), (0, 1500, 40, 0)])
def test_append_head_dim_64(n0, n, H, relu, cuda_device):
    """State, key sums and pages of an append at head_dim 64: one block, edges of a page on both sides, a
    first block that holds older tokens, several blocks per CTA, more heads than give every CTA a split."""
    from paper_2609_34606_b200 import hsa
    d = 64
    g = torch.Generator().manual_seed(77 + 1000 * n0 + n)
    K, V = _randn(g, n0 + n, H, d), _randn(g, n0 + n, H, d)
    nb = (n0 + n + 63) // 64
    order = torch.randperm(nb + 2, generator=g).to(torch.int32)
    ctx = hsa.HSAContext(H, d, max_pages=nb + 2, max_q_tokens=max(n, n0, 1), max_topk=nb, device=cuda_device,
                         page_order=order, feature_map=relu)
    ctx.k_pool.fill_(0xFF)
    ctx.v_pool.fill_(0xFF)
    for lo, hi in ((0, n0), (n0, n0 + n)):
        if hi > lo:
            ctx.append_kv(K[lo:hi].to(cuda_device), V[lo:hi].to(cuda_device))
    assert ctx.device_status() == 0
    Kd, Vd = K.double(), V.double()
    phi = Kd.clamp(min=0) if relu else torch.where(Kd > 0, Kd + 1, Kd.exp())
    rel = lambda got, ref: float((got.double().cpu() - ref).norm() / ref.norm())
    # fp32 sums of terms that carry 24 bits: every addition rounds by 2^-24 of a partial sum that is of the
    # order of the result, at most n0 + n of them one after another, of random sign
    bound = 2.0 ** -24 * (4 + (n0 + n) ** 0.5)
    assert rel(ctx.S, torch.einsum("thk,thd->hkd", phi, Vd)) <= bound
    assert rel(ctx.z, phi.sum(0)) <= bound
    pad = torch.zeros(nb * 64 - n0 - n, H, d, dtype=torch.float64)
    blocks = torch.cat([Kd, pad]).view(nb, 64, H, d)
    assert rel(ctx.ksum[:, :nb], blocks.sum(1).permute(1, 0, 2)) <= 2.0 ** -24 * 12
    for pool, ref in ((ctx.k_pool, K), (ctx.v_pool, V)):
        pages = pool.view(torch.bfloat16).view(nb + 2, H, 64, d)[order[:nb].long().to(cuda_device)].cpu()
        want = torch.cat([ref, pad.to(torch.bfloat16)]).view(nb, 64, H, d).permute(0, 2, 1, 3)
        assert torch.equal(pages, want)
    ctx.destroy()
