"""Kernels at the sizes where they can go wrong: edges of tiles, remainders, the smallest and the largest
of a range, against the oracle or plain fp64 arithmetic on the identical bf16 inputs."""
import numpy as np
import pytest
import torch

import hsa_harness as Hn
from oracle import hsa_oracle as O

pytestmark = pytest.mark.gpu

# largest relative error of a value that is computed in 32 bits and rounded to bf16 once (8 significant bits)
BF16_REL = 2.0 ** -8


def _randn(g, *shape):
    return torch.randn(*shape, generator=g).to(torch.bfloat16)


@pytest.mark.parametrize("n0,n_q,d,relu", [
    (0, 1, 128, 0), (0, 64, 128, 0), (0, 128, 128, 0), (0, 129, 128, 1), (64, 127, 128, 0), (63, 65, 128, 0),
    (1, 257, 128, 0), (190, 385, 128, 1), (33, 640, 128, 0), (0, 1, 64, 0), (63, 130, 64, 0), (17, 300, 64, 1)])
def test_causal_intra_chunk_products(n0, n_q, d, relu, cuda_device):
    """Intra-chunk part of the causal linear branch (one tile, several tiles, a ragged last one; a chunk
    that starts at, just before and just behind a page boundary) through both kernels that add it."""
    from paper_2609_34606_b200 import hsa
    H = 3
    g = torch.Generator().manual_seed(1000 * n0 + n_q)
    n = n0 + n_q
    K, V, q = _randn(g, n, H, d), _randn(g, n, H, d), _randn(g, n_q, H, d)
    n_blocks = (n + 63) // 64
    ctx = hsa.HSAContext(H, d, max_pages=n_blocks + 1, max_q_tokens=max(n_q, n0, 1), max_topk=n_blocks, causal=True,
                         device=cuda_device, feature_map=relu,
                         page_order=torch.arange(n_blocks, -1, -1, dtype=torch.int32))
    ctx.k_pool.fill_(0xFF)
    ctx.v_pool.fill_(0xFF)
    if n0:
        ctx.append_kv(K[:n0].to(cuda_device), V[:n0].to(cuda_device))
    ctx.append_kv(K[n0:].to(cuda_device), V[n0:].to(cuda_device))
    qd = q.to(cuda_device)
    budgets = torch.full((H,), -1, dtype=torch.int32, device=cuda_device)
    idx, cnt = ctx.select_blocks(qd, budgets, q_pos0=n0, causal=True)
    alone = ctx.forward(qd, idx, cnt, q_pos0=n0, causal=True, flags=hsa.HSA_FWD_NO_SPARSE)
    both = ctx.forward(qd, idx, cnt, q_pos0=n0, causal=True)
    assert ctx.device_status() == 0
    fmap = "relu" if relu else "elu1"
    lin = O.linear_parallel(Hn.f32(q), Hn.f32(K), Hn.f32(V), n0, True, fmap=fmap)
    sp = O.dense_attention(Hn.f32(q), Hn.f32(K), Hn.f32(V), n0, True)
    assert np.linalg.norm(Hn.f64(alone) - lin) <= BF16_REL * np.linalg.norm(lin)
    ref = lin + sp
    # (the sparse branch's weights are bf16 as well: one more rounding)
    assert np.linalg.norm(Hn.f64(both) - ref) <= 1.5 * BF16_REL * np.linalg.norm(ref)
    ctx.destroy()


def _causal_partials(ctx, n, size):
    """Numerator [n, H, d] and denominator [n, H] in the workspace of a context for chunks of `size` tokens: they
    come first in what the causal flag adds to it (short lists, no adaptive selection)."""
    from paper_2609_34606_b200 import hsa
    plain = hsa.hsa_config.from_buffer_copy(ctx.cfg)
    plain.flags = 0
    lo, H, d = hsa.hsa_query_sizes(plain).workspace, ctx.H, ctx.d
    num = ctx.workspace[lo:lo + 4 * n * H * d].view(torch.float32).view(n, H, d).double().cpu()
    lo += (4 * size * H * d + 255) // 256 * 256
    return num, ctx.workspace[lo:lo + 4 * n * H].view(torch.float32).view(n, H).double().cpu()


@pytest.mark.parametrize("n0,n,d,relu", [(0, 1, 128, 0), (100, 65, 128, 0), (64, 640, 128, 0), (1, 1000, 64, 0), (70, 300, 128, 1),
                                         (0, 129, 64, 1)])
def test_causal_partials_carry_24_bits(n0, n, d, relu, cuda_device):
    """Numerator and denominator of the intra-chunk part against 64 bits.  Map, weights and sums are 32-bit
    quantities: relative errors of 2^-24 per rounding, a few in a row, so 2^-21 is allowed; carried in 16 bits
    anywhere they are off by 2^-17 and more."""
    from paper_2609_34606_b200 import hsa
    H = 3
    g = torch.Generator().manual_seed(n)
    k, v, q = _randn(g, n, H, d), _randn(g, n, H, d), _randn(g, n, H, d)
    size = max(n, n0, 1)
    ctx = hsa.HSAContext(H, d, max_pages=(n0 + n + 63) // 64, max_q_tokens=size, max_topk=1, causal=True, device=cuda_device,
                         feature_map=relu)
    if n0:
        ctx.append_kv(_randn(g, n0, H, d).to(cuda_device), _randn(g, n0, H, d).to(cuda_device))
    ctx.append_kv(k.to(cuda_device), v.to(cuda_device))
    ctx.forward(q.to(cuda_device), None, None, q_pos0=n0, causal=True, flags=hsa.HSA_FWD_NO_SPARSE)
    assert ctx.device_status() == 0
    num, den = _causal_partials(ctx, n, size)
    phi = lambda x: x.clamp(min=0) if relu else torch.where(x > 0, x + 1, x.exp())
    A = torch.einsum("ihd,jhd->hij", phi(q.double()), phi(k.double())).tril()
    for got, ref in ((num, torch.einsum("hij,jhd->ihd", A, v.double())), (den, A.sum(2).T)):
        assert float((got - ref).norm()) <= 2.0 ** -21 * float(ref.norm())
    ctx.destroy()

@pytest.mark.parametrize("n0,n,relu,odd", [(0, 641, 0, False), (63, 768, 0, False), (64, 769, 1, False), (1, 1281, 0, False),
                                           (100, 1500, 0, True), (0, 700, 1, True)])
def test_causal_sums_over_groups(n0, n, relu, odd, cuda_device):
    """Chunks long enough for sums over groups of pages (the first and the last tile of a group, one row in a last
    tile or group, a group that starts inside a page): partials against 64 bits as above, and, with Inf and NaN in K and
    V inside a group, what a plain sum has."""
    from paper_2609_34606_b200 import hsa
    H, d, inf, nan = 2, 128, float("inf"), float("nan")
    g = torch.Generator().manual_seed(n)
    k, v, q = _randn(g, n, H, d), _randn(g, n, H, d), _randn(g, n, H, d)
    if odd:
        t = n - 300
        v[t, 0, 5], v[t + 70, 0, 6], v[t + 3, 0, 7] = inf, -inf, nan
        k[t, 1, 9] = inf
    ctx = hsa.HSAContext(H, d, max_pages=(n0 + n + 63) // 64, max_q_tokens=n, max_topk=1, causal=True, device=cuda_device,
                         feature_map=relu)
    if n0:
        ctx.append_kv(_randn(g, n0, H, d).to(cuda_device), _randn(g, n0, H, d).to(cuda_device))
    ctx.append_kv(k.to(cuda_device), v.to(cuda_device))
    ctx.forward(q.to(cuda_device), None, None, q_pos0=n0, causal=True, flags=hsa.HSA_FWD_NO_SPARSE)
    assert ctx.device_status() == 0
    num, den = _causal_partials(ctx, n, n)
    phi = lambda x: x.double().clamp(min=0) if relu else torch.where(x > 0, x.double() + 1, x.double().exp())
    ref_num, ref_den = torch.zeros(n, H, d, dtype=torch.float64), torch.zeros(n, H, dtype=torch.float64)
    for i in range(n):
        w = (phi(q[i])[None] * phi(k[:i + 1])).sum(2)
        ref_num[i], ref_den[i] = (w[:, :, None] * v[:i + 1].double()).sum(0), w.sum(0)
    for got, ref in ((num, ref_num), (den, ref_den)):
        wrong = ~ref.isfinite()
        assert bool(wrong.any()) == (odd and (got is num or bool((~ref_den.isfinite()).any())))
        assert torch.equal(torch.nan_to_num(got[wrong], nan=1.0), torch.nan_to_num(ref[wrong], nan=1.0))
        assert float((got[~wrong] - ref[~wrong]).norm()) <= 2.0 ** -21 * float(ref[~wrong].norm())
    ctx.destroy()


@pytest.mark.parametrize("H,n", [(1, 769), (12, 1560)])
def test_causal_sums_that_give_up_leave_the_context_usable(H, n, cuda_device):
    """The sums over page groups are given up with copies in flight (a wait limit of one nanosecond): their kernel ends by itself
    and says so, and the next forward is what it was."""
    from paper_2609_34606_b200 import hsa
    d, n0 = 128, 100
    g = torch.Generator(device=cuda_device).manual_seed(n)
    rand = lambda *s: torch.randn(*s, generator=g, device=cuda_device).to(torch.bfloat16)
    ctx = hsa.HSAContext(H, d, max_pages=(n0 + n + 63) // 64, max_q_tokens=n, max_topk=8, causal=True, device=cuda_device)
    ctx.append_kv(rand(n0, H, d), rand(n0, H, d))
    ctx.append_kv(rand(n, H, d), rand(n, H, d))
    q = rand(n, H, d)
    idx, cnt = ctx.select_blocks(q, torch.full((H,), 8, dtype=torch.int32, device=cuda_device), q_pos0=n0, causal=True)
    want = ctx.forward(q, idx, cnt, q_pos0=n0, causal=True)
    assert ctx.device_status() == 0
    ctx.set_wait_limit_ns(1)
    for _ in range(3):
        ctx.forward(q, idx, cnt, q_pos0=n0, causal=True)
        assert ctx.device_status() == hsa.HSA_ERR_DEVICE_TIMEOUT
    ctx.set_wait_limit_ns(2_000_000_000)
    out = ctx.forward(q, idx, cnt, q_pos0=n0, causal=True)
    assert ctx.device_status() == 0 and torch.equal(out, want)
    ctx.destroy()


@pytest.mark.parametrize("n0,n,d,relu", [(0, 100, 128, 0), (100, 300, 128, 0), (70, 300, 64, 0), (64, 300, 128, 1)])
def test_causal_not_finite_values_stay_behind_their_position(n0, n, d, relu, cuda_device):
    """Inf and NaN in K, V and queries of a causal chunk reach the rows at and behind them, and there what they
    reach in a plain sum, and nothing before them."""
    from paper_2609_34606_b200 import hsa
    H, inf, nan = 4, float("inf"), float("nan")
    g = torch.Generator().manual_seed(n0 + d)
    k, v, q = _randn(g, n, H, d), _randn(g, n, H, d), _randn(g, n, H, d)
    t = n - 30
    v[t, 0, 5], v[t, 0, 6], v[3, 0, 7] = inf, -inf, nan
    k[t, 1, 9], k[t + 9, 1, 2] = inf, -inf
    q[20, 2, 33], q[t, 2, 0], q[t + 1, 2, 1] = inf, -inf, nan
    size = max(n, n0)
    ctx = hsa.HSAContext(H, d, max_pages=(n0 + n + 63) // 64, max_q_tokens=size, max_topk=1, causal=True, device=cuda_device,
                         feature_map=relu)
    if n0:
        ctx.append_kv(_randn(g, n0, H, d).to(cuda_device), _randn(g, n0, H, d).to(cuda_device))
    ctx.append_kv(k.to(cuda_device), v.to(cuda_device))
    ctx.forward(q.to(cuda_device), None, None, q_pos0=n0, causal=True, flags=hsa.HSA_FWD_NO_SPARSE)
    assert ctx.device_status() == 0
    num, den = _causal_partials(ctx, n, size)

    def phi(x):
        x = x.double()  # (max(NaN, 0) is 0 on the GPU)
        return torch.nan_to_num(x, nan=0.0, posinf=inf, neginf=-inf).clamp(min=0) if relu else torch.where(x > 0, x + 1, x.exp())

    ref_num, ref_den = torch.zeros(n, H, d, dtype=torch.float64), torch.zeros(n, H, dtype=torch.float64)
    for i in range(n):
        w = (phi(q[i])[None] * phi(k[:i + 1])).sum(2)
        ref_num[i], ref_den[i] = (w[:, :, None] * v[:i + 1].double()).sum(0), w.sum(0)
    for got, ref in ((num, ref_num), (den, ref_den)):
        odd = ~ref.isfinite()
        assert torch.equal(torch.nan_to_num(got[odd], nan=1.0), torch.nan_to_num(ref[odd], nan=1.0))
        assert float((got[~odd] - ref[~odd]).norm()) <= 2.0 ** -21 * float(ref[~odd].norm())
    ctx.destroy()

@pytest.mark.parametrize("d", [64, 128])
def test_causal_nan_key_reaches_the_queries_behind_it(d, cuda_device):
    """A NaN in a key of the chunk makes the linear branch NaN for the queries at and behind it (elu), and a NaN in
    a query makes its own row NaN."""
    from paper_2609_34606_b200 import hsa
    H, n0, n = 2, 100, 300
    g = torch.Generator().manual_seed(d)
    K, V, q = _randn(g, n, H, d), _randn(g, n, H, d), _randn(g, n, H, d)
    K[150, 1, 3] = q[20, 0, 7] = float("nan")
    ctx = hsa.HSAContext(H, d, max_pages=7, max_q_tokens=n, max_topk=1, causal=True, device=cuda_device)
    ctx.append_kv(_randn(g, n0, H, d).to(cuda_device), _randn(g, n0, H, d).to(cuda_device))
    ctx.append_kv(K.to(cuda_device), V.to(cuda_device))
    out = ctx.forward(q.to(cuda_device), None, None, q_pos0=n0, causal=True, flags=hsa.HSA_FWD_NO_SPARSE).cpu()
    assert ctx.device_status() == 0
    bad = out.isnan().any(2)
    assert bad[:, 1].tolist() == [t >= 150 for t in range(n)]
    assert bad[:, 0].tolist() == [t == 20 for t in range(n)]
    ctx.destroy()

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


@pytest.mark.parametrize("n,H", [(1, 1), (63, 2), (64, 2), (1000, 16), (4680, 3)])
def test_key_sums_head_dim_64_are_rounded_sums(n, H, cuda_device):
    """Key sums of blocks that are new as a whole: bit for bit those of the page kernel of a context without a
    linear state (rounded fp32 in a fixed order), also for keys spread over 16 octaves."""
    from paper_2609_34606_b200 import hsa
    d = 64
    g = torch.Generator().manual_seed(n)
    K = (torch.randn(n, H, d, generator=g) * torch.exp2(torch.randint(-12, 4, (n, H, d), generator=g).float()))
    K, V = K.to(torch.bfloat16).to(cuda_device), _randn(g, n, H, d).to(cuda_device)
    sums = []
    for mode in (hsa.HSA_LIN_STATE, hsa.HSA_LIN_NONE):
        ctx = hsa.HSAContext(H, d, max_pages=(n + 63) // 64, max_q_tokens=n, max_topk=1, device=cuda_device, lin_mode=mode)
        ctx.append_kv(K, V)
        assert ctx.device_status() == 0
        sums.append(ctx.ksum.clone())
        ctx.destroy()
    assert torch.equal(*sums)

@pytest.mark.parametrize("n,relu", [(1, 0), (70, 0), (1000, 0), (1000, 1)])
def test_append_head_dim_64_not_finite(n, relu, cuda_device):
    """Inf and NaN in K and V reach the entries of S, z and the key sums that they reach in a plain sum, as the
    same Inf or NaN, and no other."""
    from paper_2609_34606_b200 import hsa
    H, d, inf, nan = 4, 64, float("inf"), float("nan")
    g = torch.Generator().manual_seed(n + relu)
    K, V = _randn(g, n, H, d), _randn(g, n, H, d)
    t = n // 2
    V[t, 0, 5], V[t, 1, 63] = inf, -inf       # head 0, 1: a value
    K[t, 1, 9], K[0, 2, 40], K[n - 1, 2, 41] = inf, -inf, inf  # head 1, 2: keys
    K[t, 3, 0], V[t, 3, 1] = nan, nan
    ctx = hsa.HSAContext(H, d, max_pages=(n + 63) // 64, max_q_tokens=n, max_topk=1, device=cuda_device, feature_map=relu)
    ctx.append_kv(K.to(cuda_device), V.to(cuda_device))
    assert ctx.device_status() == 0
    Kd, Vd = K.double(), V.double()
    # (max(NaN, 0) is 0 on the GPU, as it always was with this map)
    phi = torch.nan_to_num(Kd, nan=0.0, posinf=inf, neginf=-inf).clamp(min=0) if relu else torch.where(Kd > 0, Kd + 1, Kd.exp())
    S = torch.stack([(phi[:, h, :, None] * Vd[:, h, None, :]).sum(0) for h in range(H)])
    bound = 2.0 ** -24 * (4 + n ** 0.5)
    for got, ref in ((ctx.S, S), (ctx.z, phi.sum(0)), (ctx.ksum[:, 0], Kd[:64].sum(0))):
        got, odd = got.double().cpu(), ~ref.isfinite()
        assert torch.equal(torch.nan_to_num(got[odd], nan=1.0), torch.nan_to_num(ref[odd], nan=1.0))
        assert float((got[~odd] - ref[~odd]).norm()) <= bound * float(ref[~odd].norm())
    ctx.destroy()

@pytest.mark.parametrize("d,n_q,topk,layout,act,split", [
    (128, 300, 6, "dim", 1, 0), (128, 129, 1, "dim", 0, 0), (128, 128, 2, "dim", 1, 0), (128, 260, 5, "dim", 1, 2),
    (64, 300, 6, "dim", 1, 0), (64, 257, 7, "dim", 1, 2), (128, 200, 0, "dim", 1, 0), (128, 300, 6, "head", 1, 0),
    (128, 300, 6, "dim_strided", 1, 0), (128, 300, 6, "token", 1, 0), (128, 300, 6, "lin_only", 1, 0),
    (64, 300, 6, "sp_only", 0, 0), (128, 300, 6, "unaligned", 1, 0)])
def test_gate_layouts(d, n_q, topk, layout, act, split, cuda_device):
    """Gates as tiles (per dim), per token and head, broadcast over heads, strided, misaligned, and one of the
    two alone: each against the merge of the two branches as the kernel itself gives them."""
    from paper_2609_34606_b200 import hsa
    H, n = 3, 700
    g = torch.Generator().manual_seed(5 + n_q + topk)
    K, V, q = _randn(g, n, H, d), _randn(g, n, H, d), _randn(g, n_q, H, d).to(cuda_device)
    ctx = hsa.HSAContext(H, d, max_pages=11, max_q_tokens=n, max_topk=11, device=cuda_device, gate_act=act, split_blocks=split)
    ctx.append_kv(K.to(cuda_device), V.to(cuda_device))
    idx, cnt = ctx.select_blocks(q, torch.full((H,), topk, dtype=torch.int32, device=cuda_device))
    make = {"head": lambda: _randn(g, n_q, H).to(cuda_device),
            "dim_strided": lambda: _randn(g, n_q, H, 2 * d).to(cuda_device)[:, :, ::2],
            "token": lambda: _randn(g, n_q, 1, d).to(cuda_device).expand(n_q, H, d),
            "unaligned": lambda: _randn(g, n_q * H * d + 1).to(cuda_device)[1:].view(n_q, H, d)}.get(
                layout, lambda: _randn(g, n_q, H, d).to(cuda_device))
    gl = None if layout == "sp_only" else make()
    gs = None if layout == "lin_only" else make()
    out = ctx.forward(q, idx, cnt, g_lin=gl, g_sp=gs)
    lin = ctx.forward(q, idx, cnt, flags=hsa.HSA_FWD_NO_SPARSE).double()
    sp = ctx.forward(q, idx, cnt, flags=hsa.HSA_FWD_NO_LINEAR).double()
    assert ctx.device_status() == 0

    def weight(x):
        if x is None:
            return 1.0
        x = x.double() if x.dim() == 3 else x.double()[:, :, None]
        return torch.sigmoid(x) if act else x

    ref = weight(gl) * lin + weight(gs) * sp
    # the branches are rounded to bf16 before they are merged here, the result is once
    size = (weight(gl) * lin).abs() + (weight(gs) * sp).abs()
    assert float(((out.double() - ref).abs() - 2 * BF16_REL * size - 1e-6).max()) <= 0.0
    ctx.destroy()


@pytest.mark.parametrize("d,split,form", [(128, 0, "state"), (64, 0, "state"), (128, 2, "state"), (64, 2, "state"), (128, 0, "linformer")])
@pytest.mark.parametrize("which", ["g_lin", "g_sp"])
def test_one_gate_off_the_tile_alignment(d, split, form, which, cuda_device):
    """Per-dim gates of which only one starts on a 16-byte boundary (the other is a view one element into its
    buffer): both are applied."""
    from paper_2609_34606_b200 import hsa
    H, n, n_q = 3, 640, 200
    g = torch.Generator().manual_seed(d + split)
    rand = lambda *s: _randn(g, *s).to(cuda_device)
    opt = {}
    if form == "linformer":
        opt = dict(lin_mode=hsa.HSA_LIN_LINFORMER, lin_rank=64, lin_seg_tokens=n, e_k=rand(H, n, 64) * 0.04, e_v=rand(H, n, 64) * 0.04)
    ctx = hsa.HSAContext(H, d, max_pages=10, max_q_tokens=n, max_topk=10, device=cuda_device, gate_act=1, split_blocks=split, **opt)
    ctx.append_kv(rand(n, H, d), rand(n, H, d))
    q = rand(n_q, H, d)
    idx, cnt = ctx.select_blocks(q, torch.full((H,), 6, dtype=torch.int32, device=cuda_device))
    gates = {"g_lin": rand(n_q, H, d), "g_sp": rand(n_q, H, d)}
    both = ctx.forward(q, idx, cnt, **gates)
    moved = torch.empty(n_q * H * d + 1, dtype=torch.bfloat16, device=cuda_device)[1:].view(n_q, H, d)
    gates[which] = moved.copy_(gates[which])
    out = ctx.forward(q, idx, cnt, **gates)
    lin = ctx.forward(q, idx, cnt, flags=hsa.HSA_FWD_NO_SPARSE).double()
    sp = ctx.forward(q, idx, cnt, flags=hsa.HSA_FWD_NO_LINEAR).double()
    assert ctx.device_status() == 0
    a, b = torch.sigmoid(gates["g_lin"].double()) * lin, torch.sigmoid(gates["g_sp"].double()) * sp
    # the branches are rounded to bf16 before they are merged here, the result is once
    assert float(((out.double() - a - b).abs() - 2 * BF16_REL * (a.abs() + b.abs()) - 1e-6).max()) <= 0.0
    # and as with both on the boundary: the same arithmetic up to the order of two products
    assert float((out.double() - both.double()).abs().max()) <= 2 * BF16_REL * float(both.double().abs().max())
    ctx.destroy()

@pytest.mark.parametrize("d,H,n,kvb", [(128, 3, 65, 1), (128, 2, 5000, 7), (64, 5, 5000, 195), (128, 12, 70000, 195),
                                       (64, 2, 70000, 256), (128, 2, 70000, 257), (128, 1, 70000, 700), (128, 2, 70000, 5000)])
def test_kv_page_scores(d, H, n, kvb, cuda_device):
    """Scores of KV pages of one block, of less, as many and more blocks than one CTA takes, and of one page
    that is longer than the history, against fp64; the ids are the best pages in ascending order."""
    from paper_2609_34606_b200 import hsa
    g = torch.Generator().manual_seed(n + kvb)
    nb, n_q = (n + 63) // 64, 150
    K, q = _randn(g, n, H, d), _randn(g, n_q, H, d)
    ctx = hsa.HSAContext(H, d, max_pages=nb + 3, max_q_tokens=max(n, n_q), max_topk=4, lin_mode=hsa.HSA_LIN_NONE, device=cuda_device)
    kd = K.to(cuda_device)
    ctx.append_kv(kd, kd)
    ids, scores = ctx.retrieve_kv_pages(q.to(cuda_device), kvb, top_kp=3, with_scores=True)
    assert ctx.device_status() == 0
    n_pages = (nb + kvb - 1) // kvb
    qbar = q.double().mean(0)
    ref = torch.stack([(qbar * K[j * kvb * 64:(j + 1) * kvb * 64].double().mean(0)).sum() / H * d ** -0.5
                       for j in range(n_pages)])
    # key and query sums are fp32 sums of up to 128 values (2^-24 of partial sums each), the rest is fp64;
    # the scores are sums of H d products of random sign
    assert float((scores.double().cpu() - ref).abs().max()) <= 2.0 ** -20 * float(ref.abs().max())
    best = torch.sort(scores.cpu(), descending=True, stable=True).indices[:min(3, n_pages)]
    assert ids.cpu().tolist() == sorted(best.tolist())
    ctx.destroy()


@pytest.mark.parametrize("d,H,n,n_q,causal", [
    (128, 2, 1, 1, False), (128, 2, 64, 130, False), (64, 3, 65, 64, True), (128, 3, 31 * 64, 200, False),
    (128, 2, 32 * 64, 128, True), (64, 2, 33 * 64 - 5, 3200, False), (128, 2, 767 * 64, 300, False),
    (128, 1, 769 * 64 + 1, 3100, True), (64, 1, 6144 * 64, 100, False), (64, 1, 6145 * 64, 100, False)])
def test_adaptive_lists(d, H, n, n_q, causal, cuda_device):
    """Cumulative-mass lists at one block, at the edges of the sort's warp segments and of the threads' shares,
    at the largest history of the one-kernel form and behind it, with the query sums taken inside the
    clusters (up to 24 tiles) and in front of them."""
    from paper_2609_34606_b200 import hsa
    g = torch.Generator().manual_seed(n + n_q)
    K, q = _randn(g, n, H, d), _randn(g, n_q, H, d)
    nb = (n + 63) // 64
    ctx = hsa.HSAContext(H, d, max_pages=nb, max_q_tokens=max(n, n_q), max_topk=nb, lin_mode=hsa.HSA_LIN_NONE, adaptive=True,
                         device=cuda_device)
    kd = K.to(cuda_device)
    ctx.append_kv(kd, kd)
    pos = max(0, n // 2 - n_q) if causal else n
    idx, cnt, gt = ctx.select_blocks_adaptive(q.to(cuda_device), 0.35, 1.0, q_pos0=pos, causal=causal)
    assert ctx.device_status() == 0
    got = Hn.selection_lists(idx, cnt)
    ref, gini, tau = O.adaptive_selection(Hn.f32(q), Hn.f32(K), pos, causal, 0.35, 1.0)
    assert np.allclose(gt.cpu().numpy(), np.stack([gini, tau]), atol=1e-5)
    for h in range(H):
        a, b = list(got[h][0]), list(ref[h][0])
        assert a == sorted(set(a)) and abs(len(a) - len(b)) <= 1
        # (the GPU ranks scores rounded to fp32: neighbours in the order may change places at the boundary)
        assert len(set(a) ^ set(b)) <= 2
    ctx.destroy()


@pytest.mark.parametrize("d,H,n_q,n,group,ex", [
    (128, 3, 129, 64, 128, 0), (128, 2, 2048, 2049, 128, 0), (128, 2, 2049, 2112, 128, 2), (64, 3, 4300, 4000, 128, 0),
    (128, 1, 1100, 9000, 512, 2), (64, 2, 700, 2100, 256, 2), (128, 12, 300, 40000, 128, 0)])
def test_lists_per_query_tile_by_three_launches(d, H, n_q, n, group, ex, cuda_device):
    """Scores of 2, 16, 17 and 34 groups (batches of 16), one and several tiles per group with a short last one, one candidate,
    32, 33 and more, single pages and runs of pages: the lists of the grid-barrier form."""
    from paper_2609_34606_b200 import hsa
    g = torch.Generator().manual_seed(n_q + n)
    K, V, q = _randn(g, n, H, d), _randn(g, n, H, d), _randn(g, n_q, H, d).to(cuda_device)
    blocks = (n + 63) // 64
    budgets = torch.tensor([max(1, blocks // 3 - h) for h in range(H)], dtype=torch.int32, device=cuda_device)
    lists = []
    for grid_form in (False, True):
        ctx = hsa.HSAContext(H, d, max_pages=blocks, max_q_tokens=max(n_q, n), max_topk=blocks, device=cuda_device,
                             grid_barrier_select=grid_form)
        ctx.append_kv(K.to(cuda_device), V.to(cuda_device))
        if ex:
            lists.append(ctx.select_blocks_ex(q, budgets, ex, blocks // 2, None, group_tokens=group))
        else:
            lists.append(ctx.select_blocks(q, budgets, group_tokens=group))
        assert ctx.device_status() == 0
        ctx.destroy()
    (ia, ca), (ib, cb) = lists
    assert torch.equal(ca, cb) and int(ca.sum()) > 0
    keep = torch.arange(ia.shape[2], device=cuda_device) < ca[:, :, None]
    assert torch.equal(ia[keep], ib[keep])


@pytest.mark.parametrize("n_q", [3072, 3073])
def test_query_sums_inside_the_clusters(n_q, cuda_device):
    """24 query tiles are the most whose sums the clusters take themselves: lists as in the grid-barrier form."""
    from paper_2609_34606_b200 import hsa
    g = torch.Generator().manual_seed(n_q)
    H, d, n = 5, 128, 20000
    K, q = _randn(g, n, H, d).to(cuda_device), _randn(g, n_q, H, d).to(cuda_device)
    budgets = torch.tensor([1, 0, 17, 64, -1], dtype=torch.int32, device=cuda_device)
    lists = []
    for grid_form in (False, True):
        ctx = hsa.HSAContext(H, d, max_pages=313, max_q_tokens=n, max_topk=313, lin_mode=hsa.HSA_LIN_NONE, device=cuda_device,
                             grid_barrier_select=grid_form)
        ctx.append_kv(K, K)
        idx, cnt = ctx.select_blocks(q, budgets)
        assert ctx.device_status() == 0
        lists.append([r[0].tolist() for r in Hn.selection_lists(idx, cnt)])
        ctx.destroy()
    assert lists[0] == lists[1] and [len(r) for r in lists[0]] == [1, 0, 17, 64, 313]


@pytest.mark.parametrize("d,H,n_q,budgets,gates,causal", [
    (128, 2, 256, (128, 128), "", False), (128, 4, 600, (100, 0, 17, 100), "dim", False), (64, 4, 600, (100, 3, 100, 99), "head", False),
    (128, 2, 100, (128, 1), "", False), (128, 3, 300, (110, 110, 110), "", True), (64, 1, 1, (128,), "", False)])
def test_lists_of_few_items_split_over_ctas(d, H, n_q, budgets, gates, causal, cuda_device):
    """A launch with few (query tile, head) items cuts their lists into parts: against the same lists given
    per query tile, which one CTA walks from end to end (with one tile both calls take the rule, and the
    oracle tests of the split kernel cover it)."""
    from paper_2609_34606_b200 import hsa
    n = 130 * 64 - 11
    g = torch.Generator().manual_seed(n_q + H)
    K, V, q = _randn(g, n, H, d), _randn(g, n, H, d), _randn(g, n_q, H, d).to(cuda_device)
    kd, vd = K.to(cuda_device), V.to(cuda_device)
    ctx = hsa.HSAContext(H, d, max_pages=130, max_q_tokens=n, max_topk=128, device=cuda_device, causal=causal)
    n0 = n - n_q
    ctx.append_kv(kd[:n0], vd[:n0])
    ctx.append_kv(kd[n0:], vd[n0:])
    pos = n0 if causal else n
    idx, cnt = ctx.select_blocks(q, torch.tensor(budgets, dtype=torch.int32, device=cuda_device), q_pos0=pos, causal=causal)
    gl = gs = None
    if gates:
        shape = (n_q, H, d) if gates == "dim" else (n_q, H)
        gl, gs = _randn(g, *shape).to(cuda_device), _randn(g, *shape).to(cuda_device)
    for _ in range(2):  # (the tickets are back at zero for the second launch)
        out = ctx.forward(q, idx, cnt, q_pos0=pos, causal=causal, g_lin=gl, g_sp=gs)
    # several groups never take the rule: the same list for every tile
    tiles = (n_q + 127) // 128
    many = ctx.forward(q, idx.expand(H, tiles, 128).contiguous(), cnt.expand(H, tiles).contiguous(), q_pos0=pos, causal=causal,
                       group_tokens=128, g_lin=gl, g_sp=gs)
    assert ctx.device_status() == 0
    a, b = out.double(), many.double()
    # the parts take their exponent references from other keys: weights round to bf16 differently
    assert float((a - b).norm() / b.norm()) <= BF16_REL
    ctx.destroy()


@pytest.mark.parametrize("code", [-5, -6])
def test_counters_of_split_lists_start_over_with_the_status_word(code, cuda_device):
    """A part of a split list that gives up draws no ticket; reading the status word puts the counters back (written
    here by the host, as such a launch leaves them), so that the next launch merges all of its parts."""
    from paper_2609_34606_b200 import hsa
    H, d, n, n_q = 2, 128, 130 * 64, 200
    g = torch.Generator().manual_seed(3)
    ctx = hsa.HSAContext(H, d, max_pages=130, max_q_tokens=n, max_topk=128, device=cuda_device, split_blocks=4)
    ctx.append_kv(_randn(g, n, H, d).to(cuda_device), _randn(g, n, H, d).to(cuda_device))
    q = _randn(g, n_q, H, d).to(cuda_device)
    idx, cnt = ctx.select_blocks(q, torch.full((H,), 128, dtype=torch.int32, device=cuda_device))
    want = ctx.forward(q, idx, cnt)
    assert ctx.device_status() == 0
    tickets = (n + 127) // 128 * H  # the last words of the workspace, in whole 256 bytes
    words = ctx.workspace.view(torch.int32)
    end = hsa.hsa_query_sizes(ctx.cfg).workspace // 4 - (4 * tickets + 255) // 256 * 64
    assert words[end:end + tickets].abs().sum().item() == 0
    words[end:end + tickets] = 1
    words[hsa.hsa_workspace_layout(ctx.ctx)[0] // 4] = code
    assert ctx.device_status() == code
    assert words[end:end + tickets].abs().sum().item() == 0
    out = ctx.forward(q, idx, cnt)
    assert ctx.device_status() == 0 and torch.equal(out, want)
    ctx.destroy()


def test_forwards_of_short_lists_on_two_streams(cuda_device):
    """Forwards of one context with few items that run at the same time on two streams do not disturb each other."""
    from paper_2609_34606_b200 import hsa
    H, d, n, n_q = 2, 128, 130 * 64, 256
    g = torch.Generator().manual_seed(9)
    ctx = hsa.HSAContext(H, d, max_pages=130, max_q_tokens=n, max_topk=128, device=cuda_device)
    ctx.append_kv(_randn(g, n, H, d).to(cuda_device), _randn(g, n, H, d).to(cuda_device))
    q = [_randn(g, n_q, H, d).to(cuda_device) for _ in range(2)]
    idx, cnt = ctx.select_blocks(q[0], torch.full((H,), 128, dtype=torch.int32, device=cuda_device))
    streams = [torch.cuda.Stream(cuda_device) for _ in range(2)]
    torch.cuda.synchronize()

    def run(i, out):
        with torch.cuda.stream(streams[i]):
            ctx.forward(q[i], idx, cnt, out=out)

    want = [torch.empty_like(x) for x in q]
    for i in range(2):  # one after the other
        run(i, want[i])
        torch.cuda.synchronize()
    outs = [[torch.empty_like(x) for _ in range(20)] for x in q]
    for k in range(20):
        for i in range(2):
            run(i, outs[i][k])
    torch.cuda.synchronize()
    assert ctx.device_status() == 0
    assert all(torch.equal(o, want[i]) for i in range(2) for o in outs[i])
    ctx.destroy()


@pytest.mark.parametrize("d,H,n_q,cnt,gates", [(128, 2, 100, (128, 7), ""), (64, 1, 1, (128,), "head"), (128, 1, 128, (24,), "dim"),
                                               (128, 4, 600, (9, 127, 16, 0), ""), (64, 16, 200, (64,) * 16, "dim")])
def test_lists_of_few_items_against_64_bits(d, H, n_q, cnt, gates, cuda_device):
    """Lists split over the CTAs of a cluster (2, 4 and 8 of them; lists too short for as many parts, or for any)
    against the oracle on the same lists."""
    from paper_2609_34606_b200 import hsa
    n = 130 * 64 - 11
    g = torch.Generator().manual_seed(n_q + d)
    K, V, q = _randn(g, n, H, d), _randn(g, n, H, d), _randn(g, n_q, H, d)
    ctx = hsa.HSAContext(H, d, max_pages=130, max_q_tokens=n, max_topk=128, device=cuda_device)
    ctx.append_kv(K.to(cuda_device), V.to(cuda_device))
    qd = q.to(cuda_device)
    idx, num = ctx.select_blocks(qd, torch.tensor(cnt, dtype=torch.int32, device=cuda_device))
    gl = gs = gl_n = gs_n = None
    if gates:
        shape = (n_q, H, d) if gates == "dim" else (n_q, H)
        gl, gs = _randn(g, *shape), _randn(g, *shape)
        gl_n, gs_n = Hn.f64(gl), Hn.f64(gs)
        gl, gs = gl.to(cuda_device), gs.to(cuda_device)
    out = ctx.forward(qd, idx, num, g_lin=gl, g_sp=gs)
    assert ctx.device_status() == 0
    rows = sorted({0, n_q // 2, n_q - 1})
    ref = O.hsa_forward(Hn.f32(q), Hn.f32(K), Hn.f32(V), n, False, Hn.selection_lists(idx, num), 0, gl_n, gs_n, 0, rows=rows)["out"]
    got = Hn.f64(out)[rows]
    ref = ref[rows]
    # bf16 weights (2^-9 each, of random sign) and phi(q), and one rounding of the result
    assert np.linalg.norm(got - ref) <= 1.5 * BF16_REL * np.linalg.norm(ref)
    ctx.destroy()


@pytest.mark.parametrize("hot", [6, 60, 98])
@pytest.mark.parametrize("d,causal", [(128, False), (64, False), (128, True)])
def test_safe_pass_of_lists_split_over_a_cluster(d, causal, hot, cuda_device):
    """Later blocks that outscore the first by far, in one part of a list only (the merging one, one in the middle, the
    last): that part is done again with a running maximum, the others are not, and the parts merge."""
    from paper_2609_34606_b200 import hsa
    H, n_q, n = 2, 150, 100 * 64
    g = torch.Generator().manual_seed(d)
    K, V, q = _randn(g, n, H, d), _randn(g, n, H, d), _randn(g, n_q, H, d)
    K[hot * 64:(hot + 2) * 64] *= 24   # scores up to some 24 * 4 * sqrt(d) / sqrt(d) above the others
    q = q * 4
    ctx = hsa.HSAContext(H, d, max_pages=100, max_q_tokens=n, max_topk=100, device=cuda_device, causal=causal)
    n0 = n - n_q
    ctx.append_kv(K[:n0].to(cuda_device), V[:n0].to(cuda_device))
    ctx.append_kv(K[n0:].to(cuda_device), V[n0:].to(cuda_device))
    qd, pos = q.to(cuda_device), n0 if causal else n
    idx, cnt = ctx.select_blocks(qd, torch.full((H,), -1, dtype=torch.int32, device=cuda_device), q_pos0=pos, causal=causal)
    out = ctx.forward(qd, idx, cnt, q_pos0=pos, causal=causal, flags=hsa.HSA_FWD_NO_LINEAR)
    redone = ctx.safe_pass_tiles()
    assert ctx.device_status() == 0 and 0 < redone <= 4 * 2
    ref = O.dense_attention(Hn.f32(q), Hn.f32(K), Hn.f32(V), pos, causal)
    # (peaked rows: a weight is one bf16 rounding, and so is the result)
    assert np.linalg.norm(Hn.f64(out) - ref) <= 2 * BF16_REL * np.linalg.norm(ref)
    ctx.destroy()


def test_state_views_are_the_callers_own(cuda_device):
    """What a caller does to the shape or the flags of a state view stays with that view; the memory is shared."""
    from paper_2609_34606_b200 import hsa
    ctx = hsa.HSAContext(2, 64, max_pages=4, max_q_tokens=128, max_topk=4, device=cuda_device)
    x = torch.randn(100, 2, 64, device=cuda_device).to(torch.bfloat16)
    ctx.append_kv(x, x)
    for name, shape in (("S", (2, 64, 64)), ("z", (2, 64)), ("ksum", (2, 4, 64))):
        view = getattr(ctx, name)
        view.unsqueeze_(0).requires_grad_()
        again = getattr(ctx, name)
        assert tuple(again.shape) == shape and not again.requires_grad and again.data_ptr() == view.data_ptr()
    ctx.destroy()


@pytest.mark.parametrize("flags", [1, 2, 0])
def test_gates_with_a_dim_stride_beyond_32_bits(flags, cuda_device):
    """Per-dim gates whose dims lie 2^24 and more elements apart: offsets inside a row need 64 bits, in the kernel of
    both branches and in the one of the linear branch alone."""
    from paper_2609_34606_b200 import hsa
    H, d, n = 2, 128, 130
    step = (1 << 24) + (1 << 18)
    g = torch.Generator().manual_seed(flags)
    ctx = hsa.HSAContext(H, d, max_pages=3, max_q_tokens=n, max_topk=3, device=cuda_device)
    x, q = _randn(g, n, H, d).to(cuda_device), _randn(g, n, H, d).to(cuda_device)
    ctx.append_kv(x, x)
    idx, cnt = ctx.select_blocks(q, torch.full((H,), -1, dtype=torch.int32, device=cuda_device))
    near = _randn(g, n, H, d).to(cuda_device)
    far = torch.empty((d - 1) * step + n * H, dtype=torch.bfloat16, device=cuda_device).as_strided((n, H, d), (H, 1, step))
    far.copy_(near)
    want = ctx.forward(q, idx, cnt, g_lin=near, g_sp=near, flags=flags)
    out = ctx.forward(q, idx, cnt, g_lin=far, g_sp=far, flags=flags)
    assert ctx.device_status() == 0
    assert float((out.double() - want.double()).norm()) <= BF16_REL * float(want.double().norm())
    ctx.destroy()


@pytest.mark.parametrize("d,causal", [(64, False), (128, False), (128, True)])
def test_large_gates_over_a_small_denominator(d, causal, cuda_device):
    """Gates that are used as given, 1e7 and more, on rows whose phi(q) . z is below 1e-32: the gate over the denominator
    alone would be beyond fp32, the result is not; per token and head as per dim."""
    from paper_2609_34606_b200 import hsa
    H, n = 2, 200
    g = torch.Generator().manual_seed(d)
    V = _randn(g, n, H, d)
    K, q = torch.zeros_like(V), torch.full_like(V, -84.0)
    ctx = hsa.HSAContext(H, d, max_pages=4, max_q_tokens=n, max_topk=4, causal=causal, device=cuda_device)
    ctx.append_kv(K.to(cuda_device), V.to(cuda_device))
    qd, pos = q.to(cuda_device), 0 if causal else n
    idx, cnt = ctx.select_blocks(qd, torch.full((H,), -1, dtype=torch.int32, device=cuda_device), q_pos0=pos, causal=causal)
    gl = (torch.rand(n, H, generator=g) * 9e7 + 1e7).to(torch.bfloat16)
    assert float(gl.min()) / (n * d * np.exp(-84.0)) > torch.finfo(torch.float32).max  # (phi(0) = 1)
    gs = torch.zeros(n, H, dtype=torch.bfloat16)
    gates = lambda wide: {k: (x[:, :, None].expand(n, H, d).contiguous() if wide else x).to(cuda_device) for k, x in (("g_lin", gl), ("g_sp", gs))}
    per_head, per_dim = (ctx.forward(qd, idx, cnt, q_pos0=pos, causal=causal, **gates(wide)).double().cpu() for wide in (False, True))
    assert ctx.device_status() == 0
    # every key weighs the same: the branch is the mean of the visible values
    vd = V.double()
    mean = vd.cumsum(0) / torch.arange(1, n + 1).view(n, 1, 1) if causal else vd.mean(0, keepdim=True).expand(n, H, d)
    ref = gl.double()[:, :, None] * mean
    for out in (per_head, per_dim):
        assert float((out - ref).norm()) <= BF16_REL * float(ref.norm())
    ctx.destroy()


@pytest.mark.parametrize("hot", [False, True])
@pytest.mark.parametrize("form", ["plain", "causal", "linformer", "workspace", "cluster", "causal cluster"])
@pytest.mark.parametrize("d", [64, 128])
def test_gate_tiles_in_every_instance(d, form, hot, cuda_device):
    """Per-dim gates as tiles in each instance of the forward kernel, beside causal partials, in merged lists and in
    tiles that are done again with a running maximum: against the merge of the branches as the same kernel gives
    them without gates."""
    from paper_2609_34606_b200 import hsa
    if form == "linformer" and d == 64:
        pytest.skip("the Linformer form has head_dim 128")
    H, n, causal = 3, 60 * 64, "causal" in form
    n_q = 150 if "cluster" in form else 300
    g = torch.Generator().manual_seed(d + len(form))
    rand = lambda *s: _randn(g, *s).to(cuda_device)
    opt = {}
    if form == "linformer":
        opt = dict(lin_mode=hsa.HSA_LIN_LINFORMER, lin_rank=64, lin_seg_tokens=n, e_k=rand(H, n, 64) * 0.02, e_v=rand(H, n, 64) * 0.02)
    budget = 10 if form in ("plain", "causal") else 50
    ctx = hsa.HSAContext(H, d, max_pages=60, max_q_tokens=n, max_topk=budget, device=cuda_device, gate_act=1, causal=causal,
                         split_blocks=16 if form == "workspace" else 0, **opt)
    K, V, q = rand(n, H, d), rand(n, H, d), rand(n_q, H, d)
    if hot:
        K[20 * 64:22 * 64] *= 24
        q *= 4
    n0 = n - n_q if causal else 0
    for lo, hi in ((0, n0), (n0, n)):
        if hi > lo:
            ctx.append_kv(K[lo:hi], V[lo:hi])
    pos = n0 if causal else n
    # lists that hold the outscoring blocks, behind ordinary ones
    idx, cnt = ctx.alloc_selection(n_q)
    idx[:, 0] = torch.arange(60 - budget, 60) if budget < 50 and not hot else torch.arange(budget) + (14 if budget < 50 else 0)
    cnt.fill_(budget)
    gl, gs = rand(n_q, H, d), rand(n_q, H, d)
    run = lambda **kw: ctx.forward(q, idx, cnt, q_pos0=pos, causal=causal, **kw).double()
    ctx.safe_pass_tiles()
    out = run(g_lin=gl, g_sp=gs)
    assert (ctx.safe_pass_tiles() > 0) == hot
    lin, sp = run(flags=hsa.HSA_FWD_NO_SPARSE), run(flags=hsa.HSA_FWD_NO_LINEAR)
    assert ctx.device_status() == 0
    a, b = torch.sigmoid(gl.double()) * lin, torch.sigmoid(gs.double()) * sp
    # each branch and the result are rounded once, and a branch alone may take its exponent references from other
    # keys, so that its bf16 weights round differently (2^-9 each, of random sign, of a sum of many)
    assert float((out - a - b).norm()) <= 1.5 * BF16_REL * float((a + b).norm())
    ctx.destroy()


@pytest.mark.parametrize("H,tokens,rank", [(20, 600, 256), (12, 300, 128), (12, 513, 256), (3, 1088, 64), (2, 2049, 192), (1, 64, 64)])
def test_compressed_segments_by_clusters(H, tokens, rank, cuda_device):
    """A tile's token blocks in one CTA (many tiles, few blocks) and over clusters of 2, 4 and 8, parts of unequal length, a
    last block of one token, a half-filled last tile: compressed rows against 64 bits, two segments."""
    from paper_2609_34606_b200 import hsa
    d = 128
    g = torch.Generator().manual_seed(tokens)
    scale = tokens ** -0.5
    e_k, e_v = ((torch.randn(H, tokens, rank, generator=g) * scale).to(torch.bfloat16) for _ in range(2))
    ctx = hsa.HSAContext(H, d, max_pages=(2 * tokens + 63) // 64, max_q_tokens=tokens, max_topk=1, device=cuda_device,
                         lin_mode=hsa.HSA_LIN_LINFORMER, lin_rank=rank, lin_seg_tokens=tokens, e_k=e_k.to(cuda_device),
                         e_v=e_v.to(cuda_device))
    for seg in range(2):
        k, v = _randn(g, tokens, H, d), _randn(g, tokens, H, d)
        ctx.append_kv(k.to(cuda_device), v.to(cuda_device))
        assert ctx.device_status() == 0
        pages = rank // 64
        for pool, e, x in ((ctx.kc_pool, e_k, k), (ctx.vc_pool, e_v, v)):
            got = pool.view(torch.bfloat16).view(-1, H, 64, d)[seg * pages:(seg + 1) * pages].double().cpu()
            got = got.permute(1, 0, 2, 3).reshape(H, rank, d)
            ref = torch.einsum("htr,thd->hrd", e.double(), x.double())
            assert float((got - ref).norm()) <= BF16_REL * float(ref.norm())
    ctx.destroy()


@pytest.mark.parametrize("H,tokens,rank", [(4, 1216, 256), (4, 1217, 256), (2, 2049, 256), (12, 3072, 256), (12, 3073, 256), (12, 3900, 256),
                                           (16, 2000, 256), (16, 2900, 256)])
def test_segments_at_the_edges_of_the_launch_rules(H, tokens, rank, cuda_device):
    """Segments on both sides of the lengths that are split over clusters (of 2, 4 and 8 CTAs), with the page write in either of
    its forms beside them and with and without room on their SMs: compressed rows against 64 bits, pages bit for
    bit, key sums."""
    from paper_2609_34606_b200 import hsa
    d = 128
    g = torch.Generator(device=cuda_device).manual_seed(tokens)
    rand = lambda *s: torch.randn(*s, generator=g, device=cuda_device)
    e_k, e_v = ((rand(H, tokens, rank) * tokens ** -0.5).to(torch.bfloat16) for _ in range(2))
    blocks = (tokens + 63) // 64
    ctx = hsa.HSAContext(H, d, max_pages=blocks, max_q_tokens=tokens, max_topk=1, device=cuda_device,
                         lin_mode=hsa.HSA_LIN_LINFORMER, lin_rank=rank, lin_seg_tokens=tokens, e_k=e_k, e_v=e_v)
    ctx.k_pool.fill_(0xFF)
    ctx.v_pool.fill_(0xFF)
    k, v = rand(tokens, H, d).to(torch.bfloat16), rand(tokens, H, d).to(torch.bfloat16)
    ctx.append_kv(k, v)
    assert ctx.device_status() == 0
    pad = torch.zeros(blocks * 64 - tokens, H, d, dtype=torch.bfloat16, device=cuda_device)
    for pool, cpool, e, x in ((ctx.k_pool, ctx.kc_pool, e_k, k), (ctx.v_pool, ctx.vc_pool, e_v, v)):
        got = cpool.view(torch.bfloat16).view(-1, H, 64, d)[:rank // 64].double().permute(1, 0, 2, 3).reshape(H, rank, d)
        ref = torch.einsum("htr,thd->hrd", e.double(), x.double())
        # sums in 32 bits are off by no more than 2^-18 of the result here, rounding to bf16 by 2^-9.3 (2-norms): together
        # hardly more than the rounding alone
        alone = float((ref.to(torch.bfloat16).double() - ref).norm())
        assert float((got - ref).norm()) <= (1 + 2.0 ** -8) * alone <= BF16_REL * float(ref.norm())
        want = torch.cat([x, pad]).view(blocks, 64, H, d).permute(0, 2, 1, 3)
        assert torch.equal(pool.view(torch.bfloat16).view(-1, H, 64, d)[:blocks], want)
    ref = torch.cat([k, pad]).double().view(blocks, 64, H, d).sum(1).permute(1, 0, 2)
    # fp32 sums of 64 values: every addition rounds by 2^-24 of a partial sum of the order of the result
    assert float((ctx.ksum.double() - ref).norm()) <= 2.0 ** -24 * 12 * float(ref.norm())
    ctx.destroy()


@pytest.mark.parametrize("H,tokens", [(3, 300), (3, 1000), (4, 1300), (12, 3200), (1, 2100)])
def test_compression_that_gives_up_leaves_the_context_usable(H, tokens, cuda_device):
    """The products of the compression kernel are given up with copies in flight (a wait limit of one nanosecond; one CTA per tile
    with fewer and more blocks than ring stages, clusters of 2, 4 and 8): it ends by itself and says so, and the segment
    appended again is what it was."""
    from paper_2609_34606_b200 import hsa
    d, rank = 128, 256
    g = torch.Generator(device=cuda_device).manual_seed(tokens)
    rand = lambda *s: torch.randn(*s, generator=g, device=cuda_device).to(torch.bfloat16)
    ctx = hsa.HSAContext(H, d, max_pages=(tokens + 63) // 64, max_q_tokens=tokens, max_topk=1, device=cuda_device,
                         lin_mode=hsa.HSA_LIN_LINFORMER, lin_rank=rank, lin_seg_tokens=tokens, e_k=rand(H, tokens, rank),
                         e_v=rand(H, tokens, rank))
    k, v = rand(tokens, H, d), rand(tokens, H, d)
    ctx.append_kv(k, v)
    assert ctx.device_status() == 0
    want = ctx.kc_pool.clone(), ctx.vc_pool.clone(), ctx.ksum.clone(), ctx.k_pool.clone()
    ctx.set_wait_limit_ns(1)
    for _ in range(3):
        ctx.rewind(0)
        ctx.append_kv(k, v)
        assert ctx.device_status() == hsa.HSA_ERR_DEVICE_TIMEOUT
    ctx.set_wait_limit_ns(2_000_000_000)
    ctx.rewind(0)
    ctx.append_kv(k, v)
    assert ctx.device_status() == 0
    for a, b in zip((ctx.kc_pool, ctx.vc_pool, ctx.ksum, ctx.k_pool), want):
        assert torch.equal(a, b)
    ctx.destroy()


@pytest.mark.parametrize("H,n", [(1, 1), (12, 3136), (12, 4680), (16, 4680)])
def test_page_write_takes_rows_one_by_one_or_at_once(H, n, cuda_device):
    """Contexts without a linear state: few CTAs, more than fit at once with all rows asked for, as many as fit one row at a
    time, and more.  Pages bit for bit, key sums."""
    from paper_2609_34606_b200 import hsa
    d, blocks = 128, (n + 63) // 64
    g = torch.Generator(device=cuda_device).manual_seed(n)
    k, v = (torch.randn(n, H, d, generator=g, device=cuda_device).to(torch.bfloat16) for _ in range(2))
    ctx = hsa.HSAContext(H, d, max_pages=blocks, max_q_tokens=n, max_topk=1, lin_mode=hsa.HSA_LIN_NONE, device=cuda_device)
    ctx.append_kv(k, v)
    assert ctx.device_status() == 0
    pad = torch.zeros(blocks * 64 - n, H, d, dtype=torch.bfloat16, device=cuda_device)
    for pool, x in ((ctx.k_pool, k), (ctx.v_pool, v)):
        assert torch.equal(pool.view(torch.bfloat16).view(-1, H, 64, d), torch.cat([x, pad]).view(blocks, 64, H, d).permute(0, 2, 1, 3))
    ref = torch.cat([k, pad]).double().view(blocks, 64, H, d).sum(1).permute(1, 0, 2)
    assert float((ctx.ksum.double() - ref).norm()) <= 2.0 ** -24 * 12 * float(ref.norm())  # (as above)
    ctx.destroy()


@pytest.mark.parametrize("n,group", [(700, 0), (64 * 40, 0), (700, 128)])
def test_adaptive_lists_end_in_zeros(n, group, cuda_device):
    """What a list buffer held before the call is gone, behind the list as well."""
    from paper_2609_34606_b200 import hsa
    H, d, n_q = 3, 128, 200
    g = torch.Generator().manual_seed(n)
    blocks = (n + 63) // 64
    ctx = hsa.HSAContext(H, d, max_pages=blocks, max_q_tokens=n, max_topk=blocks + 3, device=cuda_device, adaptive=True)
    ctx.append_kv(_randn(g, n, H, d).to(cuda_device), _randn(g, n, H, d).to(cuda_device))
    q = _randn(g, n_q, H, d).to(cuda_device)
    idx, cnt, gt = ctx.select_blocks_adaptive(q, 0.2, 0.4, group_tokens=group)
    dirty, counts = torch.full_like(idx, 77), torch.full_like(cnt, 77)
    hsa.hsa_select_blocks_adaptive(ctx.ctx, q, n, False, 0.2, 0.4, group, dirty, counts, None)
    assert torch.equal(dirty, idx) and torch.equal(counts, cnt)
    behind = torch.arange(idx.shape[2], device=cuda_device) >= cnt[:, :, None]
    assert int(idx[behind].abs().sum()) == 0 and bool(behind.any()) and int(cnt.min()) > 0
    ctx.destroy()


def _causal_branches(q, K, V, n0, idx, cnt, group, relu):
    """Both branches of a causal forward in 64 bits on the device, [n, H, d] each: q and the chunk start at position n0."""
    n, H, d = q.shape
    lin, sp = torch.empty(n, H, d, dtype=torch.float64, device=q.device), torch.empty(n, H, d, dtype=torch.float64, device=q.device)
    phi = lambda x: x.clamp(min=0) if relu else torch.where(x > 0, x + 1, x.exp())
    seen = torch.arange(K.shape[0], device=q.device)[None] <= n0 + torch.arange(n, device=q.device)[:, None]
    for h in range(H):
        qh, kh, vh = q[:, h].double(), K[:, h].double(), V[:, h].double()
        A = (phi(qh) @ phi(kh).T) * seen
        lin[:, h] = A @ vh / (A.sum(1, keepdim=True) + (1e-6 if relu else 0.0))
        chosen = torch.zeros_like(seen)
        for g in range(cnt.shape[1]):
            rows = slice(g * group, (g + 1) * group) if group else slice(0, n)
            for b in idx[h, g, :int(cnt[h, g])].tolist():
                chosen[rows, 64 * b:64 * b + 64] = True
        s = (qh @ kh.T * d ** -0.5).masked_fill(~(seen & chosen), -torch.inf)
        sp[:, h] = torch.softmax(s, 1) @ vh
    return lin, sp


@pytest.mark.parametrize("H,n0,n,topk,group,relu", [
    (2, 70, 769, -1, 0, 0), (12, 33, 1560, 6, 0, 0), (12, 100, 1500, 9, 128, 0), (16, 64, 1153, 4, 0, 1), (12, 640, 896, 8, 0, 0)])
def test_causal_chunks_of_many_tiles_with_both_branches(H, n0, n, topk, group, relu, cuda_device):
    """Terms, sums over page groups or steps through all pages, products, and the forward that takes the partials as tiles, more
    than one wave of them: few items (clusters), 156 and 160 items, lists per query tile, against 64 bits."""
    from paper_2609_34606_b200 import hsa
    d = 128
    g = torch.Generator(device=cuda_device).manual_seed(n)
    K, V, q = (torch.randn(m, H, d, generator=g, device=cuda_device).to(torch.bfloat16) for m in (n0 + n, n0 + n, n))
    blocks = (n0 + n + 63) // 64
    ctx = hsa.HSAContext(H, d, max_pages=blocks, max_q_tokens=n, max_topk=blocks, causal=True, device=cuda_device, feature_map=relu,
                         page_order=torch.arange(blocks - 1, -1, -1, dtype=torch.int32))
    ctx.k_pool.fill_(0xFF)
    ctx.v_pool.fill_(0xFF)
    ctx.append_kv(K[:n0], V[:n0])
    ctx.append_kv(K[n0:], V[n0:])
    idx, cnt = ctx.select_blocks(q, torch.full((H,), topk, dtype=torch.int32, device=cuda_device), q_pos0=n0, causal=True, group_tokens=group)
    idx[:, :, 0] = 0  # (the first block is one every query sees, so that no row is without a key)
    cnt.clamp_(min=1)
    out = ctx.forward(q, idx, cnt, q_pos0=n0, causal=True, group_tokens=group).double()
    assert ctx.device_status() == 0
    lin, sp = _causal_branches(q, K, V, n0, idx, cnt, group, relu)
    # (the sparse branch's weights are bf16 as well as the result: two roundings, one of them of a sum's terms)
    assert float((out - lin - sp).norm()) <= 1.5 * BF16_REL * float((lin + sp).norm())
    ctx.destroy()


@pytest.mark.parametrize("hot", [False, True])
@pytest.mark.parametrize("gates", ["none", "sigmoid per head", "raw per head", "sigmoid strided per dim"])
@pytest.mark.parametrize("group", [0, 128])
def test_causal_partials_as_tiles(group, gates, hot, cuda_device):
    """The causal partials as tiles beside every form of gate that is none itself, in lists split over a cluster and in whole ones
    (per query tile), and where a tile is done again with a running maximum and asks for its partials a second time."""
    from paper_2609_34606_b200 import hsa
    H, d, n0, n = 2, 128, 58 * 64, 150
    g = torch.Generator(device=cuda_device).manual_seed(len(gates))
    rand = lambda *s: torch.randn(*s, generator=g, device=cuda_device).to(torch.bfloat16)
    K, V, q = rand(n0 + n, H, d), rand(n0 + n, H, d), rand(n, H, d)
    if hot:
        K[30 * 64:32 * 64] *= 24  # scores far above those of the blocks in front
        q *= 4
    ctx = hsa.HSAContext(H, d, max_pages=61, max_q_tokens=n0, max_topk=50, causal=True, device=cuda_device,
                         gate_act=0 if gates == "raw per head" else 1)
    ctx.append_kv(K[:n0], V[:n0])
    ctx.append_kv(K[n0:], V[n0:])
    idx, cnt = ctx.alloc_selection(n, group)
    idx[:, :] = torch.arange(50) + 8
    cnt.fill_(50)
    gl = gs = None
    if gates == "sigmoid strided per dim":
        gl, gs = rand(n, H, 2 * d)[:, :, ::2], rand(n, H, 2 * d)[:, :, ::2]
    elif gates != "none":
        gl, gs = rand(n, H), rand(n, H)
    ctx.safe_pass_tiles()
    out = ctx.forward(q, idx, cnt, q_pos0=n0, causal=True, group_tokens=group, g_lin=gl, g_sp=gs).double()
    assert (ctx.safe_pass_tiles() > 0) == hot and ctx.device_status() == 0
    lin, sp = _causal_branches(q, K, V, n0, idx, cnt, group, 0)

    def weight(x):
        if x is None:
            return 1.0
        x = x.double() if x.dim() == 3 else x.double()[:, :, None]
        return x if gates == "raw per head" else torch.sigmoid(x)

    a, b = weight(gl) * lin, weight(gs) * sp
    # (hot rows are peaked: a weight is one bf16 rounding, and so is the result)
    assert float((out - a - b).norm()) <= 2 * BF16_REL * float((a.square() + b.square()).sum().sqrt())
    ctx.destroy()
