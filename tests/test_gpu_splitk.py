"""dH of few rows: the vocabulary (its K loop) split over the CTAs of a cluster.

dH = dZ W with dZ = coef (onehot - exp(z - lse)) rounded to bf16, against the same product in float64
from torch's logits. A logit that differs in its last bits may round an element of dZ to the neighbouring
bf16 value, one ulp (2^-8 relative at most) away, and the f32 accumulation over V / 16 steps errs by at
most 2 ulps of a partial sum each, so an entry is off by at most (2^-8 + 2^-22 V / 16) sum_v |dZ_iv W_vc|.
The sizes lie around the tile's rows (128 in one half, 256) and columns, with vocabularies that leave the
ranks unequal shares of k-blocks and a ragged last one.
"""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,d,V", [(1, 8, 2000), (127, 256, 1800), (128, 264, 2047), (129, 392, 2048), (256, 520, 5001),
                                   (257, 248, 1857), (700, 1000, 4100), (1100, 1536, 3000), (5000, 264, 2300)])
def test_dh_of_few_rows(N, d, V):
    from paper_2606_29758_gb300 import _binding as B
    g = torch.Generator(device="cuda").manual_seed(N + d + V)
    H = torch.randn(N, d, device="cuda", generator=g).bfloat16()
    W = (torch.randn(V, d, device="cuda", generator=g) * 0.05).bfloat16()
    tok = torch.randint(0, V, (N,), device="cuda", generator=g, dtype=torch.int32)
    coef = torch.randn(N, device="cuda", generator=g)
    z = H.double() @ W.double().t()
    lse = torch.logsumexp(z, 1).float()
    dZ = -torch.exp(z - lse[:, None].double())
    dZ[torch.arange(N, device="cuda"), tok.long()] += 1.0
    dZ = (dZ * coef[:, None].double()).float().bfloat16().double()
    ref = dZ @ W.double()
    bound = (2.0 ** -8 + 2.0 ** -22 * V / 16) * (dZ.abs() @ W.double().abs())
    dH = torch.full((N, d), float("nan"), device="cuda")
    ws = torch.zeros(B.ps_lmhead_ppo_bwd_workspace_size(N, d, V, B.PS_DTYPE_BF16), dtype=torch.uint8, device="cuda")
    B.ps_lmhead_ppo_bwd(N, d, V, B.PS_DTYPE_BF16, H, W, tok, lse, coef, dH, None, 0, ws)
    assert B.ps_workspace_status(ws)[0] == B.PS_OK
    assert ((dH.double() - ref).abs() <= bound + 1e-30).all()
    # the same partials, added to what the buffer holds; and the same bits again
    prior = torch.randn(N, d, device="cuda", generator=g)
    acc = prior.clone()
    B.ps_lmhead_ppo_bwd(N, d, V, B.PS_DTYPE_BF16, H, W, tok, lse, coef, acc, None, B.PS_DH_ACCUMULATE, ws)
    again = torch.empty_like(dH)
    B.ps_lmhead_ppo_bwd(N, d, V, B.PS_DTYPE_BF16, H, W, tok, lse, coef, again, None, 0, ws)
    assert torch.equal(acc, prior + dH) and torch.equal(again, dH)


@pytest.mark.parametrize("N,d,V", [(1300, 128, 1024), (2500, 392, 2000), (4111, 264, 1857), (8000, 136, 300)])
def test_dw_of_a_small_vocabulary(N, d, V):
    # dW = dZ^T H with the rows (its K loop) split over a cluster: the bound of the dH test with N terms per entry;
    # accumulation and reruns exact; and two vocabulary shards give the whole head's bits, whatever their own sizes.
    from paper_2606_29758_gb300 import _binding as B
    g = torch.Generator(device="cuda").manual_seed(N + d + V)
    H = torch.randn(N, d, device="cuda", generator=g).bfloat16()
    W = (torch.randn(V, d, device="cuda", generator=g) * 0.05).bfloat16()
    tok = torch.randint(0, V, (N,), device="cuda", generator=g, dtype=torch.int32)
    coef = torch.randn(N, device="cuda", generator=g)
    z = H.double() @ W.double().t()
    lse = torch.logsumexp(z, 1).float()
    dZ = -torch.exp(z - lse[:, None].double())
    dZ[torch.arange(N, device="cuda"), tok.long()] += 1.0
    dZ = (dZ * coef[:, None].double()).float().bfloat16().double()
    bound = (2.0 ** -8 + 2.0 ** -22 * N / 16) * (dZ.abs().t() @ H.double().abs())
    ws = torch.zeros(B.ps_lmhead_ppo_bwd_workspace_size(N, d, V, B.PS_DTYPE_BF16), dtype=torch.uint8, device="cuda")
    dW = torch.full((V, d), float("nan"), device="cuda")
    B.ps_lmhead_ppo_bwd(N, d, V, B.PS_DTYPE_BF16, H, W, tok, lse, coef, None, dW, 0, ws)
    assert B.ps_workspace_status(ws)[0] == B.PS_OK
    assert ((dW.double() - dZ.t() @ H.double()).abs() <= bound + 1e-30).all()
    prior = torch.randn(V, d, device="cuda", generator=g)
    acc = prior.clone()
    B.ps_lmhead_ppo_bwd(N, d, V, B.PS_DTYPE_BF16, H, W, tok, lse, coef, None, acc, B.PS_DW_ACCUMULATE, ws)
    assert torch.equal(acc, prior + dW)
    cut = V // 3
    shards = torch.full((V, d), float("nan"), device="cuda")
    for v0, Vs in ((0, cut), (cut, V - cut)):
        B.ps_lmhead_ppo_bwd_vocab_shard(N, d, Vs, v0, V, B.PS_DTYPE_BF16, H, W[v0:v0 + Vs], tok, lse, coef, None,
                                        shards[v0:v0 + Vs], 0, ws)
    assert torch.equal(shards, dW)
