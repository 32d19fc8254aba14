"""The f32 head's products on the CUDA cores, around the edges of their tiles and of the rules that pick them.

lse, dH and dW against float64 on the same inputs. A product of K terms accumulated in f32, one rounding per
step, errs by at most K 2^-24 of the sum of the terms' magnitudes: e_z = d 2^-24 sum |h w| for a logit. With the
pass's own lse, dZ = coef (onehot - exp(z - lse)) is then off by at most |coef| p (e_z + 2^-21 (1 + |z - lse|))
(the subtraction and the exponential round too) plus 2^-23 |dZ|, and an entry of dH or dW by that error
carried through the product plus its own accumulation. The sum of V exponentials has relative error of at most
V 2^-24 + max e_z + 2^-21, which is the bound on lse beside its rounding to f32. Sizes: one row and one column;
d and V that end inside a 4-vector, a k step and a tile; few tiles (dH and dW split over clusters of 2, 4 and 8) and
hundreds; rows cut into chunks, which must not change dH.
"""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,d,V", [(1, 8, 1), (3, 12, 5), (33, 20, 63), (64, 132, 65), (65, 64, 129), (200, 100, 1001),
                                   (191, 392, 2003), (700, 68, 3001), (129, 768, 4097), (1500, 260, 2050),
                                   (5000, 128, 514),
                                   (2600, 392, 1400)])
def test_products_of_the_f32_head(N, d, V):
    from paper_2606_29758_gb300 import _binding as B
    F = B.PS_DTYPE_F32
    dev = dict(device="cuda")
    g = torch.Generator(device="cuda").manual_seed(N * 3 + d + V)
    H = torch.randn(N, d, generator=g, **dev)
    W = torch.randn(V, d, generator=g, **dev) * 0.1
    tok = torch.randint(0, V, (N,), generator=g, dtype=torch.int32, **dev)
    adv, w = torch.randn(N, generator=g, **dev), torch.rand(N, generator=g, **dev) + 0.5
    u = 2.0 ** -24
    z = H.double() @ W.double().t()
    e_z = d * u * (H.double().abs() @ W.double().abs().t())
    lse_ref = torch.logsumexp(z, 1)
    old = (z.gather(1, tok[:, None].long())[:, 0] - lse_ref).float()
    o = {k: torch.full((N,), float("nan"), **dev) for k in ("lse", "logp", "ratio", "coef", "row_loss")}
    loss = torch.zeros(1, dtype=torch.float64, **dev)
    ws = torch.zeros(B.ps_lmhead_ppo_fwd_workspace_size(N, d, V, F), dtype=torch.uint8, **dev)
    B.ps_lmhead_ppo_fwd(N, d, V, F, H, W, tok, old, adv, w, 0.2, 0.25, loss, *o.values(), ws)
    assert B.ps_workspace_status(ws)[0] == B.PS_OK
    tol = e_z.max(1).values + V * u + 2.0 ** -21 + u * lse_ref.abs()
    assert ((o["lse"].double() - lse_ref).abs() <= tol).all()

    lse, coef = o["lse"].double()[:, None], o["coef"].double()[:, None]
    p = torch.exp(z - lse)
    dZ = -coef * p
    dZ[torch.arange(N, **dev), tok.long()] += coef[:, 0]
    e_dz = coef.abs() * p * (e_z + 2.0 ** -21 * (1.0 + (z - lse).abs())) + 2.0 ** -23 * dZ.abs()
    Hd, Wd = H.double(), W.double()
    ref = {"dH": dZ @ Wd, "dW": dZ.t() @ Hd}
    bound = {"dH": e_dz @ Wd.abs() + (V + 8) * u * (dZ.abs() @ Wd.abs()),
             "dW": e_dz.t() @ Hd.abs() + (N + 8) * u * (dZ.abs().t() @ Hd.abs())}

    def backward(chunk, flags=0, dH=None, dW=None):
        dH = torch.full((N, d), float("nan"), **dev) if dH is None else dH
        dW = torch.full((V, d), float("nan"), **dev) if dW is None else dW
        b = torch.full((B.ps_lmhead_ppo_bwd_workspace_size(N, d, V, F, chunk),), 255, dtype=torch.uint8, **dev)
        B.ps_lmhead_ppo_bwd(N, d, V, F, H, W, tok, o["lse"], o["coef"], dH, dW, flags, b)
        assert B.ps_workspace_status(b)[0] == B.PS_OK
        return {"dH": dH, "dW": dW}

    whole, chunked = backward(N), backward(128)
    for k in ("dH", "dW"):
        assert ((whole[k].double() - ref[k]).abs() <= bound[k] + 1e-30).all(), k
        assert ((chunked[k].double() - ref[k]).abs() <= bound[k] + 1e-30).all(), k
    assert torch.equal(whole["dH"], chunked["dH"])
    prior = {"dH": torch.randn(N, d, generator=g, **dev), "dW": torch.randn(V, d, generator=g, **dev)}
    acc = backward(N, B.PS_DH_ACCUMULATE | B.PS_DW_ACCUMULATE, prior["dH"].clone(), prior["dW"].clone())
    for k in ("dH", "dW"):
        assert torch.equal(acc[k], prior[k] + whole[k]), k
