"""Accumulating an f32 product (dH and dW with the accumulate flags) is one f32 addition per element, subnormal numbers
included: the sums are the bits of the separately computed product plus the buffer, rounded once."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("variant", [0, 1, 2])
def test_accumulation_keeps_subnormal_sums(variant):
    from paper_2606_29758_gb300 import _binding as B
    M = N = 512
    K = 128
    g = torch.Generator(device="cuda").manual_seed(3)

    def bits(lo, hi, shape):
        return torch.randint(lo, hi, shape, device="cuda", generator=g, dtype=torch.int32)
    # one nonzero per row of A, a power of two: every product is exact, 2^-134 to 2^-118
    A = torch.zeros(M, K, device="cuda")
    A[torch.arange(M, device="cuda"), bits(0, K, (M,)).long()] = 2.0 ** -64
    Bm = torch.ldexp(1 + bits(0, 128, (N, K)).float() / 128, bits(-70, -54, (N, K)))
    Bm = torch.where(bits(0, 2, (N, K)) == 0, Bm, -Bm)
    A, Bm = A.bfloat16(), Bm.bfloat16()
    before = (bits(0, 1 << 25, (M, N)) | (bits(0, 2, (M, N)) << 31)).view(torch.float32)   # up to 2^-123
    ws = torch.empty(256, dtype=torch.uint8, device="cuda")
    product, total = torch.empty(M, N, device="cuda"), before.clone()
    B.ps_diag_gemm_bf16(M, N, K, 0, 0, A, K, Bm, K, product, N, 0, ws, variant)
    B.ps_diag_gemm_bf16(M, N, K, 0, 0, A, K, Bm, K, total, N, 1, ws, variant)
    assert B.ps_workspace_status(ws)[0] == B.PS_OK
    p, c, t = (x.cpu().numpy() for x in (product, before, total))
    assert np.array_equal(p, (A.double() @ Bm.double().t()).cpu().numpy())
    want = (p.astype(np.float64) + c.astype(np.float64)).astype(np.float32)   # exact in 64 bits, rounded once
    small = (np.abs(want) < 2.0 ** -126) & (want != 0)
    assert small.sum() > 10000
    assert np.array_equal(t.view(np.int32), want.view(np.int32))
