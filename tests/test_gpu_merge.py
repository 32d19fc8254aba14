"""The merge of a row's vocabulary partials: the bits of the sum in vocabulary order.

A partial is the (max, sum of 2^(x - max)) of 128 columns. A shard of 128 columns has one, so the statistics of
such shards are the whole head's partials; their merge is restated here in the order that the library promises, one
fused multiply-add after another, and compared bit for bit.
"""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _stats(H, W, tok, v0=0):
    from paper_2606_29758_gb300 import _binding as B
    (N, d), V = H.shape, W.shape[0]
    stats, ztok = torch.empty(N, 2, device="cuda"), torch.empty(N, device="cuda")
    ws = torch.empty(B.ps_lmhead_logit_stats_workspace_size(N, d, V, B.PS_DTYPE_BF16), dtype=torch.uint8, device="cuda")
    B.ps_lmhead_logit_stats(N, d, V, v0, B.PS_DTYPE_BF16, H, W, tok, stats, ztok, ws)
    assert B.ps_workspace_status(ws)[0] == B.PS_OK
    return stats


# blocks of 8, 16 and 32 rows, each with a last block that is not full, and rows of one chunk of parts, of several that
# are all held, and of more than the ring holds
@pytest.mark.parametrize("N,V", [(9, 1000), (3000, 1000), (37, 30003), (13, 200003), (2501, 12000), (2501, 50003),
                                 (5003, 50003), (11001, 5003), (11001, 20003)])
def test_partials_are_merged_in_vocabulary_order(N, V):
    g = torch.Generator(device="cuda").manual_seed(N)
    H = torch.randn(N, 64, device="cuda", generator=g).bfloat16()
    W = (torch.randn(V, 64, device="cuda", generator=g) * 0.3).bfloat16()
    tok = torch.zeros(N, dtype=torch.int32, device="cuda")
    whole = _stats(H, W, tok).cpu().numpy()
    parts = torch.stack([_stats(H, W[v0:v0 + 128], tok, v0) for v0 in range(0, V, 128)])
    m = parts[:, :, 0].amax(0)
    e = torch.exp2(parts[:, :, 0] - m).cpu().numpy().astype(np.float64)
    y = parts[:, :, 1].cpu().numpy().astype(np.float64)
    S = np.zeros(N, np.float32)
    for k in range(len(y)):
        S = (y[k] * e[k] + S).astype(np.float32)   # the product is exact in 64 bits
    assert np.array_equal(whole[:, 0], m.cpu().numpy())
    assert np.array_equal(whole[:, 1], S)
