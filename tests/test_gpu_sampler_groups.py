"""Cutoffs of large groups: every draw's bucket is found in its tile of 256 steps. Integers against the oracle, at steps
around the tiles' edges and with steps of no mass, and the time beside that of a small group."""
import numpy as np
import pytest
import torch

from oracle.cutoffs import ONE62, sample_cutoffs

pytestmark = pytest.mark.gpu


def _masses(P, T, rng, total=ONE62):
    q = np.zeros((P, T), dtype=np.uint64)
    for p in range(P):
        m = rng.random(T) * (rng.random(T) < 0.6)      # steps of no mass among them
        m[rng.integers(T)] = 1.0
        q[p] = np.floor(m / m.sum() * 0.999 * float(total)).astype(np.uint64)
        q[p, rng.integers(T)] += np.uint64(total - int(q[p].sum(dtype=np.uint64)))
    return q


def _gpu(q, L, K, mode):
    from paper_2606_29758_gb300 import _binding as B
    P, T = q.shape
    H, n = torch.empty(P * K, dtype=torch.int32, device="cuda"), torch.empty(P * K, dtype=torch.int32, device="cuda")
    w = torch.empty(P, T, device="cuda")
    ws = torch.empty(B.ps_sample_cutoffs_workspace_size(P, K, T), dtype=torch.uint8, device="cuda")
    dq, dL = torch.from_numpy(q.view(np.int64)).cuda(), torch.from_numpy(L).cuda()

    def call():
        B.ps_sample_cutoffs(P, K, T, dq, dL, 7, 3, 0, mode, H, n, w, ws)
    call()
    assert B.ps_workspace_status(ws)[0] == B.PS_OK
    return H, n, call


@pytest.mark.parametrize("zero", [False, True])
@pytest.mark.parametrize("P,K,T", [(2, 600, 1), (3, 300, 255), (2, 257, 256), (2, 512, 257), (1, 1000, 1025), (70, 9, 513)])
def test_large_groups(P, K, T, zero):
    from paper_2606_29758_gb300 import _binding as B
    rng = np.random.default_rng(P + K + T)
    q = _masses(P, T, rng, ONE62 // 3 if zero else ONE62)
    L = rng.integers(1, T + 1, size=P * K).astype(np.int32)
    H, n, _ = _gpu(q, L, K, B.PS_MODE_TRUNC_ZERO if zero else B.PS_MODE_TRUNC)
    H_ref, n_ref, _ = sample_cutoffs(q, L, K, 7, 3, mode="trunc_zero" if zero else "trunc")
    assert np.array_equal(H.cpu().numpy(), H_ref)
    assert np.array_equal(n.cpu().numpy(), n_ref)


def test_a_large_group_takes_little_longer_than_a_small_one():
    from paper_2606_29758_gb300 import _binding as B

    def us(K, T=100, reps=200):
        rng = np.random.default_rng(1)
        _, _, call = _gpu(_masses(8, T, rng), np.full(8 * K, T, dtype=np.int32), K, B.PS_MODE_TRUNC)
        best = 1e9
        for _ in range(5):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(reps):
                call()
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b) / reps * 1e3)
        return best
    # passes back to back: at K = 8 the calls themselves may take longer than the kernel
    assert us(512) < 1.8 * us(8) + 5.0
