"""A pass captured into a CUDA graph: the kernels of a call after its first are launched programmatically, and a
replay must give the eager pass's bits (recompute and logit store, f32 and bf16, several backward chunks)."""
import pytest
import torch

from synthetic import get_config, make_batch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,store,chunk", [("tiny", False, 1 << 20), ("mid", False, 128), ("mid", True, 1 << 20)])
def test_replayed_pass_equals_the_eager_one(name, store, chunk):
    from paper_2606_29758_gb300 import PassShape, UpdatePass
    from paper_2606_29758_gb300 import _binding as B
    cfg = get_config(name)
    b = make_batch(cfg, device="cuda")
    D = b.dev
    dt = torch.float32 if cfg.dtype == "f32" else torch.bfloat16
    u = UpdatePass(PassShape(cfg.P, cfg.K, b.T_max, cfg.d, cfg.V, b.total_len, dt, chunk, b.total_len if store else 0),
                   eps=cfg.eps, loss_scale=cfg.loss_scale)
    N = u.run(D["q"], D["L"], D["R"], D["tok_full"], D["oldlogp_full"], D["hid_full"], D["W"], cfg.seed, cfg.step)
    outs = (u.loss, u.lse[:N], u.coef[:N], u.hid[:N], u.dH[:N], u.dW)
    torch.cuda.synchronize()
    ref = [x.clone() for x in outs]

    def work():   # the row count stays the eager pass's: a captured call cannot read it back
        s = u.s
        u.sample(D["q"], D["L"], cfg.seed, cfg.step)
        B.ps_pack_prefixes(s.P, s.K, s.T_max, s.d, u.dcode, D["L"], u.n, D["R"], u.adv_mode, u.w_tab, D["tok_full"],
                           D["oldlogp_full"], D["hid_full"], s.capacity, u.cu_seqlens, u.src_row, u.row_traj, u.row_pos,
                           u.tok, u.oldlogp, u.w, u.adv, u.hid, u.ws_pack, return_num_rows=False)
        u.forward(D["W"])
        u.backward(D["W"])

    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        work()
    torch.cuda.current_stream().wait_stream(side)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        work()
    for _ in range(2):
        for x in outs:
            x.zero_()
        graph.replay()
        torch.cuda.synchronize()
        u.check_status()
        for x, r in zip(outs, ref):
            assert torch.equal(x, r)
