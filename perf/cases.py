"""Performance cases of the PS-PPO LM-head update library, run through its public entry points.

A case is a dict of plain values; `kind` says which entry points it goes through:

  update   UpdatePass.run: cutoffs, packing, fused forward and (with grads) backward of one rollout batch
  design   CutoffDesign.run: score proxy with the top-k next tokens, u_t, and the cutoff design
  cutoffs  CutoffDesign.design alone, from scores that are already there
  pack     UpdatePass.sample and UpdatePass.pack: cutoffs and the packed rows, without the head
  shards   VocabParallelHead: the head split by vocabulary rows, its shards in turn on one device

Inputs follow the synthetic workloads of the benchmark: lognormal or uniform completion lengths, a
Beta(a, b) cutoff law per prompt, Bernoulli rewards, hidden states N(0, 1), W ~ N(0, 0.02), old
log-probabilities = new + N(0, 0.05). Each hidden row also leans towards its own token's row of W by
a random amount, so that log p(token) ranges from that of a random token to nearly 0 as in a trained
policy. The completion lengths, the cutoff laws and the cutoff stream belong to the case, so that every
seed packs the same number of rows; everything else is drawn from the seed alone, on the device.
"""
import math

import numpy as np
import torch

from paper_2606_29758_gb300 import (PS_DESIGN_HEURISTIC, PS_DESIGN_OPTIMIZED, PS_DESIGN_TIME_PRIOR,
                                    PS_DESIGN_UNIFORM, PS_MODE_FULL, PS_MODE_TRUNC, CutoffDesign, DesignShape,
                                    PassShape, UpdatePass, VocabParallelHead, vocab_shards)

DEVICE = "cuda"
ONE62 = 1 << 62
EPS = 0.2
CUTOFF_SEED, CUTOFF_STEP = 11, 3
STRATEGY = {"optimized": PS_DESIGN_OPTIMIZED, "heuristic": PS_DESIGN_HEURISTIC, "uniform": PS_DESIGN_UNIFORM,
            "time_prior": PS_DESIGN_TIME_PRIOR}


def listed():
    return [
        # The benchmark's Tiny workload (f32, under a thousand packed rows): unit runs and debugging, where
        # launches and latency are all there is.
        dict(name="update_tiny_f32", kind="update", P=2, K=4, lo=32, hi=256, median=0, d=128, V=1024,
             dtype="f32", early=False, mode="trunc", store=False, grads=True),
        # A small policy's head with sizes that are a multiple of no tile, logits recomputed.
        dict(name="update_mid_bf16", kind="update", P=2, K=4, lo=40, hi=300, median=0, d=392, V=2000,
             dtype="bf16", early=False, mode="trunc", store=False, grads=True),
        # An f32 head over a few thousand rows: a full-precision reference run of a small policy.
        dict(name="update_f32", kind="update", P=4, K=8, lo=100, hi=600, median=0, d=768, V=8192,
             dtype="f32", early=False, mode="trunc", store=False, grads=True),
        # The 7B-shaped head on a few hundred packed rows: two small groups of short answers, the smallest
        # micro-batch of a gradient-accumulation loop.
        dict(name="update_7b_short", kind="update", P=2, K=4, lo=60, hi=150, median=0, d=3584, V=152064,
             dtype="bf16", early=False, mode="trunc", store=True, grads=True),
        # The 7B-shaped head on one group of four ordinary completions (8k packed rows): an ordinary
        # micro-batch.
        dict(name="update_7b_group", kind="update", P=1, K=4, lo=128, hi=8192, median=2048, d=3584, V=152064,
             dtype="bf16", early=False, mode="trunc", store=True, grads=True),
        # Half of the 7B-shaped benchmark batch (8 prompts x 8, 106k packed rows) with the logit store:
        # the ordinary large step.
        dict(name="update_7b_batch", kind="update", P=8, K=8, lo=128, hi=8192, median=2048, d=3584, V=152064,
             dtype="bf16", early=False, mode="trunc", store=True, grads=True),
        # The 1.5B-shaped head without memory for the logits: the backward recomputes them.
        dict(name="update_1.5b_recompute", kind="update", P=8, K=8, lo=64, hi=4096, median=1024, d=1536, V=151936,
             dtype="bf16", early=False, mode="trunc", store=False, grads=True),
        # The surrogate and log-probabilities of whole completions, no gradients (an evaluation pass between
        # updates).
        dict(name="eval_1.5b", kind="update", P=1, K=8, lo=64, hi=4096, median=1024, d=1536, V=151936,
             dtype="bf16", early=False, mode="full", store=False, grads=False),
        # The whole design stage under the 1.5B-shaped old policy: score proxy and top 16, u_t, design.
        dict(name="design_1.5b", kind="design", P=2, K=8, lo=64, hi=4096, median=1024, d=1536, V=151936,
             topk=16, budget=128.0),
        # The cutoff design of long traces from their scores (8 prompts x 16, up to 16k steps), at a budget
        # that keeps many early steps whole.
        dict(name="cutoffs_long", kind="cutoffs", P=8, K=16, lo=8192, hi=16384, median=0, strategy="optimized",
             budget=2048.0),
        # Cutoffs and packing of long traces (2 prompts x 16, early-skewed cutoffs): the data path without
        # the head.
        dict(name="pack_long", kind="pack", P=2, K=16, lo=8192, hi=16384, median=0, d=3584, V=152064,
             dtype="bf16", early=True),
        # The 1.5B-shaped head in four vocabulary shards run one after another.
        dict(name="shards_1.5b", kind="shards", N=6000, d=1536, V=151936, S=4, store=False),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    """One more case of the ranges that the listed ones stand for."""
    kind = rng.choice(["update", "update", "update", "update", "design", "cutoffs", "pack", "shards"])
    if kind == "update":
        f32 = rng.random() < 0.25
        d = int(_log(rng, 96, 768 if f32 else 4096)) // 8 * 8
        V = int(_log(rng, 900, 8200 if f32 else 152100))
        limit = 2.5e11 if f32 else 1.2e14                  # FLOPs of the update, 6 N d V
        tokens = _log(rng, 600, min(12000 if f32 else 150000, limit / (4.0 * d * V)) + 700)
        K = rng.choice([2, 4, 8, 16])
        P = max(1, min(32, round(tokens / K / _log(rng, 60, 2000))))
        mean = max(24, min(6000, tokens / (P * K)))
        grads = rng.random() < 0.8
        return dict(kind=kind, P=P, K=K, lo=max(8, int(mean * 0.4)), hi=int(mean * 1.6), median=0, d=d, V=V,
                    dtype="f32" if f32 else "bf16", early=rng.random() < 0.2,
                    mode="full" if rng.random() < 0.2 else "trunc",
                    store=not f32 and grads and rng.random() < 0.5, grads=grads)
    if kind == "design":
        d, V = int(_log(rng, 256, 3584)) // 8 * 8, int(_log(rng, 2000, 152064))
        P, K = rng.choice([1, 2, 4]), rng.choice([4, 8, 16])
        mean = max(40, min(2500, _log(rng, 1e3, min(4e4, 1.2e13 / (2.0 * d * V)) + 1.1e3) / (P * K)))
        return dict(kind=kind, P=P, K=K, lo=max(8, int(mean * 0.4)), hi=int(mean * 1.6), median=0, d=d, V=V,
                    topk=rng.choice([8, 16]), budget=float(int(_log(rng, 16, mean))))
    if kind == "cutoffs":
        P, K, hi = rng.choice([1, 4, 8, 16, 32]), rng.choice([4, 8, 16]), int(_log(rng, 200, 16384))
        return dict(kind=kind, P=P, K=K, lo=max(8, hi // 3), hi=hi, median=0,
                    strategy=rng.choice(["optimized", "optimized", "optimized", "heuristic", "uniform", "time_prior"]),
                    budget=float(int(_log(rng, 16, hi / 2))))
    if kind == "pack":
        P, K, hi = rng.choice([1, 2, 4, 8]), rng.choice([4, 8, 16]), int(_log(rng, 100, 8000))
        return dict(kind=kind, P=P, K=K, lo=max(8, hi // 3), hi=hi, median=0, d=int(_log(rng, 128, 4096)) // 8 * 8,
                    V=int(_log(rng, 1000, 152064)), dtype=rng.choice(["bf16", "f32"]), early=rng.random() < 0.5)
    d, V = int(_log(rng, 256, 4096)) // 8 * 8, int(_log(rng, 4000, 152064))
    return dict(kind="shards", N=int(_log(rng, 200, min(2e4, 1.5e13 / (6.0 * d * V)) + 300)), d=d, V=V,
                S=rng.choice([2, 3, 4, 8]), store=rng.random() < 0.5)


# ----------------------------------------------------------------------------- inputs
def _lengths(case, rng):
    B = case["P"] * case["K"]
    if case["median"]:
        L = np.rint(np.exp(math.log(case["median"]) + 0.5 * rng.standard_normal(B)))
        return np.clip(L, case["lo"], case["hi"]).astype(np.int32)
    return rng.integers(case["lo"], case["hi"] + 1, size=B).astype(np.int32)


def _masses(case, L, rng):
    """Cutoff masses [P][T_max] summing to 2^62: a Beta(a, b) law on 1..T_p per prompt."""
    P, K = case["P"], case["K"]
    q = np.zeros((P, int(L.max())), dtype=np.uint64)
    for p in range(P):
        T = int(L[p * K:(p + 1) * K].max())
        a, b = (rng.uniform(0.5, 1.0), rng.uniform(2.0, 4.0)) if case["early"] else rng.uniform(0.5, 3.0, size=2)
        x = (np.arange(T) + 0.5) / T
        m = x ** (a - 1.0) * (1.0 - x) ** (b - 1.0)
        m = np.floor(m / m.sum() * float(ONE62)).astype(np.uint64)
        i = int(np.argmax(m))
        m[i] = np.uint64(int(m[i]) + ONE62 - int(m.sum(dtype=np.uint64)))
        q[p, :T] = m
    return q


def _head(seed, rows, d, V, dtype, with_logp=True):
    """Hidden rows, W, tokens and old log-probabilities on the device."""
    g = torch.Generator(device=DEVICE).manual_seed(seed)
    t = torch.float32 if dtype == "f32" else torch.bfloat16
    W = torch.empty(V, d, dtype=t, device=DEVICE)
    for v0 in range(0, V, 16384):
        n = min(16384, V - v0)
        W[v0:v0 + n] = torch.randn(n, d, device=DEVICE, generator=g) * 0.02
    tok = torch.randint(0, V, (rows,), device=DEVICE, generator=g, dtype=torch.int32)
    hid = torch.empty(rows, d, dtype=t, device=DEVICE)
    logp = torch.zeros(rows, device=DEVICE)
    for r0 in range(0, rows, 2048):
        r1 = min(rows, r0 + 2048)
        own = W[tok[r0:r1].long()].float()
        lean = torch.rand(r1 - r0, 1, device=DEVICE, generator=g) * (math.log(V) + 6.0)
        h = torch.randn(r1 - r0, d, device=DEVICE, generator=g) + own * (lean / own.square().sum(1, keepdim=True))
        hid[r0:r1] = h
        if with_logp:
            z = torch.matmul(hid[r0:r1], W.t()).float()
            logp[r0:r1] = z.gather(1, tok[r0:r1, None].long())[:, 0] - torch.logsumexp(z, dim=1)
            del z
    old = (logp + 0.05 * torch.randn(rows, device=DEVICE, generator=g)).clamp_(max=0.0)
    return hid, W, tok, old


class State:
    pass


def _batch(s, case):
    """The case's completion lengths and, where it samples cutoffs, their masses (on the host)."""
    rng = np.random.default_rng([case["P"], case["K"], case["lo"], case["hi"], 5])
    s.case, s.L_host = case, _lengths(case, rng)
    if case["kind"] in ("update", "pack"):
        s.q_host = _masses(case, s.L_host, rng)
    return s


def _dev(x):
    return torch.from_numpy(np.ascontiguousarray(x)).to(DEVICE)


def prepare(case, seed):
    s = State()
    s.case = case
    rng = np.random.default_rng([seed, 77])
    if case["kind"] == "shards":
        N, d, V = case["N"], case["d"], case["V"]
        s.hid, s.W, s.tok, s.old = _head(seed, N, d, V, "bf16")
        s.adv = _dev(rng.standard_normal(N).astype(np.float32))
        s.w = _dev((1.0 / rng.uniform(0.05, 1.0, size=N)).astype(np.float32))
        s.shards = vocab_shards(V, case["S"])
        s.head = VocabParallelHead(s.shards, N, d, V, eps=EPS, loss_scale=1.0 / 16, store=case["store"])
        s.dH = torch.empty(N, d, device=DEVICE)
        s.dW = torch.empty(V, d, device=DEVICE)
        return s
    _batch(s, case)
    P, K, T, total = case["P"], case["K"], int(s.L_host.max()), int(s.L_host.sum())
    s.L = _dev(s.L_host)
    s.R = _dev((rng.random(P * K) < 0.5).astype(np.float32))
    if case["kind"] == "cutoffs":
        # scores of a decaying trend times lognormal noise: neighbouring steps often violate the monotone order
        t = np.concatenate([np.arange(n) for n in s.L_host])
        s.cd = CutoffDesign(DesignShape(P, K, T, 8, 32, total, 16), device=DEVICE)
        s.cd.gamma.copy_(_dev((1536.0 * (1.0 + 3.0 * np.exp(-t / 200.0)) *
                               np.exp(0.7 * rng.standard_normal(total))).astype(np.float32)))
        s.cd.u.copy_(_dev(rng.uniform(0.02, 0.25, size=(P, T)).astype(np.float32)))
        return s
    if case["kind"] == "design":
        s.hid, s.W, s.tok, s.old = _head(seed, total, case["d"], case["V"], "bf16", with_logp=False)
        s.cd = CutoffDesign(DesignShape(P, K, T, case["d"], case["V"], total, case["topk"]), device=DEVICE)
        return s
    s.q = _dev(s.q_host.view(np.int64))
    s.hid, s.W, s.tok, s.old = _head(seed, total, case["d"], case["V"], case["dtype"],
                                     with_logp=case["kind"] == "update")
    shape = PassShape(P, K, T, case["d"], case["V"], total,
                      torch.float32 if case["dtype"] == "f32" else torch.bfloat16, bwd_chunk_rows=4096 if case.get("store") else 32768,
                      store_rows=total if case.get("store") else 0)
    s.up = UpdatePass(shape, device=DEVICE, eps=EPS,
                      mode=PS_MODE_FULL if case.get("mode") == "full" else PS_MODE_TRUNC)
    return s


def run(s):
    case = s.case
    if case["kind"] == "update":
        u = s.up
        N = u.run(s.q, s.L, s.R, s.tok, s.old, s.hid, s.W, CUTOFF_SEED, CUTOFF_STEP, grads=case["grads"])
        out = dict(H=u.H, n=u.n, loss=u.loss, lse=u.lse[:N], logp=u.logp[:N], ratio=u.ratio[:N], coef=u.coef[:N],
                   row_loss=u.row_loss[:N])
        if case["grads"]:
            out.update(dH=u.dH[:N], dW=u.dW)
        return out
    if case["kind"] == "pack":
        u = s.up
        u.sample(s.q, s.L, CUTOFF_SEED, CUTOFF_STEP)
        N = u.pack(s.L, s.R, s.tok, s.old, s.hid)
        return dict(H=u.H, n=u.n, w_tab=u.w_tab, cu_seqlens=u.cu_seqlens, src_row=u.src_row[:N],
                    row_traj=u.row_traj[:N], row_pos=u.row_pos[:N], tok=u.tok[:N], oldlogp=u.oldlogp[:N], w=u.w[:N],
                    adv=u.adv[:N], hid=u.hid[:N])
    if case["kind"] == "cutoffs":
        s.cd.design(s.L, case["budget"], STRATEGY[case["strategy"]])
        return dict(q=s.cd.q, xi=s.cd.xi)
    if case["kind"] == "design":
        # The masses are the differences of xi in units of 2^-62: every change of rounding in the scores moves
        # their last digits, so the survival xi stands for them here (the cutoffs cases return the masses).
        c = s.cd
        c.run(s.hid, s.W, s.tok, s.L, s.R, case["budget"])
        return dict(gamma=c.gamma, logp=c.logp, top_idx=c.top_idx, top_prob=c.top_prob, u=c.u, xi=c.xi)
    h, N = s.head, case["N"]
    for r, (v0, Vs) in enumerate(s.shards):
        h.stats(r, N, s.hid, s.W[v0:v0 + Vs], s.tok)
    h.forward(N, s.tok, s.old, s.adv, s.w)
    for r, (v0, Vs) in enumerate(s.shards):
        h.backward(r, N, s.hid, s.W[v0:v0 + Vs], s.tok, s.dH, s.dW[v0:v0 + Vs], add_to_dH=r > 0)
    return dict(loss=h.loss, lse=h.lse, logp=h.logp, ratio=h.ratio, coef=h.coef, row_loss=h.row_loss, dH=s.dH,
                dW=s.dW)


# ----------------------------------------------------------------------------- what a pass cannot do without
def work(case):
    kind = case["kind"]
    if kind == "shards":
        n, d, V = case["N"], case["d"], case["V"]
        return {"bytes": 6.0 * d * (n + V) + 40.0 * n, "flops": 6.0 * n * d * V}
    s = _batch(State(), case)
    total, PT = int(s.L_host.sum()), case["P"] * int(s.L_host.max())
    if kind == "cutoffs":
        return {"bytes": 4.0 * total + PT * (4 + 8 + 8), "flops": 0.0}
    d, V = case["d"], case["V"]
    if kind == "design":
        return {"bytes": 2.0 * d * (total + V) + total * (12 + 8 * case["topk"]) + PT * (4 + 8 + 8),
                "flops": 2.0 * total * d * V}
    n, es = int(_cutoffs64(s)[1].sum()), 4 if case["dtype"] == "f32" else 2
    if kind == "pack":
        return {"bytes": 2.0 * n * d * es + 44.0 * n + 12.0 * PT, "flops": 0.0}
    if not case["grads"]:
        return {"bytes": es * d * (n + V) + 36.0 * n + 12.0 * PT, "flops": 2.0 * n * d * V}
    return {"bytes": (es + 4.0) * d * (n + V) + 36.0 * n + 12.0 * PT, "flops": 6.0 * n * d * V}


def tolerance(case):
    kind = case["kind"]
    if kind in ("cutoffs", "pack"):
        return "exact"                     # integers, and floats whose every rounding is defined
    if kind == "design":
        # f32 logits and sums of exact bf16 products; equal logits within their rounding may trade places
        return {"rel": 2e-5, "max": 1e-3, "differ": 1e-3}
    if case["kind"] == "update" and case["dtype"] == "f32":
        return {"rel": 1e-5, "max": 1e-3}
    # bf16: dZ is rounded to bf16 (2^-9) before it enters dH and dW
    return {"rel": 1e-2, "max": 0.1}


# ----------------------------------------------------------------------------- the same in 64 bits
_MOST = 1.4e13        # FLOPs in 64 bits that exact() takes on (about 20 seconds)


def _cutoffs64(s):
    """H, n and the weight table of the state's masses: Philox4x64-10 draws x = word >> 2, H = min{h : x < U[h]}."""
    case = s.case
    P, K, B = case["P"], case["K"], case["P"] * case["K"]
    if case.get("mode") == "full":
        return s.L_host.copy(), s.L_host.copy(), np.ones(s.q_host.shape)
    H = np.zeros(B, np.int32)
    w = np.full(s.q_host.shape, np.inf)
    for p in range(P):
        U = np.cumsum(s.q_host[p])
        S = np.uint64(ONE62) - np.concatenate([[np.uint64(0)], U[:-1]])
        ok = S > 0
        w[p, ok] = float(ONE62) / S[ok].astype(np.float64)
        for k in range(p * K, (p + 1) * K):
            # numpy steps its counter before it draws
            c = (k + (CUTOFF_STEP << 64) - 1) % (1 << 256)
            g = np.random.Philox(counter=c, key=CUTOFF_SEED + (0x5053505030303031 << 64))
            H[k] = int(np.searchsorted(U, g.random_raw(1)[0] >> np.uint64(2), side="right")) + 1
    return H, np.minimum(H, s.L_host), w


def _packed64(s):
    case = s.case
    P, K = case["P"], case["K"]
    H, n, w = _cutoffs64(s)
    R = s.R.double().cpu().numpy().reshape(P, K)
    A = ((R - R.mean(1, keepdims=True)) / (R.std(1, keepdims=True) + 1e-6)).reshape(-1)
    off = np.concatenate([[0], np.cumsum(s.L_host)[:-1]])
    traj = np.repeat(np.arange(P * K), n)
    pos = np.concatenate([np.arange(int(x)) for x in n])
    return H, n, w, traj, pos, off[traj] + pos, w[traj // K, pos], A[traj]


def _head64(hid, W, tok, old, adv, w, scale, grads):
    """The surrogate through the head, and its gradients, in 64 bits."""
    N, W64 = hid.shape[0], W.double()
    cols = [torch.empty(N, dtype=torch.float64, device=DEVICE) for _ in range(5)]
    dH = torch.empty(N, W.shape[1], dtype=torch.float64, device=DEVICE) if grads else None
    dW = torch.zeros_like(W64) if grads else None
    for r0 in range(0, N, 1024):
        r = slice(r0, min(N, r0 + 1024))
        h = hid[r].double()
        z = h @ W64.t()
        t = tok[r, None].long()
        lse = torch.logsumexp(z, 1)
        logp = z.gather(1, t)[:, 0] - lse
        ratio = torch.exp(logp - old[r].double())
        a, c = adv[r], scale * w[r]
        sur = torch.minimum(ratio * a, ratio.clamp(1 - EPS, 1 + EPS) * a)
        bind = ((a > 0) & (ratio > 1 + EPS)) | ((a < 0) & (ratio < 1 - EPS))
        coef = torch.where(bind, torch.zeros_like(a), -c * a * ratio)
        for col, v in zip(cols, (lse, logp, ratio, coef, -c * sur)):
            col[r] = v
        if grads:
            z.sub_(lse[:, None]).exp_().mul_(-coef[:, None])
            z.scatter_add_(1, t, coef[:, None])
            dH[r] = z @ W64
            dW.addmm_(z.t(), h)
    return cols, dH, dW


def _design64(case, L, gamma, u):
    """xi [P][T_max] in 64 bits."""
    P, K, T = case["P"], case["K"], int(L.max())
    strategy, xi, o = case.get("strategy", "optimized"), np.zeros((P, T)), 0
    for p in range(P):
        Ls = L[p * K:(p + 1) * K]
        Tp = int(Ls.max())
        B = min(case["budget"], float(Tp))
        w = np.zeros(Tp)
        for n in Ls:
            w[:n] += gamma[o:o + n]
            o += int(n)
        w = w / K * u[p, :Tp]
        w = np.maximum(w, 1e-12 * w.max())
        if strategy == "uniform":
            x = (Tp - np.arange(Tp)) / Tp
        elif strategy == "heuristic":
            x = np.minimum(np.minimum.accumulate(B * np.sqrt(w) / np.sqrt(w).sum()), 1.0)
        elif strategy == "time_prior":
            lo, hi, t = 0.0, 1.0, np.arange(Tp)
            while np.exp(-hi * t).sum() > B:
                hi *= 2
            for _ in range(200):
                mid = 0.5 * (lo + hi)
                lo, hi = (mid, hi) if np.exp(-mid * t).sum() > B else (lo, mid)
            x = np.exp(-hi * t) if Tp > B else np.ones(Tp)
        else:
            def pooled(first):
                # blocks of every suffix by pooling from the right; D = sum of n_m sqrt(W_m / n_m) over them
                st, D, best = [], 0.0, None
                for t in range(Tp - 1, first - 1, -1):
                    Wc, nc = w[t], 1
                    while st and st[-1][0] * nc > Wc * st[-1][1]:
                        Wp, n_ = st.pop()
                        D -= math.sqrt(Wp * n_)
                        Wc, nc = Wc + Wp, nc + n_
                    st.append((Wc, nc))
                    D += math.sqrt(Wc * nc)
                    if (B - t) * math.sqrt(Wc / nc) <= D:
                        best = t          # prefixes below t saturated, this suffix starts at or below 1
                return st, best
            first = pooled(0)[1]
            x = np.ones(Tp)
            if first is not None:
                st = pooled(first)[0][::-1]
                D, t = sum(math.sqrt(W * n) for W, n in st), first
                for W, n in st:
                    x[t:t + n] = (B - first) * math.sqrt(W / n) / D
                    t += n
        xi[p, :Tp] = x
    return xi


def _unc64(case, L, R, idx, prob):
    P, K, T = case["P"], case["K"], int(L.max())
    u, off = np.zeros((P, T)), np.concatenate([[0], np.cumsum(L)[:-1]])
    for p in range(P):
        ks = range(p * K, (p + 1) * K)
        phat = np.mean([R[k] >= 0.5 for k in ks])
        for t in range(int(max(L[k] for k in ks))):
            live = [k for k in ks if L[k] > t]
            g = sum(R[k] >= 0.5 for k in live)
            sums, other = {}, 0.0
            for k in live:
                c = phat / g if R[k] >= 0.5 else -(1.0 - phat) / (len(live) - g)
                for a, v in zip(idx[off[k] + t], prob[off[k] + t]):
                    sums[a] = sums.get(a, 0.0) + c * v
                other += c * (1.0 - prob[off[k] + t].sum())
            u[p, t] = min(0.5, max(0.0, 0.5 - 0.5 * (sum(abs(v) for v in sums.values()) + abs(other))))
    return u


def exact(case, seed):
    kind, grads = case["kind"], case.get("grads", True)
    flops = work(case)["flops"]
    forward = flops / 3.0 if grads and kind in ("update", "shards") else flops
    if forward > _MOST:
        return None
    grads = grads and flops <= _MOST
    s = prepare(case, seed)
    if kind == "cutoffs":
        return dict(q=None, xi=_design64(case, s.L_host, s.cd.gamma.double().cpu().numpy(),
                                         s.cd.u.double().cpu().numpy()))
    if kind == "shards":
        (lse, logp, ratio, coef, rl), dH, dW = _head64(s.hid, s.W, s.tok, s.old, s.adv.double(), s.w.double(),
                                                       1.0 / 16, grads)
        return dict(loss=rl.sum().reshape(1), lse=lse, logp=logp, ratio=ratio, coef=coef, row_loss=rl, dH=dH, dW=dW)
    if kind == "design":
        W64, N, k = s.W.double(), s.hid.shape[0], case["topk"]
        gamma, logp = (torch.empty(N, dtype=torch.float64, device=DEVICE) for _ in range(2))
        idx = torch.empty(N, k, dtype=torch.int32, device=DEVICE)
        prob = torch.empty(N, k, dtype=torch.float64, device=DEVICE)
        for r0 in range(0, N, 1024):
            r = slice(r0, min(N, r0 + 1024))
            h = s.hid[r].double()
            z = torch.log_softmax(h @ W64.t(), 1)
            logp[r] = z.gather(1, s.tok[r, None].long())[:, 0]
            top, at = z.topk(k, dim=1)
            prob[r], idx[r] = top.exp(), at.int()
            z.exp_()
            gamma[r] = h.square().sum(1) * (z.square().sum(1) + 1.0 - 2.0 * logp[r].exp())
        u = _unc64(case, s.L_host, s.R.cpu().numpy(), idx.cpu().numpy(), prob.cpu().numpy())
        return dict(gamma=gamma, logp=logp, top_idx=idx, top_prob=prob, u=u,
                    xi=_design64(case, s.L_host, gamma.cpu().numpy(), u))
    H, n, w_tab, traj, pos, src, w, A = _packed64(s)
    rows = _dev(src)
    if kind == "pack":
        return dict(H=H, n=n, w_tab=w_tab, cu_seqlens=None, src_row=None, row_traj=None, row_pos=None, tok=None,
                    oldlogp=s.old[rows].double(), w=w, adv=A, hid=s.hid[rows])
    (lse, logp, ratio, coef, rl), dH, dW = _head64(s.hid[rows], s.W, s.tok[rows], s.old[rows], _dev(A), _dev(w),
                                                   1.0 / (case["P"] * case["K"]), grads)
    out = dict(H=H, n=n, loss=rl.sum().reshape(1), lse=lse, logp=logp, ratio=ratio, coef=coef, row_loss=rl)
    if case["grads"]:
        out.update(dH=dH, dW=dW)
    return out
