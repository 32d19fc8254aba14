"""The capped design's search for the saturated prefix, where many prefixes lie on the cap, against the oracle bit for
bit, and its time beside that of an ordinary trace of the same length (which takes one or two poolings)."""
import numpy as np
import pytest
import torch

from oracle import design

pytestmark = pytest.mark.gpu


def _run(w, budget, reps=3):
    """(q, xi, milliseconds) of one prompt of one completion whose scores, and so its weights, are w."""
    from paper_2606_29758_gb300 import PS_DESIGN_OPTIMIZED, CutoffDesign, DesignShape
    T = len(w)
    cd = CutoffDesign(DesignShape(1, 1, T, 8, 32, T, 0))
    cd.gamma.copy_(torch.from_numpy(w))
    cd.u.fill_(1.0)
    L = torch.tensor([T], dtype=torch.int32, device="cuda")
    ms = []
    for _ in range(reps):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        cd.design(L, budget, PS_DESIGN_OPTIMIZED)
        b.record()
        torch.cuda.synchronize()
        ms.append(a.elapsed_time(b))
    cd.check_status()
    return cd.q.cpu().numpy().view(np.uint64), cd.xi.cpu().numpy(), min(ms)


def _ordinary(T):
    rng = np.random.default_rng(1)
    return np.exp(0.7 * rng.standard_normal(T) - np.arange(T) / T).astype(np.float32)


# (trace, the most poolings' worth of time: an ordinary trace's is 1) at a budget of the whole trace, where every
# suffix that pools to one block starts at exactly 1
def _flat_tail(T):            # the first prefix on the cap passes
    w = _ordinary(T)
    w[-100:] = 1e-3
    return w


def _rising(T):               # hundreds on the cap, the first of them passes
    w = _ordinary(T)
    w[T // 2:] *= np.linspace(3.0, 30.0, T - T // 2, dtype=np.float32)
    return w


def _slow_fall(T):            # every prefix within the band, none passes but the last few
    return np.linspace(1.0, 1.0 - 3e-6, T).astype(np.float32)


@pytest.mark.parametrize("trace,most", [(_flat_tail, 20.0), (_rising, 20.0), (_slow_fall, 1500.0)])
def test_many_prefixes_on_the_cap(trace, most):
    T = 1500
    w = trace(T)
    q, xi, ms = _run(w, float(T))
    q_ref, xi_ref = design.design_cutoff_masses(np.array([T], dtype=np.int32), 1, w, np.ones((1, T), np.float32),
                                                float(T), "optimized")
    assert np.array_equal(xi, xi_ref)
    assert np.array_equal(q, q_ref)
    assert ms < most * _run(_ordinary(T), 100.0)[2], ms


# Traces whose blocks the float slopes cannot propose, so that pooling has to repair them: weights of ten decades next to
# each other (tokens a trained policy is sure of), and weights that differ in their last float bits
def _ten_decades(T):
    rng = np.random.default_rng(5)
    q = np.where(rng.random(T) < 0.5, np.exp(rng.uniform(np.log(1e-6), np.log(1e-2), T)), rng.uniform(0.01, 1.0, T))
    return (3072.0 * q * q * rng.uniform(0.02, 0.25, T)).astype(np.float32)


def _nearly_flat(T):
    return (1.0 + 1e-7 * np.random.default_rng(4).standard_normal(T)).astype(np.float32)


@pytest.mark.parametrize("trace,T,most", [(_ten_decades, 15000, 3.0), (_nearly_flat, 8000, 12.0),
                                          (_ten_decades, 4097, 50.0), (_nearly_flat, 1025, 50.0)])
def test_pooling_repairs_wrong_links(trace, T, most):
    w = trace(T)
    q, xi, ms = _run(w, 20.0)
    q_ref, xi_ref = design.design_cutoff_masses(np.array([T], dtype=np.int32), 1, w, np.ones((1, T), np.float32), 20.0,
                                                "optimized")
    assert np.array_equal(xi, xi_ref)
    assert np.array_equal(q, q_ref)
    assert ms < most * _run(_ordinary(T), 20.0)[2], ms


@pytest.mark.parametrize("trace", [_ordinary, _ten_decades])
@pytest.mark.parametrize("T", [(1 << 18) + 3, 1 << 20])
def test_long_traces(trace, T):
    # sums over a thousand windows and more; a small budget, so that the oracle pools once
    w = trace(T)
    q, xi, _ = _run(w, 5.0, reps=1)
    q_ref, xi_ref = design.design_cutoff_masses(np.array([T], dtype=np.int32), 1, w, np.ones((1, T), np.float32), 5.0,
                                                "optimized")
    assert np.array_equal(xi, xi_ref)
    assert np.array_equal(q, q_ref)


@pytest.mark.parametrize("T", [1, 2, 20, 511, 512, 513, 1025])
@pytest.mark.parametrize("strategy", ["optimized", "heuristic"])
def test_weights_of_one_part_and_of_several(T, strategy):
    # traces of up to 512 steps are weighed by the design kernel, longer ones by a launch of their own; several
    # prompts of unequal completions, so that every prompt's first row counts
    from paper_2606_29758_gb300 import PS_DESIGN_HEURISTIC, PS_DESIGN_OPTIMIZED, CutoffDesign, DesignShape
    rng = np.random.default_rng(T)
    P, K = 5, 3
    L = rng.integers(1, T + 1, size=P * K).astype(np.int32)
    L[rng.integers(P * K)] = T
    gamma = rng.lognormal(0.0, 1.0, int(L.sum())).astype(np.float32)
    u = rng.uniform(0.01, 0.5, (P, T)).astype(np.float32)
    cd = CutoffDesign(DesignShape(P, K, T, 8, 32, int(L.sum()), 16))
    cd.gamma.copy_(torch.from_numpy(gamma))
    cd.u.copy_(torch.from_numpy(u))
    for budget in (1.0, 0.4 * T + 0.7):
        cd.design(torch.from_numpy(L).cuda(), budget,
                  PS_DESIGN_OPTIMIZED if strategy == "optimized" else PS_DESIGN_HEURISTIC)
        cd.check_status()
        q_ref, xi_ref = design.design_cutoff_masses(L, K, gamma, u, budget, strategy)
        assert np.array_equal(cd.xi.cpu().numpy().reshape(P, T), xi_ref)
        assert np.array_equal(cd.q.cpu().numpy().view(np.uint64).reshape(P, T), q_ref)


def test_a_short_trace_is_weighed_without_a_launch_of_its_own():
    # graph replays, so that the host's calls do not count
    from paper_2606_29758_gb300 import PS_DESIGN_HEURISTIC, PS_DESIGN_UNIFORM, CutoffDesign, DesignShape
    P, K, T = 5, 3, 20
    cd = CutoffDesign(DesignShape(P, K, T, 8, 32, P * K * T, 0))
    cd.gamma.uniform_(0.5, 1.5)
    cd.u.fill_(0.1)
    L = torch.full((P * K,), T, dtype=torch.int32, device="cuda")

    def us(strategy, calls=100):
        cd.design(L, 8.0, strategy)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            for _ in range(calls):
                cd.design(L, 8.0, strategy)
        best = 1e9
        for _ in range(5):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            g.replay()
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b) / calls * 1e3)
        return best
    heuristic, uniform = us(PS_DESIGN_HEURISTIC), us(PS_DESIGN_UNIFORM)
    assert heuristic < 2.0 * uniform, (heuristic, uniform)
