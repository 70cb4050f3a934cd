"""What a call costs follows from what has to be priced, not from the size of
the buffers it lies in: passes timed with CUDA events against one another
(medians; the limits leave a third for noise)."""

import statistics

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def h(heddle_lib):
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    return heddle_lib


@pytest.fixture(scope="module")
def W():
    from paper_2609_34244_gb300 import workloads
    return workloads


def pass_us(f, reps=20):
    """Microseconds of one pass among others (the median of nine groups)."""
    import torch
    for _ in range(5):
        f()
    torch.cuda.synchronize()
    out = []
    for _ in range(9):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        for _ in range(reps):
            f()
        e1.record()
        torch.cuda.synchronize()
        out.append(e0.elapsed_time(e1) * 1e3 / reps)
    return statistics.median(out)


def test_split_rule_cost_follows_the_entries(h, W):
    """A hundred admissible structures of 32 stages among 60,000 invalid ones
    and among 140,000: a thread's chain of 32 stages is twice a warp's."""
    us = []
    for n in (60_000, 140_000):
        w = W.make_workload("stress128", seed=7, n=n)
        live = np.zeros(n, bool)
        live[np.random.default_rng(1).choice(n, 100, replace=False)] = True
        w.cands["code"][0, ~live] |= 0x20
        ctx = h.heddle_create(0)
        try:
            h.heddle_load_cluster(ctx, w.cluster)
            h.heddle_load_model(ctx, w.model)
            h.heddle_set_search(ctx, h.SEARCH_DISTRIBUTE)
            dc, res, state = h.cands_to_device(w.cands), h.alloc_results(n), h.alloc_topk_state()
            h.heddle_topk_reset(ctx, state, 16)
            us.append(pass_us(lambda: h.heddle_price_topk(ctx, dc, res, state)))
            assert h.heddle_device_errors(ctx) == 0
        finally:
            h.heddle_destroy(ctx)
    assert us[1] < 1.33 * us[0], us


def test_plan_walk_cost_follows_the_depth(h, W):
    """Plans of up to two stages in buffers of two planes and of 32: the walk
    goes by the plans' depth."""
    n = 200_003
    w = W.make_workload("dense32", seed=5, n=n)
    w.cluster["mem_bytes"][:] = 192 * 10**9
    plans = W.make_plans(w, n, 4, seed=5)
    plans["S"] = np.minimum(plans["S"], 2).astype(plans["S"].dtype)
    us = []
    for planes in (2, 32):
        code = np.zeros((4, planes, n), np.uint8)
        code[:, :2] = plans["code"][:, :2]
        code[:, 1][plans["S"] < 2] = 0
        dp = h.plans_to_device(dict(plans, code=code))
        ctx = h.heddle_create(0)
        try:
            h.heddle_load_cluster(ctx, w.cluster)
            h.heddle_load_model(ctx, w.model)
            pr = h.alloc_plan_results(n, 4)
            us.append(pass_us(lambda: h.heddle_price_plans(ctx, dp, pr)))
            assert (pr["placed"] >= 2).float().mean() > 0.3
            assert h.heddle_device_errors(ctx) == 0
        finally:
            h.heddle_destroy(ctx)
    assert us[1] < 1.33 * us[0], us


def test_topk_cost_does_not_follow_the_order(h):
    """300,000 results in random order, sorted either way and all equal: the
    separate top-k reads the same planes."""
    import torch
    n = 300_000
    T = torch.randint(1 << 30, 1 << 40, (n,), generator=torch.Generator().manual_seed(3)).cuda()
    one = torch.ones(n, dtype=torch.int16, device="cuda")
    cands = {"S": torch.ones(n, dtype=torch.uint8, device="cuda"), "M": one,
             "code": torch.zeros((1, n), dtype=torch.uint8, device="cuda")}
    ctx = h.heddle_create(0)
    try:
        state = h.alloc_topk_state()
        us = {}
        for order, t in (("random", T), ("rising", T.sort().values), ("falling", T.sort(descending=True).values),
                         ("equal", torch.full_like(T, 1 << 35))):
            res = {"T": t, "bottleneck": t, "n_dp": one, "status": torch.zeros(n, dtype=torch.uint8, device="cuda")}

            def one_pass():
                h.heddle_topk_reset(ctx, state, 64)
                h.heddle_topk(ctx, cands, res, state)

            us[order] = pass_us(one_pass)
        assert max(us.values()) < 1.1 * us["random"], us
    finally:
        h.heddle_destroy(ctx)
