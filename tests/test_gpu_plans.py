"""Multi-template plans (Algorithm 1) on the GPU through the C ABI against
the oracle's plan pricing: bit-exact per-template T, bottleneck, n_dp and
status (the plan's degree on the GPUs earlier templates left, SKIPPED past
the end), templates placed and the summed throughput (IEEE double)."""

import json
import os

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


def price_plans_gpu(h, cluster, model, plans, search=None, bounds=False, thread_min=None):
    import torch
    ctx = h.heddle_create(0)
    try:
        h.heddle_load_cluster(ctx, cluster)
        h.heddle_load_model(ctx, model)
        if search is not None:
            h.heddle_set_search(ctx, search)
        if thread_min is not None:
            h.heddle_set_thread_search_min(ctx, thread_min)
        dp = h.plans_to_device(plans)
        n = int(plans["n_tmpl"].shape[0])
        pr = h.alloc_plan_results(n, len(dp["slots"]), bounds=bounds)
        h.heddle_price_plans(ctx, dp, pr)
        torch.cuda.synchronize()
        out = {k: np.stack([h.results_to_numpy(r)[k] for r in pr["slots"]]) for k in ("T", "bottleneck", "n_dp", "status")}
        out["placed"] = pr["placed"].cpu().numpy()
        out["thr"] = pr["thr"].cpu().numpy()
        out["errors"] = h.heddle_device_errors(ctx)
        if bounds:
            out["bounds"] = [r["bounds"].cpu().numpy() for r in pr["slots"]]
        return out
    finally:
        h.heddle_destroy(ctx)


def _same(got, ref, what):
    for k in ("T", "bottleneck", "n_dp", "status"):
        bad = np.argwhere(got[k] != ref[k])
        assert bad.size == 0, "%s %s differs at %s: gpu %s oracle %s" % (
            what, k, bad[:5].tolist(), got[k][tuple(bad[0])], ref[k][tuple(bad[0])])
    assert (got["placed"] == ref["placed"]).all(), what
    bad = np.nonzero(got["thr"] != ref["thr"])[0]
    assert bad.size == 0, "%s thr differs at %s: %s vs %s" % (what, bad[:5], got["thr"][bad[:3]], ref["thr"][bad[:3]])


@pytest.mark.parametrize("deepest", [1, 2, 4, 8])
@pytest.mark.parametrize("n", [1, 127, 129, 20011])
def test_plans_that_mostly_walk(h, W, oracle_mod, deepest, n):
    """Shallow templates, most of which fit, on one plan and on all SMs (a CTA
    queues at most 17 of 20,011, which it walks a warp each by default), and a
    thread each; bounds as well."""
    w = W.make_workload("dense32", seed=5, n=n)
    plans = W.make_plans(w, n, 4, seed=5)
    plans["S"] = np.minimum(plans["S"], deepest).astype(plans["S"].dtype)
    plans["code"] = np.ascontiguousarray(plans["code"][:, :deepest])
    plans["code"][np.arange(deepest)[None, :, None] >= plans["S"][:, None, :]] = 0
    orc = oracle_mod.Oracle(w.cluster, w.model)
    ref = orc.price_plans(plans)
    for bounds in (False, True):
        for thread_min in (None, 0):
            got = price_plans_gpu(h, w.cluster, w.model, plans, bounds=bounds, thread_min=thread_min)
            assert got["errors"] == 0
            _same(got, ref, "deepest %d" % deepest)
            if bounds:
                _bounds_same(orc, plans, got)


@pytest.mark.parametrize("name,n", [("tiny", 300), ("dense32", 4001), ("dense80", 1501), ("moe48", 4001),
                                    ("stress128", 701)])
@pytest.mark.parametrize("seed", [0, 1])
def test_plans_parity(h, W, oracle_mod, name, n, seed):
    w = W.make_workload(name, seed=seed, n=n)
    plans = W.make_plans(w, n, 4, seed=seed)
    ref = oracle_mod.Oracle(w.cluster, w.model).price_plans(plans)
    got = price_plans_gpu(h, w.cluster, w.model, plans)
    assert got["errors"] == 0
    _same(got, ref, "%s plans" % name)
    assert (ref["placed"] >= 1).any()
    if name in ("dense32", "dense80", "stress128"):  # later templates priced on what is left
        assert (ref["placed"] >= 2).any()


@pytest.mark.parametrize("search", [1, 3], ids=["general", "distribute"])
def test_plans_other_split_modes(h, W, oracle_mod, search):
    w = W.make_workload("dense32", seed=5, n=2001)
    plans = W.make_plans(w, 2001, 3, seed=5)
    orc = oracle_mod.Oracle(w.cluster, w.model)
    if search == 3:
        orc.set_split("distribute")
    ref = orc.price_plans(plans)
    got = price_plans_gpu(h, w.cluster, w.model, plans, search=search)
    _same(got, ref, "dense32 search %d" % search)


def test_plans_bounds(h, W, oracle_mod):
    """With bound planes requested: an OK template keeps the split of its
    standalone price (the oracle's, slot by slot), every other template's
    planes are zero (slots that no plan reaches included)."""
    w = W.make_workload("dense32", seed=3, n=3001)
    plans = W.make_plans(w, 3001, 3, seed=3)
    ref = oracle_mod.Oracle(w.cluster, w.model).price_plans(plans)
    got = price_plans_gpu(h, w.cluster, w.model, plans, bounds=True)
    _same(got, ref, "dense32 plans with bounds")
    orc = oracle_mod.Oracle(w.cluster, w.model)
    for t in range(3):
        alone = orc.price({"S": np.ascontiguousarray(plans["S"][t]), "M": np.ascontiguousarray(plans["M"][t]),
                           "code": np.ascontiguousarray(plans["code"][t])}, bounds=True)
        b = got["bounds"][t]
        ok = got["status"][t] == 0
        assert ok.any() and (~ok).any(), t
        assert (b[:, ok] == alone["bounds"][:, ok]).all(), t
        assert (b[:, ~ok] == 0).all(), t


def test_plans_hand_cases(h, W):
    path = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "hand_plans.json")
    d = json.load(open(path))
    cl = d["cluster"]
    cluster = W.make_cluster(cl["tflops"], cl["mem_bytes"], cl["intra_bw"], [tuple(x) for x in cl["nodes"]])
    model = W.make_model(d["flops"], 0, 0, 0, 0, 0, 0)
    import pin_checks as PC
    for case in d["cases"]:
        got = price_plans_gpu(h, cluster, model, PC._plans_from(case["templates"], case["n_tmpl"], W))
        e = case["expect"]
        assert got["status"][:, 0].tolist() == e["status"], case["name"]
        assert got["n_dp"][:, 0].tolist() == e["n_dp"], case["name"]
        assert got["T"][:, 0].tolist() == e["T"], case["name"]
        assert int(got["placed"][0]) == e["placed"], case["name"]
        assert float(got["thr"][0]) == e["thr"], case["name"]


def test_plans_limits(h, W):
    import torch
    w = W.make_workload("tiny", seed=0)
    plans = W.make_plans(w, 10, 2, seed=0)
    ctx = h.heddle_create(0)
    try:
        h.heddle_load_cluster(ctx, w.cluster)
        h.heddle_load_model(ctx, w.model)
        dp = h.plans_to_device(plans)
        pr = h.alloc_plan_results(10, 2)
        h.heddle_price_plans(ctx, dp, pr)
        torch.cuda.synchronize()
        big = W.make_cluster([1000.0], [10**11], [10**11], [(0, 72, 10**10)])
        h.heddle_load_cluster(ctx, big)
        with pytest.raises(h.HeddleError) as e:
            h.heddle_price_plans(ctx, dp, pr)
        assert e.value.status == 3  # E_LIMIT: a node above the plan limit
    finally:
        h.heddle_destroy(ctx)


ROUTES = {"threads": 0, "warps": 2**31 - 1, "default": None}


def _bounds_same(orc, plans, got, idx=None):
    """OK templates hold their standalone split (the oracle's), others zeros;
    of every plan, or of plans idx."""
    idx = slice(None) if idx is None else idx
    for t, b in enumerate(got["bounds"]):
        alone = orc.price({"S": np.ascontiguousarray(plans["S"][t][idx]), "M": np.ascontiguousarray(plans["M"][t][idx]),
                           "code": np.ascontiguousarray(plans["code"][t][:, idx])}, bounds=True)
        ok = got["status"][t][idx] == 0
        assert (b[:, idx][:, ok] == alone["bounds"][:, ok]).all(), t
        assert (b[:, got["status"][t] != 0] == 0).all(), t


@pytest.mark.parametrize("name,n", [("tiny", 33), ("dense32", 1), ("dense32", 4001), ("moe48", 2003),
                                    ("stress128", 1501)])
@pytest.mark.parametrize("route", ROUTES)
def test_plan_walk_routes(h, W, oracle_mod, name, n, route):
    """Every walking plan by a thread, by a warp, and by the default rule, with
    memory that most templates fit (so that plans walk to their last one)."""
    w = W.make_workload(name, seed=2, n=n)
    w.cluster["mem_bytes"][:] = 10**12
    plans = W.make_plans(w, n, 4, seed=2)
    orc = oracle_mod.Oracle(w.cluster, w.model)
    ref = orc.price_plans(plans)
    got = price_plans_gpu(h, w.cluster, w.model, plans, bounds=True, thread_min=ROUTES[route])
    assert got["errors"] == 0
    _same(got, ref, "%s %s" % (name, route))
    _bounds_same(orc, plans, got)
    if n > 1000:
        assert (ref["placed"] >= 2).mean() > 0.2


@pytest.mark.parametrize("deepest", [2, 5])
def test_plan_walk_queues_fill(h, W, oracle_mod, deepest):
    """200,003 plans, most of which walk: a CTA looks at 128 at a time, its
    queue passes 128 and leaves a remainder.  The routes against each other,
    and the default one against the oracle on a sample."""
    n = 200_003
    w = W.make_workload("dense32", seed=5, n=n)
    w.cluster["mem_bytes"][:] = 10**12
    plans = W.make_plans(w, n, 4, seed=5)
    plans["S"] = np.minimum(plans["S"], deepest).astype(plans["S"].dtype)
    plans["code"] = np.ascontiguousarray(plans["code"][:, :deepest])
    plans["code"][np.arange(deepest)[None, :, None] >= plans["S"][:, None, :]] = 0
    got = {r: price_plans_gpu(h, w.cluster, w.model, plans, bounds=True, thread_min=m) for r, m in ROUTES.items()}
    walks = (got["warps"]["status"][0] == 0) & (plans["n_tmpl"] >= 2)
    assert walks.mean() > 0.6
    for r in ROUTES:
        assert got[r]["errors"] == 0
        _same(got[r], got["warps"], "%s against warps" % r)
        for t in range(4):
            assert (got[r]["bounds"][t] == got["warps"]["bounds"][t]).all(), (r, t)
    idx = np.random.default_rng(1).choice(n, 3000, replace=False)
    some = {"n_tmpl": plans["n_tmpl"][idx], "S": np.ascontiguousarray(plans["S"][:, idx]),
            "M": np.ascontiguousarray(plans["M"][:, idx]), "code": np.ascontiguousarray(plans["code"][:, :, idx])}
    orc = oracle_mod.Oracle(w.cluster, w.model)
    ref = orc.price_plans(some)
    d = got["default"]
    _same({k: d[k][..., idx] for k in ("T", "bottleneck", "n_dp", "status", "placed", "thr")}, ref, "sample")
    _bounds_same(orc, plans, d, idx)
