"""The paper's own layer split (search mode DISTRIBUTE, §5.3 "Layer split
and DP degree") on the GPU through the C ABI against the oracle's same
rule: bit-exact T, bottleneck, n_dp, status, bounds and top-k."""

import numpy as np
import pytest

import gpu_helpers as G

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


@pytest.mark.parametrize("name,n", [("tiny", None), ("tiny_ext", None), ("dense32", 6007), ("dense80", 1531),
                                    ("moe48", 6011), ("stress128", 613)])
@pytest.mark.parametrize("seed", [0, 1])
def test_distribute_parity(h, W, oracle_mod, name, n, seed):
    w = W.make_workload(name, seed=seed, n=n)
    ref = oracle_mod.Oracle(w.cluster, w.model).set_split("distribute").price(w.cands, threads=8)
    got = G.price_gpu(h, w.cluster, w.model, w.cands, k=16, search=h.SEARCH_DISTRIBUTE)
    assert got["errors"] == 0
    assert got["search"] == h.SEARCH_DISTRIBUTE
    G.assert_same(got, ref, what="%s distribute" % name)
    tk = oracle_mod.topk(ref, w.cands["M"], 16)
    assert got["topk"]["idx"].tolist() == tk["idx"].tolist()


def test_distribute_hand_cases(h, W, oracle_mod):
    """The hand-worked cases of the paper's rule, on the GPU."""
    import json
    import os
    path = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "hand_distribute.json")
    for case in json.load(open(path))["cases"]:
        nt = len(case["tflops"])
        cluster = W.make_cluster(case["tflops"], case["mem_bytes"], [300 * 10**9] * nt,
                                 [tuple(x) for x in case["nodes"]])
        model = W.make_model(case["flops"], 0, case["state_bytes"], case["act_bytes"], 0, 0, 0)
        cands = W.from_structures([[tuple(s) for s in case["stages"]]], [4])
        got = G.price_gpu(h, cluster, model, cands, search=h.SEARCH_DISTRIBUTE)
        e = case["expect"]
        assert int(got["status"][0]) == e["status"], case["name"]
        assert int(got["T"][0]) == e["T"], case["name"]
        assert int(got["bottleneck"][0]) == e["bottleneck"], case["name"]
        if e["bounds"] is not None:
            S = len(case["stages"])
            assert got["bounds"][: S + 1, 0].tolist() == e["bounds"], case["name"]


def test_distribute_never_beats_the_exact_bottleneck(h, W):
    w = W.make_workload("dense80", seed=3, n=20011)
    exact = G.price_gpu(h, w.cluster, w.model, w.cands, bounds=False)
    dist = G.price_gpu(h, w.cluster, w.model, w.cands, bounds=False, search=h.SEARCH_DISTRIBUTE)
    ok = dist["status"] == 0
    assert ok.sum() > 100
    assert (exact["status"][ok] == 0).all()
    assert (dist["bottleneck"][ok] >= exact["bottleneck"][ok]).all()


@pytest.mark.parametrize("L", [1, 2, 7, 31, 32, 33, 128, 255])
@pytest.mark.parametrize("kind", ["near_tie", "wide", "tight"])
def test_distribute_equal_layers(h, W, oracle_mod, L, kind):
    """The thread-per-entry split of equal-layer models at every depth up to
    the layer count: types of almost the same speed (remainders that differ
    in their last bits), of very different speed (stages with no layer of
    their own, surplus layers to take back), and memory that rejects the
    first alternatives; the fused top-k as well, and the warp kernel that
    small batches take."""
    rng = np.random.default_rng(L)
    nt = 5
    tflops = 100.0 * (1.0 + 1e-9 * np.arange(nt)) if kind == "near_tie" else np.geomspace(1.0, 1000.0, nt)
    mem = rng.integers(2, 9, nt) * 10**9 if kind == "tight" else np.full(nt, 10**15)
    cluster = W.make_cluster(tflops, mem, rng.integers(50, 900, nt) * 10**9,
                             [(g, z, int(rng.integers(1, 50)) * 10**9) for g in range(nt) for z in (2, 4, 8)] * 8)
    model = W.make_model(np.full(L, 3.3e12), 10**8, 8 * 10**9 // max(1, L // 8), 10**8 // max(1, L // 8), 10**6, 0,
                         10**6)
    n = 3000
    S = rng.integers(1, min(L, 32) + 1, n).astype(np.uint8)
    code = W.encode(rng.integers(0, nt, (32, n)), rng.integers(0, 3, (32, n)))
    code[np.arange(32)[:, None] >= S[None, :]] = 0
    cands = W.make_cands(S, rng.choice([1, 3, 64], n).astype(np.uint16), code)
    ref = oracle_mod.Oracle(cluster, model).set_split("distribute").price(cands, threads=8)
    for fused, thread_min in ((False, 0), (True, 0), (False, None)):
        got = G.price_gpu(h, cluster, model, cands, k=16, search=h.SEARCH_DISTRIBUTE, fused=fused,
                          thread_min=thread_min)
        assert got["errors"] == 0
        G.assert_same(got, ref, what="%s L %d" % (kind, L))
        tk = oracle_mod.topk(ref, cands["M"], 16)
        assert got["topk"]["idx"].tolist() == tk["idx"].tolist()


def test_distribute_routes_meet(h, W, oracle_mod):
    """Both kernels of the equal-layer split launched, the entries just enough
    for the thread kernel and one too few; one chunk and several."""
    w = W.make_workload("stress128", seed=6, n=9001)
    ref = oracle_mod.Oracle(w.cluster, w.model).set_split("distribute").price(w.cands, threads=8)
    count = G.price_gpu(h, w.cluster, w.model, w.cands, bounds=False, count=True)["counters"]["priced"]
    assert 0 < count < 9001
    tk = oracle_mod.topk(ref, w.cands["M"], 16)
    for thread_min in (count, count + 1, 9001):
        for chunk in (None, 4000):
            got = G.price_gpu(h, w.cluster, w.model, w.cands, k=16, search=h.SEARCH_DISTRIBUTE, fused=True,
                              chunk=chunk, thread_min=thread_min)
            assert got["errors"] == 0
            G.assert_same(got, ref, what="thread_min %d chunk %s" % (thread_min, chunk))
            assert got["topk"]["idx"].tolist() == tk["idx"].tolist()
