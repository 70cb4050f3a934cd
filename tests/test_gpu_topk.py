"""heddle_topk over seeded result planes built to stress its filters:
throughput rising along the batch (so an unsorted slice keeps producing new
bests), near-ties whose float keys n*M / T are equal while their exact order
is not, exact ties in throughput with other factors, and a second call into
the filled state; k on both sides of 32 (the first pass that sets a floor
runs for k <= 32 while the state is not full).  Compared with the oracle's
top-k of everything offered so far."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

KS = (1, 16, 32, 33, 64)


def _planes(n, seed, n_top):
    rng = np.random.default_rng(seed)
    # T falls along the batch: n*M / T rises with the index
    T = (np.int64(1) << 40) - np.arange(n, dtype=np.int64) * 4096 - rng.integers(0, 4096, n)
    ndp = np.full(n, 8, np.uint16)
    M = np.full(n, 64, np.uint16)
    status = np.where(rng.random(n) < 0.7, 0, rng.integers(1, 4, n)).astype(np.uint8)
    # the best n_top: T within 2 of 2^39 (equal float keys, distinct exact
    # keys), a third of them at twice T with twice n (exact ties)
    top = rng.choice(n, n_top, replace=False)
    T[top] = (np.int64(1) << 39) + rng.integers(0, 3, n_top)
    status[top] = 0
    twin = top[: n_top // 3]
    T[twin] *= 2
    ndp[twin] = 16
    return {"T": T, "n_dp": ndp, "M": M, "status": status}


def _run_topk(h, ctx, planes, base, state):
    import torch
    n = int(planes["T"].shape[0])
    dev = {key: torch.from_numpy(v.view(np.int16) if v.dtype == np.uint16 else v).cuda()
           for key, v in planes.items()}
    c = h.heddle_candidates(dev["M"].data_ptr(), dev["M"].data_ptr(), dev["M"].data_ptr(), n, n, 1, 0, base)
    r = h.heddle_results(dev["T"].data_ptr(), dev["T"].data_ptr(), dev["n_dp"].data_ptr(),
                         dev["status"].data_ptr(), None)
    h.heddle_topk(ctx, c, r, state)
    torch.cuda.synchronize()
    return h.read_topk_state(state)


def _same_state(got, exp, what):
    assert got["count"] == exp["count"], what
    n = exp["count"]
    for key in ("idx", "T", "nM"):
        assert np.array_equal(np.asarray(got[key])[:n], np.asarray(exp[key])[:n]), "%s: %s" % (what, key)


@pytest.mark.parametrize("k", KS)
@pytest.mark.parametrize("n_top", (10, 150))
def test_topk_rising_batch_and_near_ties(heddle_lib, oracle_mod, k, n_top):
    import torch
    h = heddle_lib
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    first = _planes(300_001, 3 + k, n_top)
    second = _planes(123_457, 7 + k, n_top)
    state = h.alloc_topk_state()
    ctx = h.heddle_create(0)
    try:
        h.heddle_topk_reset(ctx, state, k)
        got1 = _run_topk(h, ctx, first, 0, state)
        exp1 = oracle_mod.topk({key: first[key] for key in ("T", "n_dp", "status")}, first["M"], k)
        assert exp1["count"] == k
        _same_state(got1, exp1, "k=%d, %d best, first call" % (k, n_top))
        got2 = _run_topk(h, ctx, second, first["T"].shape[0], state)
        union = {key: np.concatenate([first[key], second[key]]) for key in ("T", "n_dp", "status", "M")}
        exp2 = oracle_mod.topk({key: union[key] for key in ("T", "n_dp", "status")}, union["M"], k)
        _same_state(got2, exp2, "k=%d, %d best, second call" % (k, n_top))
    finally:
        h.heddle_destroy(ctx)


@pytest.mark.parametrize("n", (1, 31, 32, 33, 127, 129, 1023, 1024, 1025, 2049, 40_000, 500_009))
@pytest.mark.parametrize("kind", ("all_tie", "two_levels", "few_ok", "zero_time"))
def test_topk_gather_edges(heddle_lib, oracle_mod, n, kind):
    """Batch sizes around one entry a lane, one CTA and several, with ties
    that overflow the gather (every throughput equal; half of them), fewer OK
    entries than k, and iteration times of zero; two calls into one state."""
    h = heddle_lib
    rng = np.random.default_rng(n)
    T = rng.integers(1 << 30, 1 << 40, 2 * n)
    status = np.zeros(2 * n, np.uint8)
    if kind == "all_tie":
        T[:] = 1 << 35
    elif kind == "two_levels":
        T = np.where(rng.random(2 * n) < 0.5, 1 << 35, 1 << 34)
    elif kind == "few_ok":
        status[:] = 1
        status[rng.choice(2 * n, min(2 * n, 5), replace=False)] = 0
    else:
        T[rng.random(2 * n) < 0.3] = 0
    planes = {"T": T.astype(np.int64), "status": status, "n_dp": rng.integers(1, 3, 2 * n).astype(np.uint16)
              if kind == "zero_time" else np.full(2 * n, 4, np.uint16), "M": np.full(2 * n, 16, np.uint16)}
    ctx = h.heddle_create(0)
    try:
        for k in (1, 16, 64):
            state = h.alloc_topk_state()
            h.heddle_topk_reset(ctx, state, k)
            for lo in (0, n):
                got = _run_topk(h, ctx, {key: v[lo:lo + n] for key, v in planes.items()}, lo, state)
                part = {key: v[:lo + n] for key, v in planes.items()}
                exp = oracle_mod.topk(part, part["M"], k)
                _same_state(got, exp, "%s n=%d k=%d up to %d" % (kind, n, k, lo + n))
    finally:
        h.heddle_destroy(ctx)


@pytest.mark.parametrize("layers", ("all_free", "some_types_free"))
@pytest.mark.parametrize("chunk", (None, 701))
def test_price_topk_keeps_iteration_times_of_zero(heddle_lib, oracle_mod, layers, chunk):
    """Layers that round to 0 ns on every GPU type, or on the fast one only,
    with no P2P and no gradient bytes: an OK candidate whose iteration time is
    0 ranks first.  The fused call (one chunk, several) and the host call hold
    the same state as the oracle's ranking of all results."""
    from paper_2609_34244_gb300 import workloads as W
    import gpu_helpers as G
    h = heddle_lib
    rng = np.random.default_rng(3)
    cluster = W.make_cluster([1000.0, 100.0, 10.0], [10**12] * 3, [10**11] * 3,
                             [(g, z, 10**10) for g in range(3) for z in (4, 8)] * 4)
    # 3e5 FLOPs: 0.3 ns on the first type, 3 and 30 on the others
    model = W.make_model(np.full(12, 0.0 if layers == "all_free" else 3e5), 0, 10**6, 10**5, 0, 0, 0)
    n = 3001
    S = rng.integers(1, 4, n).astype(np.uint8)
    code = W.encode(rng.integers(0, 3, (3, n)), rng.integers(0, 3, (3, n)))
    code[np.arange(3)[:, None] >= S[None, :]] = 0
    cands = W.make_cands(S, rng.choice([1, 4, 64], n).astype(np.uint16), code)
    ref = oracle_mod.Oracle(cluster, model).price(cands, threads=8)
    assert ((ref["T"] == 0) & (ref["status"] == 0)).sum() > 64
    for k in (1, 16, 64):
        exp = oracle_mod.topk(ref, cands["M"], k)
        for search in (0, 1):
            got = G.price_gpu(h, cluster, model, cands, k=k, search=search, fused=True, chunk=chunk)
            assert got["errors"] == 0
            G.assert_same(got, ref, what=layers)
            _same_state(got["topk"], exp, "%s k=%d search %d" % (layers, k, search))
        ctx = h.heddle_create(0)
        try:
            h.heddle_load_cluster(ctx, cluster)
            h.heddle_load_model(ctx, model)
            state = h.new_topk_state(k)
            h.heddle_price_topk_host(ctx, cands, None, state, chunk or n)
            _same_state(h.topk_state_to_dict(state), exp, "%s k=%d host" % (layers, k))
        finally:
            h.heddle_destroy(ctx)


@pytest.mark.parametrize("kind", ("random", "rising", "falling", "equal", "few_ok"))
def test_topk_posted_bars(heddle_lib, oracle_mod, kind):
    """CTA counts on both sides of the number from which bars are posted (4,096 /
    k CTAs of 1,024 entries), in every order, thrice into one state and again
    in another batch: the flags are clear for the next launch."""
    h = heddle_lib
    rng = np.random.default_rng(5)
    ctx = h.heddle_create(0)
    try:
        for k, ns in ((64, (64_000, 66_000, 400_000)), (16, (261_000, 264_000, 400_000)), (13, (320_000,))):
            for n in ns:
                T = rng.integers(1 << 30, 1 << 40, 3 * n)
                status = np.zeros(3 * n, np.uint8)
                if kind == "rising":
                    T.sort()
                elif kind == "falling":
                    T = np.sort(T)[::-1].copy()
                elif kind == "equal":
                    T[:] = 1 << 35
                elif kind == "few_ok":
                    status[:] = 1
                    status[rng.choice(3 * n, 9, replace=False)] = 0
                planes = {"T": T, "status": status, "n_dp": np.full(3 * n, 4, np.uint16),
                          "M": np.full(3 * n, 16, np.uint16)}
                state = h.alloc_topk_state()
                h.heddle_topk_reset(ctx, state, k)
                for i in range(3):
                    lo, hi = i * n, (i + 1) * n
                    got = _run_topk(h, ctx, {key: v[lo:hi] for key, v in planes.items()}, lo, state)
                    part = {key: v[:hi] for key, v in planes.items()}
                    _same_state(got, oracle_mod.topk(part, part["M"], k), "%s n=%d k=%d call %d" % (kind, n, k, i))
    finally:
        h.heddle_destroy(ctx)
