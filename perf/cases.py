"""Cases of use for timing the pricer: what a planner has it do, through the
public entry points of ``paper_2609_34244_gb300.heddle``.

A case is a dict of plain values: which call is made (``path``), the model
(``layers``, ``hidden``, ``seq``, ``moe``, ``ragged``), the cluster
(``types``, ``gpus``, ``nodes``, ``speed_lo``, ``mem_lo`` .. ``mem_hi`` GB),
the candidates (``n``, ``s_max``, ``micro``: the microbatch counts they draw
from) and the call's options (``k``, ``bounds``, ``levels``, ``slots``,
``batch``, ``planes``).  Every array comes from the seed alone.
"""

import fractions
import math

import numpy as np
import torch

from paper_2609_34244_gb300 import heddle as h
from paper_2609_34244_gb300 import workloads as W

GB = 10**9

# The repository's workload shapes.
_DENSE32 = dict(layers=32, hidden=4096, seq=2048, moe=False, ragged=False, types=3, gpus=64, nodes="4,8",
                speed_lo=0.3, mem_lo=24, mem_hi=80, s_max=8, degree=4, micro="32")
_DENSE80 = dict(layers=80, hidden=8192, seq=4096, moe=False, ragged=False, types=5, gpus=256, nodes="4,8",
                speed_lo=0.2, mem_lo=16, mem_hi=80, s_max=16, degree=8, micro="16,32,64,128")
_STRESS = dict(layers=128, hidden=12288, seq=4096, moe=False, ragged=False, types=8, gpus=1024, nodes="2,4,8",
               speed_lo=0.1, mem_lo=16, mem_hi=192, s_max=32, degree=8, micro="256")
_MOE48 = dict(layers=48, hidden=4096, seq=2048, moe=True, ragged=False, types=4, gpus=128, nodes="4,8",
              speed_lo=0.3, mem_lo=40, mem_hi=141, s_max=12, degree=8, micro="64")
_OPTIONS = dict(k=16, bounds=False, levels=0, slots=0, batch=0, planes=False)


def _case(name, path, shape, n, **options):
    return {"name": name, "path": path, **shape, **_OPTIONS, "n": n, **options}


def listed():
    return [
        # the cluster changed (a node joined or left): load the new cluster
        # and model, price every small structure with its split, rank
        _case("replan_small", "replan", dict(_DENSE32, layers=8, types=2, gpus=16, s_max=3, degree=2, micro="1,2,4,8"),
              336, bounds=True),
        # one rollout batch of a planner's search: a thousand structures,
        # their splits wanted; latency and launches count
        _case("rollout_1k", "price_topk", _DENSE32, 1000, bounds=True),
        # a sweep of random structures of a mid-size dense model
        _case("dense32_100k", "price_topk", _DENSE32, 100_000),
        # the same of a large dense model, several microbatch counts
        _case("dense80_1m", "price_topk", _DENSE80, 1_000_000),
        # the largest sweep: 1e7 structures, 1024 GPUs of 8 types
        _case("stress128_10m", "price_topk", _STRESS, 10_000_000),
        # the large sweep streamed from host memory in batches
        _case("stress128_host", "host", _STRESS, 3_000_001, batch=1_000_000),
        # alternating dense and expert blocks (layers differ, memory binds)
        _case("moe48_1m", "price_topk", _MOE48, 1_000_000),
        # a profiled model whose layers all differ; splits wanted, priced and
        # ranked in two calls, an odd batch size
        _case("profiled80_300k", "price", dict(_DENSE80, ragged=True), 300_007, bounds=True),
        # micro-batch-size fill over four profiled sizes
        _case("fill_dense80_250k", "mbs", _DENSE80, 250_000, levels=4),
        # plans of up to four pipelines sharing the cluster
        _case("plans_200k", "plans", _STRESS, 200_003, slots=4),
        # expert tiling of every stage
        _case("tiling_moe48_200k", "tiled", _MOE48, 200_001),
        # the paper's proportional split, to compare plans against
        _case("split_rule_1m", "split", _STRESS, 1_000_000),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


# per call: the shapes it is used with and its largest batch
_DRAWN = {
    "replan": ((_DENSE32, _DENSE80, _STRESS), 20_000),
    "price_topk": ((_DENSE32, _DENSE80, _STRESS, _STRESS, _MOE48), 10_000_000),
    "price": ((_DENSE32, _DENSE80, _STRESS, _MOE48), 1_000_000),
    "host": ((_DENSE80, _STRESS), 3_000_000),
    "mbs": ((_DENSE32, _DENSE80), 250_000),
    "plans": ((_DENSE80, _STRESS), 200_000),
    "tiled": ((_MOE48,), 200_000),
    "split": ((_DENSE80, _STRESS), 1_000_000),
}


def draw(rng):
    path = rng.choice(("replan", "price_topk", "price_topk", "price_topk", "price", "price", "host", "mbs", "plans",
                       "tiled", "split"))
    shapes, most = _DRAWN[path]
    c = {"path": path, **rng.choice(shapes), **_OPTIONS}
    c["layers"] = rng.randint(max(6, c["layers"] // 4), c["layers"])
    c["types"] = rng.randint(1 if not c["moe"] else 2, c["types"])
    c["gpus"] = rng.randint(max(16, c["gpus"] // 4), c["gpus"])
    c["s_max"] = rng.randint(2, min(c["s_max"], c["layers"]))
    c["micro"] = rng.choice((c["micro"], "1,2,4,8", "12,48", "64"))
    c["ragged"] = path in ("replan", "price_topk", "price") and not c["moe"] and rng.random() < 0.4
    if c["ragged"] or c["moe"]:
        most = min(most, 300_000)  # the general search costs more per candidate
    c["n"] = _log_int(rng, 64, most)
    c["k"] = rng.choice((1, 8, 16, 16, 16, 64))
    c["bounds"] = path not in ("host", "tiled") and c["n"] <= 300_000 and rng.random() < 0.5
    c["levels"] = rng.randint(2, 4) if path == "mbs" else 0
    c["slots"] = rng.randint(2, 4) if path == "plans" else 0
    c["batch"] = rng.choice((100_000, 1_000_000)) if path == "host" else 0
    c["planes"] = path == "host" and c["n"] <= 1_000_000 and rng.random() < 0.5
    return c


# ------------------------------------------------------------------- inputs

def _cluster(case, rng):
    """Types of random speed and memory; nodes of the listed sizes, every
    type owning at least one."""
    nt = case["types"]
    sizes = [int(z) for z in case["nodes"].split(",")]
    nodes, left = [], case["gpus"]
    while left >= min(sizes):
        nodes.append(int(rng.choice([z for z in sizes if z <= left])))
        left -= nodes[-1]
    while len(nodes) < nt:
        i = int(np.argmax(nodes))
        nodes[i:i + 1] = [nodes[i] // 2, nodes[i] - nodes[i] // 2]
    types = list(range(nt)) + [int(t) for t in rng.integers(0, nt, len(nodes) - nt)]
    nic = rng.choice(np.asarray([25, 100, 400]), len(nodes)) * (GB // 8)
    return W.make_cluster(1000.0 * rng.uniform(case["speed_lo"], 1.0, nt),
                          rng.integers(case["mem_lo"], case["mem_hi"] + 1, nt) * GB,
                          rng.choice(np.asarray([64, 300, 900]), nt) * GB,
                          [(t, z, int(b)) for t, z, b in zip(types, nodes, nic)])


def _model(case, cluster, rng):
    """Transformer blocks in bf16 with Adam.  MoE: every second block holds
    64 experts (top-2).  Ragged: a profile in which every layer differs, the
    first and last (embedding, head) most."""
    L, hid, s = case["layers"], case["hidden"], case["seq"]
    tok, attn = 2 * s * hid, 4 * hid * hid
    if case["moe"]:
        ffn, experts = 14336, 64
        expert = np.arange(L) % 2 == 1
        e_only = np.where(expert, experts * 3 * hid * ffn, 0)
        params = np.where(expert, attn + e_only + hid * experts, attn + 3 * hid * ffn)
        used = np.where(expert, attn + 2 * 3 * hid * ffn, attn + 3 * hid * ffn)
        flops = 3.0 * (2 * s * used + 4 * s * s * hid)
        act = np.where(expert, 68, 34) * s * hid
        return W.make_model(flops, 2 * params, 16 * params, act, np.where(expert, tok // 2, tok),
                            np.where(expert, tok, 0), tok, moe=True, expert_state=16 * e_only,
                            expert_param=2 * e_only)
    params = np.full(L, 12 * hid * hid)
    flops = 3.0 * (2 * s * params + 4 * s * s * hid)
    profile = None
    if case["ragged"]:
        w = rng.uniform(0.9, 1.1, L)
        w[0], w[-1] = 0.3, 1.6
        params[[0, -1]] = params[[0, -1]] * 13 // 10
        k = 2.0 ** np.arange(4)
        base = flops.mean() / (cluster["tflops"] * 1e12)
        profile = base[:, None, None] * (1.0 + 0.05 * np.arange(4))[None, :, None] / k[None, :, None] * w
    return W.make_model(flops, 2 * params, 16 * params, np.full(L, 34 * s * hid), tok, 0, tok, profile_s=profile)


def _size_profiles(case, cluster, rng):
    """Seconds per layer at micro-batch sizes 2**i: a larger one uses the GPU better."""
    nt, L = case["types"], case["layers"]
    tau, rho = rng.uniform(0.5e-3, 2e-3, nt), rng.uniform(0.6, 0.95, nt)
    j = np.arange(4.0)
    return [np.ascontiguousarray(np.broadcast_to(
        (tau[:, None] * (1.0 + 0.15 * j) / 2.0 ** j * ((2.0 * rho) ** i)[:, None])[:, :, None], (nt, 4, L)))
        for i in range(case["levels"])]


def _candidates(case, cluster, gen):
    """Random structures on the GPU: depth ~ U{1..s_max}, per stage a type
    and a degree it admits; one in a hundred has an inadmissible stage."""
    n, s_max, nt = case["n"], case["s_max"], case["types"]
    biggest = np.zeros(8, np.int64)
    np.maximum.at(biggest, cluster["node_type"], cluster["node_gpus"])
    degrees = [1 << j for j in range(4) if (1 << j) <= case["degree"]]
    allowed = [max(1, len([d for d in degrees if case["moe"] or d <= biggest[t]])) for t in range(nt)]
    cnt = torch.tensor(allowed, dtype=torch.int32, device="cuda")

    def draw_int(high, size, dtype):
        return torch.randint(0, high, size, generator=gen, dtype=dtype, device="cuda")

    S = draw_int(s_max, (n,), torch.uint8) + 1
    code = torch.empty((s_max, n), dtype=torch.uint8, device="cuda")
    for s in range(s_max):
        g = draw_int(nt, (n,), torch.int32)
        j = (draw_int(1 << 16, (n,), torch.int32) * cnt[g]) >> 16
        code[s] = torch.where(S > s, (g | (j << 3)).to(torch.uint8), 0)
    bad = draw_int(n, (n // 100,), torch.int64)
    at = (torch.rand(bad.shape, generator=gen, device="cuda") * S[bad]).to(torch.int64)
    code[at, bad] = code[at, bad] | 0x20
    counts = torch.tensor([int(m) for m in case["micro"].split(",")], dtype=torch.int16, device="cuda")
    M = counts[draw_int(len(counts), (n,), torch.int64)]
    return {"S": S, "M": M, "code": code}


class _State:
    """What a planner keeps between calls: its context and buffers."""

    def __init__(self):
        self.ctx = h.heddle_create(0)

    def __del__(self):
        h.heddle_destroy(self.ctx)


def _inputs(case, seed):
    rng = np.random.default_rng(seed)
    cluster = _cluster(case, rng)
    model = _model(case, cluster, rng)
    profiles = _size_profiles(case, cluster, rng) if case["path"] == "mbs" else None
    gen = torch.Generator(device="cuda").manual_seed(seed)
    cands = [_candidates(case, cluster, gen) for _ in range(max(1, case["slots"]))]
    return cluster, model, profiles, cands, gen


def prepare(case, seed):
    st = _State()
    st.path, st.k, st.batch = case["path"], case["k"], case["batch"]
    st.cluster, st.model, profiles, cands, gen = _inputs(case, seed)
    n = case["n"]
    if st.path != "replan":
        h.heddle_load_cluster(st.ctx, st.cluster)
        h.heddle_load_model(st.ctx, st.model)
    if st.path == "host":
        st.cands = {"S": cands[0]["S"].cpu().pin_memory(), "M": cands[0]["M"].cpu().pin_memory(),
                    "code": cands[0]["code"].cpu().pin_memory()}
        st.res = None
        if case["planes"]:
            dtypes = {"T": torch.int64, "bottleneck": torch.int64, "n_dp": torch.int16, "status": torch.uint8}
            st.res = {key: torch.empty(n, dtype=d, pin_memory=True) for key, d in dtypes.items()}
        return st
    if st.path == "plans":
        st.plans = {"n_tmpl": torch.randint(1, case["slots"] + 1, (n,), generator=gen, dtype=torch.uint8,
                                            device="cuda"), "slots": cands}
        st.res = h.alloc_plan_results(n, case["slots"], bounds=case["bounds"])
        return st
    st.cands = cands[0]
    st.res = h.alloc_results(n, bounds=case["bounds"])
    st.topk = h.alloc_topk_state()
    if st.path == "mbs":
        h.heddle_load_mbs(st.ctx, case["levels"], profiles)
        st.mbs = torch.empty(n, dtype=torch.uint8, device="cuda")
    elif st.path == "tiled":
        h.heddle_load_experts(st.ctx, st.model["expert_state_bytes"], st.model["expert_param_bytes"])
        st.tiling = torch.empty((h.MAX_STAGES, n), dtype=torch.uint8, device="cuda")
    elif st.path == "split":
        h.heddle_set_search(st.ctx, h.SEARCH_DISTRIBUTE)
    return st


def run(st):
    ctx = st.ctx
    if st.path == "host":
        top = h.new_topk_state(st.k)
        h.heddle_price_topk_host(ctx, st.cands, st.res, top, st.batch)
        return {"topk": h.topk_state_to_dict(top), "planes": st.res}
    if st.path == "plans":
        h.heddle_price_plans(ctx, st.plans, st.res)
        return st.res
    if st.path == "mbs":
        h.heddle_price_mbs(ctx, st.cands, st.res, st.mbs)
        return {"planes": st.res, "mbs": st.mbs}
    if st.path == "tiled":
        h.heddle_price_tiled(ctx, st.cands, st.res, st.tiling)
        return {"planes": st.res, "tiling": st.tiling}
    if st.path == "replan":
        h.heddle_load_cluster(ctx, st.cluster)
        h.heddle_load_model(ctx, st.model)
    h.heddle_topk_reset(ctx, st.topk, st.k)
    if st.path == "price":
        h.heddle_price_candidates(ctx, st.cands, st.res)
        h.heddle_topk(ctx, st.cands, st.res, st.topk)
    else:
        h.heddle_price_topk(ctx, st.cands, st.res, st.topk)
    return {"planes": st.res, "topk": st.topk}


def work(case):
    """Each candidate's depth, microbatch count and stage bytes read once,
    its result row written once; integer operations: eight to decode a stage
    and add up its demand and memory, twenty to decide a candidate."""
    n, stages = case["n"], (case["s_max"] + 1) / 2
    priced = n * max(1, case["slots"]) * max(1, case["levels"])
    read = n * max(1, case["slots"]) * (3 + stages)
    row = 19 + (33 if case["bounds"] else 0)
    if case["path"] == "host":
        row = 19 if case["planes"] else 0
    written = n * max(1, case["slots"]) * row
    if case["path"] == "mbs":
        written += n
    if case["path"] == "tiled":
        written += h.MAX_STAGES * n
    if case["path"] == "plans":
        read += n
        written += 9 * n
    return {"bytes": read + written, "flops": priced * (8 * stages + 20)}


def tolerance(case):
    """Whole nanoseconds, counts and codes (and a sum of doubles in a stated
    order): there is one right answer."""
    return "exact"


# ------------------------------------------------------- plain 64-bit answers

_INF = 1 << 62


def _tables(case, cluster, model):
    """Per (type, degree) the prefix of the layer times in ns, and the
    cluster's statistics per type, by the header's formula."""
    nt, L = case["types"], case["layers"]
    owner, size, nic = cluster["node_type"], cluster["node_gpus"], cluster["node_nic"]
    maxn = np.array([size[owner == t].max() for t in range(nt)])
    far = np.array([nic[owner == t].min() for t in range(nt)])
    cap = np.array([[int((size[owner == t] >> e << e).sum()) for e in range(4)] for t in range(nt)])
    q = np.zeros((nt, 4, L), np.int64)
    for t in range(nt):
        for j in range(4):
            k = float(1 << j)
            if model["profile_s"] is not None:
                s = model["profile_s"][t, j]
            else:
                s = model["flops"] / (k * cluster["tflops"][t] * 1e12)
                if j:
                    bw = float(cluster["intra_bw"][t] if (1 << j) <= maxn[t] else far[t])
                    s = s + 4.0 * (2.0 * (k - 1.0) / k) * model["ar_bytes"].astype(np.float64) / bw
                    s = s + 4.0 * ((k - 1.0) / k) * model["a2a_bytes"].astype(np.float64) / bw
            ns = s * 1e9
            q[t, j] = np.trunc(ns) + (ns - np.trunc(ns) >= 0.5)
    prefix = np.concatenate([np.zeros((nt, 4, 1), np.int64), np.cumsum(q, axis=2)], axis=2)
    p2p = np.zeros((nt, nt, 2), np.int64)
    for a in range(nt):
        for b in range(nt):
            for same in range(2):
                bw = int(cluster["intra_bw"][a]) if same else int(min(far[a], far[b]))
                p2p[a, b, same] = -(-2 * model["boundary_bytes"] * GB // bw)
    return {"maxn": maxn, "far": far, "cap": cap, "prefix": prefix, "p2p": p2p}


def _price_block(case, cluster, model, tab, S, M, code):
    """Candidates of one block (GPU tensors): status, n, T, B and boundaries
    by a dynamic programme over every split."""
    dev, L, nt, s_max = S.device, case["layers"], case["types"], case["s_max"]
    n = S.shape[0]
    as_t = lambda x: torch.as_tensor(np.ascontiguousarray(x), device=dev)  # noqa: E731
    S, M, code = S.long(), M.long(), code.long()
    live = torch.arange(s_max, device=dev)[:, None] < S[None, :]
    g, j = code & 7, (code >> 3) & 3
    gc = g.clamp(max=nt - 1)
    maxn = as_t(tab["maxn"])
    bad = ((code >> 5) != 0) | (g >= nt)
    if not case["moe"]:
        bad |= (1 << j) > maxn[gc]
    invalid = (bad & live).any(0) | (S > L) | (M < 1)
    # replicas: groups of size >= 2^e against the capacity in blocks of 2^e
    block = as_t(np.array([max(b for b in (1, 2, 4, 8) if b <= m) for m in tab["maxn"]]))
    unit = torch.minimum(1 << j, block[gc])
    reps = torch.full((n,), _INF, device=dev)
    for t in range(nt):
        for e in range(4):
            dem = torch.where(live & (g == t) & (unit >= (1 << e)), 1 << j, 0).sum(0)
            reps = torch.where(dem > 0, torch.minimum(reps, int(tab["cap"][t, e]) // dem.clamp(min=1)), reps)
    SA = as_t(np.concatenate([[0], np.cumsum(model["state_bytes"])]))
    AA = as_t(np.concatenate([[0], np.cumsum(model["act_bytes"])]))
    mem = as_t(cluster["mem_bytes"])
    prefix, p2p = as_t(tab["prefix"]), as_t(tab["p2p"])
    pos = torch.arange(L + 1, device=dev)
    later = pos[None, :] > pos[:, None]

    def stage_times(s):  # [n, i, j]: time of layers [i, j) on stage s, _INF where it does not fit
        gs, js = gc[s], j[s]
        nxt = min(s + 1, s_max - 1)
        near = (gs == gc[nxt]) & ((1 << js) + (1 << j[nxt]) <= maxn[gs])
        c = torch.where(S > s + 1, p2p[gs, gc[nxt], near.long()], 0)
        row = prefix[gs, js]
        f = torch.minimum(S - s, M)
        foot = SA[None, :] + f[:, None] * AA[None, :]
        fits = (foot[:, None, :] - foot[:, :, None] <= (mem[gs] << js)[:, None, None]) & later
        return torch.where(fits, row[:, None, :] - row[:, :, None] + c[:, None, None], _INF)

    best = torch.full((n, L + 1), _INF, device=dev)
    best[:, 0] = 0
    B = torch.full((n,), _INF, device=dev)
    for s in range(s_max):
        best = torch.maximum(best[:, :, None], stage_times(s)).amin(1)
        B = torch.where(S == s + 1, best[:, L], B)
    status = torch.where(invalid, 3, torch.where(reps < 1, 2, torch.where(B >= _INF, 1, 0)))
    ok = status == 0
    # the smallest boundaries: from the suffixes that can be finished within B
    can = torch.zeros((s_max + 1, n, L + 1), dtype=torch.bool, device=dev)
    for s in range(s_max - 1, -1, -1):
        can[s + 1, :, L] |= S == s + 1
        can[s] = ((stage_times(s) <= B[:, None, None]) & can[s + 1][:, None, :]).any(2)
    rows = torch.arange(n, device=dev)
    bounds = torch.zeros((33, n), dtype=torch.int64, device=dev)
    at = torch.zeros(n, dtype=torch.int64, device=dev)
    total, grad = torch.zeros_like(B), torch.zeros_like(B)
    PB = as_t(np.concatenate([[0], np.cumsum(model["param_bytes"])]))
    far = as_t(tab["far"])
    for s in range(s_max):
        times = stage_times(s)[rows, at]
        end = ((times <= B[:, None]) & can[s + 1]).to(torch.uint8).argmax(1)
        on = ok & live[s]
        total += torch.where(on, times[rows, end], 0)
        # ceil(2 (n - 1) G 1e9 / (n k bw)) by long division in base 1000
        den = (reps.clamp(max=1 << 20) * far[gc[s]]).clamp(min=1) << j[s]
        num = torch.where(on, 2 * (reps.clamp(max=1 << 20) - 1) * (PB[end] - PB[at]), 0)
        quo, rem = num // den, num % den
        for _ in range(3):
            quo, rem = quo * 1000 + rem * 1000 // den, rem * 1000 % den
        grad = torch.maximum(grad, quo + (rem > 0).long())
        at = torch.where(on, end, at)
        bounds[s + 1] = torch.where(on, end, 0)
    T = torch.where(ok, (M - 1) * B + total + grad, -1)
    return {"T": T, "bottleneck": torch.where(ok, B, -1), "n_dp": torch.where(status <= 1, reps, 0).to(torch.int16),
            "status": status.to(torch.uint8), "bounds": bounds.to(torch.uint8)}


def _rank(case, planes, M):
    """The k best by throughput n M / T, exactly compared, then by index."""
    k = case["k"]
    nM = (planes["n_dp"].long() & 0xffff) * M.long()
    key = torch.where(planes["status"] == 0, nM.double() / planes["T"].double(), -1.0)
    few = torch.nonzero(key >= max(0.0, float(key.topk(min(k, case["n"])).values[-1]) * (1 - 1e-12)))[:, 0].tolist()
    T, nM = planes["T"].tolist(), nM.tolist()
    few = sorted(few, key=lambda i: (-fractions.Fraction(nM[i], T[i]), i))[:k]
    return few, [T[i] for i in few], [nM[i] for i in few]


def _state_bytes(case, few, T, nM):
    """The top-k as the device structure lays it out (-1 and 0 past the end)."""
    pad = h.MAX_TOPK - len(few)
    return torch.from_numpy(np.concatenate([
        np.array([case["k"], len(few)], np.int32).view(np.uint8),
        np.array(few + [-1] * pad, np.int64).view(np.uint8), np.array(T + [-1] * pad, np.int64).view(np.uint8),
        np.array(nM + [0] * pad, np.uint32).view(np.uint8)]).copy())


def exact(case, seed):
    """The pricing calls' answer; the fill, the plans, the tiling and the
    paper's split have none here, nor have batches too large for a dynamic
    programme over every split."""
    if case["path"] not in ("replan", "price", "price_topk", "host"):
        return None
    cells = case["s_max"] * (case["layers"] + 1) ** 2
    if case["n"] * cells > 4e9:
        return None
    cluster, model, _, cands, _ = _inputs(case, seed)
    c, tab = cands[0], _tables(case, cluster, model)
    step = max(1, int(2e8) // (case["layers"] + 1) ** 2)
    blocks = [_price_block(case, cluster, model, tab, c["S"][lo:lo + step], c["M"][lo:lo + step],
                           c["code"][:, lo:lo + step]) for lo in range(0, case["n"], step)]
    planes = {key: torch.cat([b[key] for b in blocks], dim=-1) for key in blocks[0]}
    few, T, nM = _rank(case, planes, c["M"])
    if not case["bounds"]:
        planes["bounds"] = None
    if case["path"] == "host":
        planes.pop("bounds")
        top = {"k": case["k"], "count": len(few), "idx": np.array(few, np.int64), "T": np.array(T, np.int64),
               "nM": np.array(nM, np.uint32)}
        return {"topk": top, "planes": planes if case["planes"] else None}
    return {"planes": planes, "topk": _state_bytes(case, few, T, nM)}
