// heddle_eqsearch.cu -- PartitionLayers + Evaluate for models whose layers
// all cost the same (§3.1 listing, §5.2 memory validation, §5.3 iteration
// time), over the worklist the screen kernel produced.
//
// When every layer has the same quantised cost q_s on a stage's (type,
// degree) and the same state and activation bytes, stage s holds exactly
//     cap_s(B) = min(m_s, floor((B - c_s) / q_s))
// layers within bound B (m_s: the longest run of layers that fits the
// stage's memory, c_s: its P2P).  A split with every stage time <= B exists
// iff every cap_s >= 1 and sum_s cap_s >= L, so a probe costs O(S), and
// B* is the smallest such B -- a breakpoint c_s + k q_s of some stage.
//
// First guess, in float only: the continuous balance
// sum_s min(m_s, (B - c_s) / q_s) = L + (stages below their run) / 2 (the
// floors lose half a layer per such stage on average), solved by at most
// three Newton steps from the unsaturated balance.  One exact probe then
// gives every stage's cap at the guess.  The caps are off by a layer or two
// in all, and B* is reached from them one breakpoint at a time:
//   too many: the stages at the largest stage time hi lose their top layer
//   while the count stays at least L and none of them holds its only layer;
//   B* is the largest stage time at which that ends;
//   too few: the stages at the next breakpoint gain a layer until the count
//   is L and every stage holds one; B* is the last of these breakpoints.
// A walk pass costs half a probe.  After kWalk of them, or from further away,
// the next bound interpolates the cap count between the bracket's probes (a
// Newton step while one side is missing), else bisects, and is probed.
// Every stage's cap stays in that stage's word, so Evaluate needs no
// division.  The caps at B* give the componentwise smallest split -- hence
// the lexicographically smallest -- a_{s+1} = max(a_s + 1, L - sum_{t > s}
// cap_t).
//
// Scheduling: the screen files every entry in a bucket per depth S; warp w
// takes entries [32 w, 32 w + 32) of the buckets read in order of
// decreasing S, so its lanes run stage loops of equal length, and then the
// next 32 untaken entries from a counter whenever it is free.  Warps work
// independently (no CTA barrier after the tables are staged): every thread
// packs its candidate's stages once into 32-bit words (cost index | P2P
// index | memory run | cap) held in shared memory interleaved by thread,
// runs the float guess, the exact probe and Evaluate.
//
// Instructions bound it, beside a screen that runs at the same time: hence the
// tables by pair of stages, the float bounds of the guess, the probe that
// keeps the slack to B instead of stage times, the walk instead of a second
// level tracked in every probe, and Evaluate's float comparison.  Largest
// workload, 1e6 candidates: 84 -> 50 us alone; 32-layer workload, 1e5: 28.8 ->
// 19.1; 80-layer workload at four micro-batch sizes, 2.5e5: 37.7 -> 24.3.

#include <algorithm>

#include "heddle_eq.cuh"

namespace hd {
namespace {

constexpr int kMaxIters = 256;
constexpr int kWalk = 4;  // breakpoints walked before the next probe

// Continuous count at Bf (float): sum_s min(m_s, (Bf - c_s) / q_s), with
// the slope sum 1/q_s and the number of stages below their run.
__device__ __forceinline__ float eq_count(const EqTabs& t, const uint32_t* sw, int S, float Bf, float& slope,
                                          int& below) {
    float cnt = 0.f, sl = 0.f;
    int nb = 0;
    for (int s = 0; s < S; ++s) {
        const uint32_t w = sw[s * kEqBlock];
        const float rq = t.rq[w & 31];
        const float m = count_float((w >> 13) & 255u);
        const float x = (Bf - t.cf[p2p_of(w)]) * rq;
        const bool sat = rq == 0.f || x >= m;
        cnt += sat ? m : x;
        sl += sat ? 0.f : rq;
        nb += sat ? 0 : 1;
    }
    slope = sl;
    below = nb;
    return cnt;
}

// The caps at a bound, as counted by a probe or a walk pass.
struct Caps {
    int64_t hi;   // largest stage time c + k q over stages holding a layer (-1: none)
    int64_t lo;   // next breakpoint: min c + (k + 1) q over stages below their run (kInf: none)
    int tot;      // layers the stages hold
    int nhi, nlo; // stages attaining hi / lo
    int empty;    // stages holding no layer
    bool stop;    // a stage attaining hi holds a single layer, or its layers are free
    bool jump;    // a stage holds none of its free layers (it gains them all at once)
    float slope;  // sum of 1/q over stages below their run (a probe's only)
    __device__ bool feasible(int L) const { return empty == 0 && tot >= L; }
};

// Exact probe of bound B for the stages in column sw; stores each stage's
// cap in its word.
__device__ __forceinline__ void eq_probe(const EqTabs& t, uint32_t* sw, int S, int64_t B, Caps& p) {
    int64_t rmin = kInf, gmin = kInf;  // B - hi, lo - B
    p.tot = p.nhi = p.nlo = p.empty = 0;
    p.stop = p.jump = false;
    p.slope = 0.f;
    for (int s = 0; s < S; ++s) {
        const uint32_t w = sw[s * kEqBlock];
        const int64_t q = t.q[w & 31];
        const int64_t x = B - t.p2p[p2p_of(w)];
        const float rq = t.rq[w & 31];
        const int m = run_of(w);
        const int64_t mq = (int64_t)m * q;
        // k layers take x - r; unsaturated the float estimate is off by at
        // most one (x < m q with m <= 255)
        const bool sat = x >= mq, none = x < q;
        int k = sat ? m : none ? 0 : (int)(u64_to_float((uint64_t)x) * rq);
        int64_t r = x - (int64_t)k * q;
        if (!sat && !none) {
            if (r < 0) {
                --k;
                r += q;
            } else if (r >= q) {
                ++k;
                r -= q;
            }
        }
        sw[s * kEqBlock] = (w & kNoCap) | ((uint32_t)k << kCapShift);
        p.tot += k;
        if (k < m) {
            p.slope += rq;
            const int64_t g = q - r;
            p.nlo = g < gmin ? 1 : p.nlo + (g == gmin ? 1 : 0);
            gmin = min(gmin, g);
        }
        if (k > 0) {
            const bool stop = k == 1 || q == 0;
            p.stop = r < rmin ? stop : p.stop || (r == rmin && stop);
            p.nhi = r < rmin ? 1 : p.nhi + (r == rmin ? 1 : 0);
            rmin = min(rmin, r);
        } else {
            ++p.empty;
            p.jump |= q == 0;
        }
    }
    p.hi = rmin == kInf ? -1 : B - rmin;
    p.lo = gmin == kInf ? kInf : B + gmin;
}

// The caps just below p.hi: the stages at hi lose their top layer.
__device__ __forceinline__ void eq_walk_down(const EqTabs& t, uint32_t* sw, int S, Caps& p) {
    const int64_t from = p.hi;
    int64_t hi = -1;
    int nhi = 0;
    bool stop = false;
    for (int s = 0; s < S; ++s) {
        const uint32_t w = sw[s * kEqBlock];
        const int64_t q = t.q[w & 31];
        int k = cap_of(w);
        int64_t v = t.p2p[p2p_of(w)] + (int64_t)k * q;
        if (v == from) {
            --k;
            v -= q;
            sw[s * kEqBlock] = (w & kNoCap) | ((uint32_t)k << kCapShift);
        }
        const bool st = k == 1 || q == 0;
        stop = v > hi ? st : stop || (v == hi && st);
        nhi = v > hi ? 1 : nhi + (v == hi ? 1 : 0);
        hi = max(hi, v);
    }
    p.tot -= p.nhi;
    p.hi = hi;
    p.nhi = nhi;
    p.stop = stop;
}

// The caps at p.lo: the stages whose next breakpoint it is gain a layer.
__device__ __forceinline__ void eq_walk_up(const EqTabs& t, uint32_t* sw, int S, Caps& p) {
    const int64_t at = p.lo;
    int64_t lo = kInf;
    int nlo = 0, empty = 0;
    for (int s = 0; s < S; ++s) {
        const uint32_t w = sw[s * kEqBlock];
        const int64_t q = t.q[w & 31];
        const int m = run_of(w);
        int k = cap_of(w);
        int64_t v = t.p2p[p2p_of(w)] + (int64_t)(k + 1) * q;
        if (k < m && v == at) {
            ++k;
            v += q;
            sw[s * kEqBlock] = (w & kNoCap) | ((uint32_t)k << kCapShift);
        }
        if (k < m) {
            nlo = v < lo ? 1 : nlo + (v == lo ? 1 : 0);
            lo = min(lo, v);
        }
        empty += k == 0 ? 1 : 0;
    }
    p.tot += p.nlo;
    p.hi = at;
    p.lo = lo;
    p.nlo = nlo;
    p.empty = empty;
}

// Exact lower and feasible upper bound of B*: every stage at one layer, at
// its memory run (which the screen guarantees covers L).
__device__ __noinline__ void eq_span(const EqTabs& t, const uint32_t* sw, int S, int64_t& lo, int64_t& hi) {
    lo = hi = 0;
    for (int s = 0; s < S; ++s) {
        const uint32_t w = sw[s * kEqBlock];
        const int64_t q = t.q[w & 31], c = t.p2p[p2p_of(w)];
        lo = max(lo, c + q);
        hi = max(hi, c + (int64_t)run_of(w) * q);
    }
}

// B* from the first guess B: returns it, leaves the caps at B* in the stage
// words and their sum in total.  (walk: kWalk, or 0 to probe only)
__device__ __forceinline__ int64_t eq_threshold(const EqTabs& t, uint32_t* sw, int S, int L, int64_t B, int walk,
                                                int& total, unsigned long long& probes, uint32_t* err) {
    int64_t lo = 0, hi = -1;        // B* in [lo, hi] (hi < 0: not computed yet)
    int64_t Blo = -1, Bhi = -1;     // last infeasible / feasible bound probed
    int clo = 0, chi = 0;           // layer counts of those probes
    Caps p;
    for (int it = 0;; ++it) {
        ++probes;
        eq_probe(t, sw, S, B, p);
        const bool feas = p.feasible(L);
        const int tot = p.tot;
        if (feas) {
            int64_t top = p.hi;
            for (int w = 0;; ++w) {
                // just below hi every stage attaining hi loses a layer
                top = p.hi;
                if (p.tot - p.nhi < L || p.stop) {
                    total = p.tot;
                    return p.hi;
                }
                if (w >= walk || p.tot - L > 2 * walk) break;
                eq_walk_down(t, sw, S, p);
            }
            if (hi < 0) eq_span(t, sw, S, lo, hi);
            hi = min(hi, top);
            Bhi = B;
            chi = tot;
        } else {
            const int64_t next = p.lo;
            if (!p.jump && L - tot <= 2 * walk) {
                for (int w = 0; w < walk && p.lo < kInf; ++w) {
                    eq_walk_up(t, sw, S, p);
                    if (p.feasible(L)) {
                        total = p.tot;
                        return p.hi;
                    }
                }
            }
            if (hi < 0) eq_span(t, sw, S, lo, hi);
            // after a walk every bound below its last breakpoint is known to fail
            lo = min(max(lo, max(next, p.hi + 1)), hi);
            Blo = B;
            clo = tot;
        }
        if (it > kMaxIters) {
            atomicOr(err, kErrSearchBound);
            total = p.tot;
            return hi;
        }
        // next bound: interpolate the cap count between the bracket's
        // probes, else a Newton step, else bisect; a closed bracket is
        // probed at hi for its caps
        if (lo >= hi) {
            B = hi;
            continue;
        }
        float target = -1.f;
        if (Blo >= 0 && Bhi >= 0 && chi > clo) {
            target = u64_to_float(Blo) +
                     ((float)L - 0.5f - (float)clo) / (float)(chi - clo) * u64_to_float(Bhi - Blo);
        } else if (p.slope > 0.f) {
            const float Bf = u64_to_float(B);
            target = feas ? Bf - ceilf(((float)tot - (float)L + 0.5f) / p.slope)
                          : Bf + ceilf(((float)L - (float)tot) / p.slope);
        }
        B = (target >= u64_to_float(lo) && target <= u64_to_float(hi - 1)) ? (int64_t)float_to_u64(target)
                                                                             : lo + (hi - lo) / 2;
        B = min(max(B, lo), hi - 1);
    }
}

// The smallest boundaries from the caps at B*, then Evaluate:
// T = (M-1) max t_s + sum t_s + max g_s; writes entry p and returns T.
__device__ __forceinline__ int64_t eq_evaluate(const PriceArgs& a, const EqTabs& t, const int64_t* PB, int64_t pbytes,
                                               const uint32_t* sw, int64_t p, int S, int M, int64_t n, int L,
                                               int64_t Bstar, int total) {
    const int64_t c = a.wl_idx[p];
    if (!in_range(c, a.n, a.err)) return -1;
    int64_t tsum = 0, tmax = 0;
    GradMax grad;
    int pre = 0, at = 0;
    for (int s = 0; s < S; ++s) {
        const uint32_t w = sw[s * kEqBlock];
        const int k = cap_of(w);
        pre += k;
        const int nxt = s + 1 == S ? L : max(at + 1, L - (total - pre));
        if (a.bounds) a.bounds[(int64_t)(s + 1) * a.bstride + c] = (uint8_t)nxt;
        const int len = nxt - at;
        if (len > k) atomicOr(a.err, kErrInternal);
        const int64_t ts = (int64_t)len * t.q[w & 31] + t.p2p[p2p_of(w)];
        tmax = max(tmax, ts);
        tsum += ts;
        if (n > 1) grad.add(t, PB, pbytes, w & 31, at, nxt);
        at = nxt;
    }
    if (a.bounds) {
        a.bounds[c] = 0;
        if (!a.bounds_scratch)
            for (int s = S + 1; s <= kMaxStages; ++s) a.bounds[(int64_t)s * a.bstride + c] = 0;
    }
    // (a bound above B* would pass the test of the lengths)
    if (pre != total || tmax != Bstar) atomicOr(a.err, kErrInternal);
    const int64_t gmax = n > 1 ? grad.sync_ns(n, pbytes, a.err) : 0;
    const int64_t T = (int64_t)(M - 1) * Bstar + tsum + gmax;
    a.T[c] = T;
    a.wl_T[p] = T;
    a.wl_nM[p] = (uint32_t)n * (uint32_t)M;
    a.B[c] = Bstar;
    a.ndp[c] = (uint16_t)n;
    a.status[c] = HEDDLE_CAND_OK;
    return T;
}

template <bool kCount>
__global__ void __launch_bounds__(kEqBlock, 1024 / kEqBlock) eq_search_kernel(PriceArgs a) {
    __shared__ __align__(16) EqShared sh;
    __shared__ int end_of[kMaxStages + 2];  // entries of depths >= S, [S]
    const Layout& y = a.lay;
    const int L = y.L;
    load_eq_tables(a, sh.tab, sh.run);
    allow_dependents();
    await_previous();  // the screen's worklist
    depth_ends(a.wl_count, end_of);
    __syncthreads();
    const EqTabs& t = sh.tab;
    const int64_t* PB = reinterpret_cast<const int64_t*>(a.img + y.offPB);
    const int64_t pbytes = reinterpret_cast<const ModelInfo*>(a.img + y.offModel)->grad_uniform ? PB[1] - PB[0] : -1;
    uint32_t* mysw = sh.sw + threadIdx.x;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    unsigned long long units = 0, probes = 0, searched = 0;
    // the entries filed in the depth buckets (every worklist entry here)
    const int64_t entries = min((int64_t)*a.wl_count, (int64_t)a.wl_cap);
    const int64_t count = min((int64_t)end_of[1], entries);
    // warp w of CTA b takes entries [32 (4 b + w), +32) of the order by
    // decreasing S, so its lanes have nearly equal S, then the next 32
    // untaken ones whenever it is free; warps never wait on one another
    const int64_t first = (int64_t)gridDim.x * kEqBlock;
    auto take = [&]() {
        int b = 0;
        if (lane == 0) b = atomicAdd(a.wl_count + kWlTakeThread, 32);
        return first + __shfl_sync(0xffffffffu, b, 0);
    };
    for (int64_t base = ((int64_t)blockIdx.x * kEqWarps + warp) * 32; base < count; base = take()) {
        const int64_t g = base + lane;
        bool have = g < count;
        int64_t p = 0;
        int S = 0, M = 0;
        int64_t n = 0;
        int64_t T = -1;
        if (have) have = deepest_first(a, end_of, g, entries, p);
        if (have) {
            S = a.wl_S[p];
            M = a.wl_M[p];
            n = a.wl_n[p];
            if (kCount) {
                ++searched;
                units += S;
            }
            // pack the stages; the unsaturated continuous balance, and the
            // least bound at which every stage holds a layer
            float inv = 0.f, cw = 0.f, flo = 0.f;
            for_stages(a, t, sh.run, p, S, M, [&](int s, int code, int pidx, uint32_t m) {
                mysw[s * kEqBlock] = (uint32_t)code | ((uint32_t)pidx << 5) | (m << 13);
                const float rq = t.rq[code], cf = t.cf[pidx];
                inv += rq;
                cw += cf * rq;
                flo = fmaxf(flo, cf + t.qf[code]);
            });
            // first guess: Newton on the saturating continuous count
            float Bf = fmaxf(flo, inv > 0.f ? ((float)L + 0.5f * (float)S + cw) / inv : flo);
            for (int it = 0; it < 3; ++it) {  // the exact probes finish the job
                float sl;
                int below;
                const float cnt = eq_count(t, mysw, S, Bf, sl, below);
                const float tgt = (float)L + 0.5f * (float)below;
                if (cnt >= tgt - 0.25f || sl <= 0.f) break;
                Bf += (tgt - cnt) / sl;
            }
            int total = 0;
            // (the checked build probes only for every second entry, so that
            // both the walk and the bracketing run)
            const int walk = kChecked && (p & 1) ? 0 : kWalk;
            const int64_t Bstar =
                eq_threshold(t, mysw, S, L, (int64_t)float_to_u64(Bf), walk, total, probes, a.err);
            T = eq_evaluate(a, t, PB, pbytes, mysw, p, S, M, n, L, Bstar, total);
        }
        if (a.sv_count) {
            // inside a top-k pricing: the entries whose n*M / T reaches the
            // running threshold (float, below the k-th key by a margin that
            // covers the rounding) go to the top-k's survivor list.  The
            // warp first raises the threshold to its own k-th best key (for
            // k <= 32): any k entries' smallest key is at most the call's
            // final k-th, so the raised value keeps the filter exact
            const uint32_t nM = (uint32_t)n * (uint32_t)M;
            // (T = 0, where every layer rounds to 0 ns: the key is infinite,
            // and so is a threshold that k such entries raised)
            const float key = have && T >= 0 ? (float)nM / (float)T : -1.0f;
            const int kk = min(max(*a.topk_k, 1), kMaxTopK);
            float own = 0.f;
            const float thr0 = __uint_as_float(__ldcg(a.thr));
            // (only if k of its entries lie above it)
            if (kk <= 32 && __popc(__ballot_sync(0xffffffffu, key > thr0)) >= kk) {
                float v = key;  // bitonic sort of the warp's keys, descending
#pragma unroll
                for (int size = 2; size <= 32; size <<= 1)
#pragma unroll
                    for (int stride2 = size >> 1; stride2 > 0; stride2 >>= 1) {
                        const float o = __shfl_xor_sync(0xffffffffu, v, stride2);
                        const bool desc = (lane & size) == 0 || size == 32;
                        v = (((lane & stride2) == 0) == desc) ? fmaxf(v, o) : fminf(v, o);
                    }
                const float kth = __shfl_sync(0xffffffffu, v, kk - 1);
                if (kth > 0.f) {
                    own = kth * (1.0f - 1.0f / 65536.0f);
                    if (lane == 0) atomicMax(a.thr, __float_as_uint(own));
                }
            }
            const float thr = fmaxf(thr0, own);
            const bool keep = key > 0.f && key >= thr;
            const unsigned mask = __ballot_sync(0xffffffffu, keep);
            if (mask) {
                int base0 = 0;
                if (lane == __ffs(mask) - 1) base0 = atomicAdd(a.sv_count, __popc(mask));
                const int pos = __shfl_sync(0xffffffffu, base0, __ffs(mask) - 1) + __popc(mask & ((1u << lane) - 1));
                if (keep && pos < a.wl_cap) {
                    a.sv_idx[pos] = a.wl_idx[p];
                    a.sv_T[pos] = T;
                    a.sv_nM[pos] = nM;
                }
            }
        }
    }
    if (kCount) {
        unsigned long long v0 = units, v1 = probes, v2 = searched;
        for (int o = 16; o > 0; o >>= 1) {
            v0 += __shfl_down_sync(0xffffffffu, v0, o);
            v1 += __shfl_down_sync(0xffffffffu, v1, o);
            v2 += __shfl_down_sync(0xffffffffu, v2, o);
        }
        if (lane == 0) {
            atomicAdd(&a.counters[0], v0);
            atomicAdd(&a.counters[1], v1);
            atomicAdd(&a.counters[2], v2);
        }
    }
}

template <bool kCount>
cudaError_t launch(const PriceArgs& a, int num_sms, cudaStream_t st) {
    int per_sm = 0;
    const cudaError_t e = resident_blocks(reinterpret_cast<const void*>(&eq_search_kernel<kCount>), kEqBlock, 0, &per_sm);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    // the worklist length is only known on the device: size for the batch,
    // at most seven of the eight CTAs that fit an SM -- warps fetch further
    // entries when free, and the free slot lets the next chunk's screen
    // start beside this search's last warps
    const int64_t need = (a.n + kEqBlock - 1) / kEqBlock;
    const int grid = (int)std::min<int64_t>(need, (int64_t)num_sms * std::min(per_sm, 7));
    return launch_after(a.chained, eq_search_kernel<kCount>, grid, kEqBlock, 0, st, a);
}

}  // namespace

cudaError_t launch_eq_search(const PriceArgs& a, int num_sms, cudaStream_t st) {
    return a.counters ? launch<true>(a, num_sms, st) : launch<false>(a, num_sms, st);
}

}  // namespace hd
