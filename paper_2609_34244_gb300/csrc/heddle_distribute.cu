// heddle_distribute.cu -- the paper's own layer split as a second split mode
// (§5.3 "Layer split and DP degree"): each stage gets layers in proportion
// to its profiled speed; if that split exceeds a stage's memory, a fixed
// list of alternative splits is priced and the fastest one that fits is
// kept.  The hot path's min-max PartitionLayers replaces this rule; this
// mode prices the same candidates the paper's way so the two can be
// compared (the quality gap of the heuristic).
//
// Readings (shared with the oracle only through their statement): the speed
// of stage s is 2^40 divided by the time of all L layers on its type and
// degree, rounded down; the list is (1) in proportion to speed, (2) equal
// layer counts, (3) in proportion to the longest run of consecutive layers
// each stage's memory holds; shares are floors of L w_s / sum w with at
// least one layer per stage, missing layers to the largest remainders (the
// earlier stage on ties), surplus layers off the stage holding the most
// (the later stage on ties); the fastest is the smallest pipeline time
// (M-1) max t_s + sum t_s, the earlier alternative on ties (Algorithm 1
// splits the layers before the fill picks the DP degree, so the choice
// cannot see the gradient term).  No alternative fits: OOM.
//
// Two kernels.  On a model whose layers all cost the same in time and memory
// a stage's time is layers times one layer's and its memory is a run length,
// so an alternative is a sum and a maximum over the stages: one thread per
// entry, the warps taking 32 at a time, deepest first, like the equal-layer
// search.  The floors come from float quotients corrected exactly; the
// largest remainders from 32-bit keys (27 leading bits of the remainder and
// the stage), compared with one another, and from the exact remainders where
// two that differ share a key at the cut.  1e6 candidates of the largest
// workload: 260 -> 62 us (one warp per entry, a lane per stage: 64-bit
// divisions, sums and ranks by shuffles, half the lanes past the depth).
// Other models keep that warp kernel, whose lanes read the prefix tables, and so
// do few entries, for which a thread's serial chain is the longer: both are
// launched, and by the entries per depth one of them returns at once (100
// entries of 70,000 candidates: 74 us a pass by threads, 33 so).

#include <algorithm>

#include "heddle_eq.cuh"

namespace hd {
namespace {

constexpr int kDistBlock = 128;
constexpr unsigned kFull = 0xffffffffu;

__device__ __forceinline__ int64_t warp_sum64(int64_t v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    return v;
}

__device__ __forceinline__ int64_t warp_max64(int64_t v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = max(v, (int64_t)__shfl_xor_sync(kFull, v, o));
    return v;
}

// This lane's layer count when L layers go to the S live lanes in
// proportion to w (sum V > 0): floor of the exact share, at least one;
// missing layers one each to the largest remainders (the earlier stage on
// ties); surplus layers one at a time off the stage holding the most (the
// later stage on ties).
__device__ int share_count(bool live, int S, int L, int64_t w, int64_t V, int lane) {
    int64_t q = 0, rem = 0;
    if (live) {
        const int64_t share = (int64_t)L * w;
        q = share / V;
        rem = share - q * V;
    }
    int cnt = live ? (q < 1 ? 1 : (int)q) : 0;
    int total = __reduce_add_sync(kFull, (unsigned)cnt);
    if (total < L) {
        // the L - total largest remainders gain one layer
        int rank = 0;
        for (int t = 0; t < S; ++t) {
            const int64_t rt = __shfl_sync(kFull, rem, t);
            rank += (rt > rem || (rt == rem && t < lane)) ? 1 : 0;
        }
        if (live && rank < L - total) ++cnt;
    }
    while (total > L) {
        // the stage holding the most (the later one on ties) gives one up
        const int key = live && cnt > 1 ? (cnt << 8) | lane : -1;
        const int top = __reduce_max_sync(kFull, (unsigned)(key + 1)) - 1;
        if (lane == (top & 0xff)) --cnt;
        --total;
    }
    return cnt;
}

// Whether the entries are priced by a thread each (split_kernel) or a warp each
// (distribute_kernel); every lane of a warp calls it.
__device__ __forceinline__ bool split_by_threads(const PriceArgs& a) {
    const int here = a.wl_count[1 + 1 + (threadIdx.x & 31)];  // entries of depth 1 + lane
    const int deepest = 32 - __clz(__ballot_sync(kFull, here > 0));
    return __reduce_add_sync(kFull, (unsigned)here) >= (unsigned)(a.split_min + a.split_per_stage * deepest);
}

// (both_launched: split_kernel follows, for the entries it takes)
__global__ void __launch_bounds__(kDistBlock) distribute_kernel(PriceArgs a, int both_launched) {
    const Layout& y = a.lay;
    allow_dependents();
    await_previous();
    if (both_launched && split_by_threads(a)) return;
    const int L = y.L;
    const int64_t* P = reinterpret_cast<const int64_t*>(a.img + y.offP);
    const longlong2* SA = reinterpret_cast<const longlong2*>(a.img + y.offSA);
    const int64_t* PB = reinterpret_cast<const int64_t*>(a.img + y.offPB);
    const int64_t* p2p = reinterpret_cast<const int64_t*>(a.img + y.offP2P);
    const int64_t* mem = reinterpret_cast<const int64_t*>(a.img + y.offMem);
    const int64_t* inter = reinterpret_cast<const int64_t*>(a.img + y.offInter);
    const int32_t* maxn = reinterpret_cast<const int32_t*>(a.img + y.offMaxN);
    const uint8_t* win = a.img + y.offWin;
    const int lane = threadIdx.x & 31;
    const int64_t count = min((int64_t)*a.wl_count, (int64_t)a.wl_cap);
    // each warp prices its own first entry, then the next untaken one
    // whenever it is free
    const int64_t first = (int64_t)gridDim.x * (blockDim.x >> 5);
    auto take = [&]() {
        int e = 0;
        if (lane == 0) e = atomicAdd(a.wl_count + kWlTakeWarp, 1);
        return first + __shfl_sync(kFull, e, 0);
    };
    for (int64_t p = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); p < count; p = take()) {
        const int64_t c = a.wl_idx[p];
        const int S = a.wl_S[p];
        if (!in_range(c, a.n, a.err) || !in_range(S - 1, kMaxStages, a.err)) continue;
        const int M = a.wl_M[p];
        const int64_t n = a.wl_n[p];
        const bool live = lane < S;
        // this lane's stage: cost row, P2P, memory capacity, in-flight count,
        // NIC x degree, and its weight under each alternative
        const int code = a.wl_code[p * kMaxStages + lane];
        const int nxt = __shfl_down_sync(kFull, code, 1);
        const int g = code & 7, j = (code >> 3) & 3;
        const int row = (g * 4 + j) * (L + 1);
        const int64_t capk = mem[g] << j;
        const int f = min(S - lane, M);
        const uint64_t D = (uint64_t)inter[g] << j;
        int64_t cs = 0;
        if (lane + 1 < S) {
            const int h = nxt & 7, jn = (nxt >> 3) & 3;
            const int same = (g == h) && ((1 << j) + (1 << jn) <= maxn[g]);
            cs = p2p[(g * 8 + h) * 2 + same];
        }
        int64_t w[3] = {0, 0, 0};
        if (live) {
            const int64_t all = P[row + L] - P[row];
            w[0] = all > 0 ? ((int64_t)1 << 40) / all : ((int64_t)1 << 40);
            w[1] = 1;
            w[2] = win[(g * 4 + j) * 33 + f];
        }
        bool found = false;
        int64_t bestPipe = 0, bestB = 0;
        int bestLo = 0, bestHi = 0;  // this lane's stage [bestLo, bestHi) in the chosen split
#pragma unroll
        for (int alt = 0; alt < 3; ++alt) {
            const int64_t V = warp_sum64(w[alt]);
            if (V <= 0) continue;
            const int cnt = share_count(live, S, L, w[alt], V, lane);
            // boundaries: inclusive scan of the counts
            int hi = cnt;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int t = __shfl_up_sync(kFull, hi, o);
                if (lane >= o) hi += t;
            }
            const int lo = hi - cnt;
            bool fits = true;
            int64_t t = 0;
            if (live) {
                const longlong2 a0 = SA[lo], a1 = SA[hi];
                fits = (a1.x - a0.x) + (int64_t)f * (a1.y - a0.y) <= capk;
                t = P[row + hi] - P[row + lo] + cs;
            }
            if (!__all_sync(kFull, fits)) continue;
            // the pipeline time of this split decides between alternatives
            const int64_t tmax = warp_max64(t), tsum = warp_sum64(t);
            const int64_t pipe = (int64_t)(M - 1) * tmax + tsum;
            if (!found || pipe < bestPipe) {
                found = true;
                bestPipe = pipe;
                bestB = tmax;
                bestLo = lo;
                bestHi = hi;
            }
        }
        int64_t T = bestPipe;
        if (found && n > 1) {
            // Evaluate adds the gradient term: the stage with the largest
            // G_s / (k_s bw_s), compared exactly, then ceil(2(n-1) G 1e9 / (n k bw))
            uint64_t G = live ? (uint64_t)(PB[bestHi] - PB[bestLo]) : 0;
            uint64_t Dd = live ? D : 1;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const uint64_t G2 = __shfl_xor_sync(kFull, G, o), D2 = __shfl_xor_sync(kFull, Dd, o);
                if ((u128)G2 * Dd > (u128)G * D2) {
                    G = G2;
                    Dd = D2;
                }
            }
            const u128 num = (u128)(2 * (uint64_t)(n - 1) * 1000000000ull) * G;
            bool ok = true;
            T += (int64_t)ceil_div_u128(num, (uint64_t)n * Dd, &ok);
            if (!ok && lane == 0) atomicOr(a.err, kErrInternal);
        }
        if (lane == 0) {
            if (found) {
                a.T[c] = T;
                a.B[c] = bestB;
                a.status[c] = HEDDLE_CAND_OK;
                a.wl_T[p] = T;
            } else {
                a.T[c] = -1;
                a.B[c] = -1;
                a.status[c] = HEDDLE_CAND_OOM;
                a.wl_T[p] = -1;
            }
            a.ndp[c] = (uint16_t)n;  // OOM keeps the DP degree
            a.wl_nM[p] = (uint32_t)n * (uint32_t)M;
        }
        if (a.bounds) {
            // plane s + 1 from lane s; plane 0 from lane 31 (always 0)
            const int plane = lane == 31 ? 0 : lane + 1;
            a.bounds[(int64_t)plane * a.bstride + c] = (lane != 31 && found && live) ? (uint8_t)bestHi : 0;
            if (lane == 0) a.bounds[(int64_t)kMaxStages * a.bstride + c] = (found && S == kMaxStages) ? (uint8_t)L : 0;
        }
    }
}

// ---- equal layers: one thread per entry

struct SplitShared {
    EqTabs tab;
    uint16_t run[32 * 33 + 256];         // ScreenTabs::run
    int64_t speed[32];                   // 2^40 / the time of all layers, per stage byte
    uint32_t sw[kMaxStages * kEqBlock];  // stage words (heddle_eq.cuh): the cap field holds the stage's layers
    uint32_t key[kMaxStages * kEqBlock];
};

// floor(share / V) and the remainder, the float quotient off by at most one
// (the quotient is at most 255)
__device__ __forceinline__ int share_floor(int64_t share, int64_t V, float rV, int64_t& rem) {
    int q = (int)(u64_to_float((uint64_t)share) * rV);
    rem = share - (int64_t)q * V;
    if (rem < 0) {
        --q;
        rem += V;
    } else if (rem >= V) {
        ++q;
        rem -= V;
    }
    return q;
}

// The weight of a stage under an alternative (0: speed, 2: memory run).
__device__ __forceinline__ int64_t split_weight(const SplitShared& sh, uint32_t w, int alt) {
    return alt == 0 ? sh.speed[w & 31] : (int64_t)run_of(w);
}

// The stages that gain a layer by exact remainders (only where keys cannot
// tell): counts of stages with a larger remainder, or as large and earlier.
__device__ __noinline__ void exact_gains(const SplitShared& sh, uint32_t* sw, int S, int L, int64_t V, float rV, int alt,
                                         int missing) {
    for (int s = 0; s < S; ++s) {
        int64_t rs, rt;
        share_floor((int64_t)L * split_weight(sh, sw[s * kEqBlock], alt), V, rV, rs);
        int rank = 0;
        for (int t = 0; t < S; ++t) {
            share_floor((int64_t)L * split_weight(sh, sw[t * kEqBlock], alt), V, rV, rt);
            rank += (rt > rs || (rt == rs && t < s)) ? 1 : 0;
        }
        if (rank < missing) sw[s * kEqBlock] += 1u << kCapShift;
    }
}

// Layers per stage in proportion to the alternative's weights (sum V > 0),
// into the cap fields (see share_count).
__device__ __forceinline__ void proportional(const SplitShared& sh, uint32_t* sw, uint32_t* key, int S, int L, int64_t V,
                                             int alt) {
    const float rV = 1.0f / u64_to_float((uint64_t)V);
    const int shift = max(0, 64 - __clzll(V) - 27);
    int total = 0;
    for (int s = 0; s < S; ++s) {
        const uint32_t w = sw[s * kEqBlock] & kNoCap;
        int64_t rem;
        const int q = max(share_floor((int64_t)L * split_weight(sh, w, alt), V, rV, rem), 1);
        sw[s * kEqBlock] = w | ((uint32_t)q << kCapShift);
        key[s * kEqBlock] = ((uint32_t)(rem >> shift) << 5) | (uint32_t)(31 - s);
        total += q;
    }
    const int missing = L - total;
    if (missing > 0) {
        // ranks of four stages at a time; the last key that gains, the first
        // that does not
        uint32_t cut = 0xffffffffu, next = 0;
        for (int s0 = 0; s0 < S; s0 += 4) {
            uint32_t k[4];
            int r[4] = {0, 0, 0, 0};
#pragma unroll
            for (int i = 0; i < 4; ++i) k[i] = s0 + i < S ? key[(s0 + i) * kEqBlock] : 0xffffffffu;
            for (int t = 0; t < S; ++t) {
                const uint32_t kt = key[t * kEqBlock];
#pragma unroll
                for (int i = 0; i < 4; ++i) r[i] += kt > k[i] ? 1 : 0;
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                if (s0 + i >= S) continue;
                if (r[i] < missing) {
                    sw[(s0 + i) * kEqBlock] += 1u << kCapShift;
                    cut = min(cut, k[i]);
                } else {
                    next = max(next, k[i]);
                }
            }
        }
        if (shift > 0 && missing < S && (cut >> 5) == (next >> 5)) {
            // a tie at the cut: exact if one weight (the same remainder) has it all
            bool same = true;
            const uint32_t code = sw[(31 - (cut & 31)) * kEqBlock] & 31;
            for (int s = 0; s < S; ++s)
                same = same && ((key[s * kEqBlock] >> 5) != (cut >> 5) || (sw[s * kEqBlock] & 31) == code);
            if (!same) {
                for (int s = 0; s < S; ++s) {
                    int64_t rem;
                    const uint32_t w = sw[s * kEqBlock] & kNoCap;
                    const int q = max(share_floor((int64_t)L * split_weight(sh, w, alt), V, rV, rem), 1);
                    sw[s * kEqBlock] = w | ((uint32_t)q << kCapShift);
                }
                exact_gains(sh, sw, S, L, V, rV, alt, missing);
            }
        }
    }
    for (; total > L; --total) {
        // the stage holding the most (the later one on ties) gives one up
        int most = 0, at = 0;
        for (int s = 0; s < S; ++s) {
            const int c = cap_of(sw[s * kEqBlock]);
            if (c >= most) {
                most = c;
                at = s;
            }
        }
        if (most <= 1) break;  // (S <= L: never)
        sw[at * kEqBlock] -= 1u << kCapShift;
    }
}

__global__ void __launch_bounds__(kEqBlock, 5) split_kernel(PriceArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    SplitShared& sh = *reinterpret_cast<SplitShared*>(smem);
    __shared__ int end_of[kMaxStages + 2];
    const Layout& y = a.lay;
    const int L = y.L;
    load_eq_tables(a, sh.tab, sh.run);
    allow_dependents();
    await_previous();  // the screen's worklist
    if (!split_by_threads(a)) return;  // distribute_kernel has priced it
    depth_ends(a.wl_count, end_of);
    __syncthreads();
    if (threadIdx.x < 32) {
        const int64_t all = sh.tab.q[threadIdx.x] * L;
        sh.speed[threadIdx.x] = all > 0 ? ((int64_t)1 << 40) / all : ((int64_t)1 << 40);
    }
    __syncthreads();
    const EqTabs& t = sh.tab;
    const int64_t* PB = reinterpret_cast<const int64_t*>(a.img + y.offPB);
    const int64_t pbytes = reinterpret_cast<const ModelInfo*>(a.img + y.offModel)->grad_uniform ? PB[1] - PB[0] : -1;
    uint32_t* sw = sh.sw + threadIdx.x;
    uint32_t* key = sh.key + threadIdx.x;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t entries = min((int64_t)*a.wl_count, (int64_t)a.wl_cap);
    const int64_t count = min((int64_t)end_of[1], entries);
    const int64_t first = (int64_t)gridDim.x * kEqBlock;
    auto take = [&]() {
        int b = 0;
        if (lane == 0) b = atomicAdd(a.wl_count + kWlTakeThread, 32);
        return first + __shfl_sync(kFull, b, 0);
    };
    for (int64_t base = ((int64_t)blockIdx.x * kEqWarps + warp) * 32; base < count; base = take()) {
        const int64_t g = base + lane;
        int64_t p = 0;
        if (g >= count || !deepest_first(a, end_of, g, entries, p)) continue;
        const int64_t c = a.wl_idx[p];
        const int S = a.wl_S[p], M = a.wl_M[p];
        const int64_t n = a.wl_n[p];
        if (!in_range(c, a.n, a.err)) continue;
        int64_t V0 = 0, csum = 0;
        int V2 = 0;
        for_stages(a, t, sh.run, p, S, M, [&](int s, int code, int pidx, uint32_t m) {
            sw[s * kEqBlock] = (uint32_t)code | ((uint32_t)pidx << 5) | (m << 13);
            V0 += sh.speed[code];
            V2 += (int)m;
            csum += t.p2p[pidx];
        });
        // the alternatives from the last to the first: an earlier one wins a
        // tie, and the first, which fits most often, is left in the words
        int best = -1;
        int64_t bestPipe = 0, bestB = 0;
        for (int alt = 2; alt >= 0; --alt) {
            const int64_t V = alt == 0 ? V0 : V2;
            if (alt != 1) {
                if (V <= 0) continue;
                proportional(sh, sw, key, S, L, V, alt);
            } else {
                // equal counts, the earlier stages one more
                const int each = L / S, more = L - each * S;
                for (int s = 0; s < S; ++s)
                    sw[s * kEqBlock] = (sw[s * kEqBlock] & kNoCap) | ((uint32_t)(each + (s < more ? 1 : 0)) << kCapShift);
            }
            bool fits = true;
            int64_t tmax = 0, tsum = csum;
            for (int s = 0; s < S; ++s) {
                const uint32_t w = sw[s * kEqBlock];
                const int k = cap_of(w);
                fits = fits && k <= run_of(w);
                const int64_t ts = (int64_t)k * t.q[w & 31];
                tsum += ts;
                tmax = max(tmax, ts + t.p2p[p2p_of(w)]);
            }
            const int64_t pipe = (int64_t)(M - 1) * tmax + tsum;
            if (fits && (best < 0 || pipe <= bestPipe)) {
                best = alt;
                bestPipe = pipe;
                bestB = tmax;
            }
        }
        a.ndp[c] = (uint16_t)n;  // OOM keeps the DP degree
        a.wl_nM[p] = (uint32_t)n * (uint32_t)M;
        if (best < 0) {
            a.T[c] = -1;
            a.B[c] = -1;
            a.status[c] = HEDDLE_CAND_OOM;
            a.wl_T[p] = -1;
            if (a.bounds)
                for (int s = 0; s <= kMaxStages; ++s) a.bounds[(int64_t)s * a.bstride + c] = 0;
            continue;
        }
        if (best == 2) proportional(sh, sw, key, S, L, V2, 2);
        GradMax grad;
        int at = 0;
        for (int s = 0; s < S; ++s) {
            const uint32_t w = sw[s * kEqBlock];
            const int each = L / S;
            const int nxt = at + (best == 1 ? each + (s < L - each * S ? 1 : 0) : cap_of(w));
            if (n > 1) grad.add(t, PB, pbytes, w & 31, at, nxt);
            if (a.bounds) a.bounds[(int64_t)(s + 1) * a.bstride + c] = (uint8_t)nxt;
            at = nxt;
        }
        if (at != L) atomicOr(a.err, kErrInternal);
        if (a.bounds) {
            a.bounds[c] = 0;
            for (int s = S + 1; s <= kMaxStages; ++s) a.bounds[(int64_t)s * a.bstride + c] = 0;
        }
        const int64_t T = bestPipe + (n > 1 ? grad.sync_ns(n, pbytes, a.err) : 0);
        a.T[c] = T;
        a.B[c] = bestB;
        a.status[c] = HEDDLE_CAND_OK;
        a.wl_T[p] = T;
    }
}

}  // namespace

cudaError_t launch_distribute(const PriceArgs& a, int num_sms, cudaStream_t st) {
    // one warp per entry; the worklist length is only known on the device
    const int grid = (int)std::min<int64_t>((a.n + kDistBlock / 32 - 1) / (kDistBlock / 32), (int64_t)num_sms * 16);
    // (a batch too small for the thread kernel at any depth does without it)
    const bool threads = a.equal_layers && a.n >= (int64_t)a.split_min + a.split_per_stage;
    cudaError_t e = launch_after(a.chained, distribute_kernel, grid, kDistBlock, 0, st, a, threads ? 1 : 0);
    if (e != cudaSuccess || !threads) return e;
    const size_t smem = sizeof(SplitShared);
    int per_sm = 0;
    e = resident_blocks(reinterpret_cast<const void*>(&split_kernel), kEqBlock, smem, &per_sm);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    const int tgrid = (int)std::min<int64_t>((a.n + kEqBlock - 1) / kEqBlock, (int64_t)num_sms * per_sm);
    return launch_after(a.chained, split_kernel, tgrid, kEqBlock, smem, st, a);
}

}  // namespace hd
