// heddle_plans.cu -- multi-template plan pricing (Algorithm 1: a plan is a
// sequence of structural templates, each holding its own GPUs; the reward
// of a step is the throughput the new template adds).
//
// The library first prices the template slots as standalone candidates
// (screen + search, unchanged): PartitionLayers and the memory decision do
// not depend on the DP degree n, so the split, the bottleneck and OOM carry
// over.  Slot t is priced only for the plans whose templates 0 .. t-1 are
// each OK alone (a walk ends at its first template that is not OK, and a
// template is OK in the walk only if it is OK alone); for the others the
// screen writes SKIPPED.  The first template, on the whole free cluster,
// keeps its standalone price.  This kernel then walks each plan in
// order against the GPUs the earlier templates left: the template's n
// comes from the free GPUs per node -- n = min over (type, size class e) of
// floor(cap / demand), cap = sum over nodes of floor(free / 2^e) 2^e, exact
// for power-of-two groups placed largest first -- then T is re-evaluated
// with that n (only the gradient term depends on it), and the template's
// groups are placed largest first on a node of its type whose free GPUs
// equal the group size, else on the node with the fewest free GPUs above
// it (§5.1).  Decisions depend on nodes only through their free counts, so a
// walk keeps, per GPU type, a histogram of nodes by free GPUs.  The first
// template that is not OK ends the plan; the plan's throughput is the sum
// over placed templates of n M 1e9 / T, each term rounded in IEEE double, in
// template order.
//
// Where few plans of a CTA walk, one warp walks a plan: a lane per stage for
// the demand and Evaluate, a lane per (type, size class) for n, a lane per
// type for the placement.  Deep plans mostly end at their first template, so
// their walks are few and their latency is the kernel's time: one thread a walk took 173 us for 200,003 plans of up to
// four templates on the 1,024-GPU cluster, this takes 66 us (a cold launch).
// A CTA looks at no more plans at a time than spread the batch over all SMs
// (1,308 plans of up to twelve stages: 229 -> 128 us a call, 212 by threads).
// Where most plans of a large batch walk -- shallow templates -- a thread each
// does several times the walks per instruction, 128 at a time.  A warp's walks
// take about 4 us / 4 warps each, a thread's alone 20 us and 5 us a stage: from
// 20 queued plans of a CTA on, and 5 more per stage of the deepest of them, they
// are walked so (52,002 plans of up to five stages: 205 us a call by warps
// alone, 140 with both).  The depth is the plans' own, not the planes of the
// buffers they lie in: 200,003 plans of up to two stages in 32 planes took 540 us
// by the planes, 267 in two.

#include <algorithm>

#include "heddle_wprobe.cuh"

namespace hd {
namespace {

constexpr int kPlanBlock = 128;
constexpr int kPlanWarps = kPlanBlock / 32;
constexpr unsigned kFull = 0xffffffffu;
// queued plans of a CTA from which a thread walks each (see the head of this file)
constexpr int kAloneMin = 20, kAlonePerStage = 5;

// Dynamic shared memory: per thread (interleaved by thread, element e of thread t
// at [e * kPlanBlock + t]) the demand word per type and the node histogram, or,
// while warps walk, an area per warp in the same place.
constexpr size_t plan_smem(int NT, int vmax) {
    return (size_t)kPlanBlock * (2 * (size_t)NT * (vmax + 1) + 8 * kMaxTypes);
}
struct WarpWalk {
    uint16_t hist[kMaxTypes][kPlanMaxNode + 1];  // nodes of type g with v free GPUs
    uint32_t dem[4 * kMaxTypes];                 // GPUs of groups of size class e on type g, at [4 g + e]
};
static_assert(sizeof(WarpWalk) * kPlanWarps <= plan_smem(1, 1), "the warps' areas fit where the threads' lie");
struct PlanShared {
    alignas(4) uint16_t init[kMaxTypes][kPlanMaxNode + 1];  // the cluster's nodes per type and GPU count
    int32_t queue[2 * kPlanBlock];
    int queued;
    int deep[kPlanWarps];  // per warp: the deepest template of the queued plans it looked at
};
// Thread walks wait on shared and global memory, so the CTAs an SM holds decide
// them: on eight types in nodes of up to eight GPUs, seven (120,000 plans of up
// to two stages, most of which walk: 910 us a call with six, the warps' areas
// beside the threads', 585 with seven; 800,000: 2.86 and 2.59 ms).
static_assert(7 * (plan_smem(8, 8) + sizeof(PlanShared) + 1024) <= 227 * 1024, "seven CTAs an SM");

__global__ void __launch_bounds__(kPlanBlock, 8) plan_kernel(PlanArgs a) {
    const Layout& y = a.lay;
    const int L = y.L, NT = y.NT, V = a.vmax;
    const int64_t* P = reinterpret_cast<const int64_t*>(a.img + y.offP);
    const int64_t* PB = reinterpret_cast<const int64_t*>(a.img + y.offPB);
    const int64_t* p2p = reinterpret_cast<const int64_t*>(a.img + y.offP2P);
    const int64_t* inter = reinterpret_cast<const int64_t*>(a.img + y.offInter);
    const int32_t* maxn = reinterpret_cast<const int32_t*>(a.img + y.offMaxN);
    const int32_t* pow2 = reinterpret_cast<const int32_t*>(a.img + y.offPow2);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    extern __shared__ __align__(16) unsigned char psm[];
    __shared__ PlanShared sh;
    WarpWalk& ww = reinterpret_cast<WarpWalk*>(psm)[warp];
    auto& hist = ww.hist;
    uint32_t* dem = ww.dem;
    auto& init = sh.init;
    for (int i = threadIdx.x; i < kMaxTypes * (kPlanMaxNode + 1); i += blockDim.x) (&init[0][0])[i] = 0;
    __syncthreads();
    for (int b = threadIdx.x; b < a.n_nodes; b += blockDim.x) {
        // 16-bit counts: at most 65535 nodes (the library's GPU limit)
        unsigned int* w = reinterpret_cast<unsigned int*>(&init[0][0]) +
                          ((a.node_type[b] * (kPlanMaxNode + 1) + a.node_gpus[b]) >> 1);
        atomicAdd(w, ((a.node_type[b] * (kPlanMaxNode + 1) + a.node_gpus[b]) & 1) ? 0x10000u : 1u);
    }
    __syncthreads();
    // Most plans end at their first template, whose standalone price is
    // already what the walk would give it (the whole cluster is free, so
    // its degree, split and T are the standalone ones): a quick pass writes
    // such plans, and the others are queued in shared memory and walked a
    // warp each.
    int32_t* queue = sh.queue;
    int& queued = sh.queued;
    if (threadIdx.x == 0) queued = 0;
    __syncthreads();
    // ---- one thread a plan: the node histogram H(g, v) and the demand word
    // my_dem[g] (GPUs of groups per size class e in 16-bit field e)
    uint64_t* my_dem = reinterpret_cast<uint64_t*>(psm) + threadIdx.x;  // [g * kPlanBlock]
    uint16_t* my_hist = reinterpret_cast<uint16_t*>(psm + (size_t)8 * kMaxTypes * kPlanBlock) + threadIdx.x;
    auto H = [&](int g, int v) -> uint16_t& { return my_hist[(size_t)(g * (V + 1) + v) * kPlanBlock]; };
    auto walk_alone = [&](int64_t c) {
        for (int g = 0; g < NT; ++g)
            for (int v = 0; v <= V; ++v) H(g, v) = init[g][v];
        const int nt = min((int)a.n_tmpl[c], a.slots);
        bool ended = false;
        int placed = 0;
        double thr = 0.0;
        // (the slots past the plan's templates were priced SKIPPED)
        for (int t = 0; t < nt; ++t) {
            const PlanSlot& sl = a.slot[t];
            uint8_t st = HEDDLE_CAND_SKIPPED;
            int64_t T = -1, B = -1;
            int64_t n = 0;
            const int S = sl.S[c];
            const int M = sl.M[c];
            if (!ended) {
                const uint8_t st0 = sl.status[c];
                if (st0 == HEDDLE_CAND_INVALID) {
                    st = HEDDLE_CAND_INVALID;
                } else {
                    // demand per (type, size class) in GPUs of groups of that class
                    for (int g = 0; g < NT; ++g) my_dem[g * kPlanBlock] = 0;
                    uint32_t present = 0;
                    for (int s = 0; s < S; ++s) {
                        const int b = sl.code[(int64_t)s * sl.stride + c];
                        const int g = b & 7, j = (b >> 3) & 3;
                        const int unit = (1 << j) <= maxn[g] ? (1 << j) : pow2[g];
                        my_dem[g * kPlanBlock] += (uint64_t)(1u << j) << (16 * (31 - __clz(unit)));
                        present |= 1u << g;
                    }
                    // n = min over (type, class e) of floor(cap / demand),
                    // cap = sum over nodes of floor(free / 2^e) 2^e
                    int64_t best = -1;
                    for (uint32_t pm = present; pm; pm &= pm - 1) {
                        const int g = __ffs(pm) - 1;
                        int64_t cap[4] = {0, 0, 0, 0};
                        for (int v = 1; v <= V; ++v) {
                            const int64_t h = H(g, v);
                            if (!h) continue;
                            cap[0] += h * v;
                            cap[1] += h * ((v >> 1) << 1);
                            cap[2] += h * ((v >> 2) << 2);
                            cap[3] += h * ((v >> 3) << 3);
                        }
                        const uint64_t dw = my_dem[g * kPlanBlock];
                        uint32_t d = 0;
#pragma unroll
                        for (int e = 3; e >= 0; --e) {
                            const uint32_t f = (uint32_t)(dw >> (16 * e)) & 0xffffu;
                            d += f;
                            if (f == 0) continue;  // dominated by the class above
                            const int64_t q = cap[e] / d;
                            if (best < 0 || q < best) best = q;
                        }
                    }
                    n = best < 0 ? 0 : best;
                    if (n == 0) {
                        st = HEDDLE_CAND_NO_FIT;
                    } else if (st0 == HEDDLE_CAND_OOM) {
                        st = HEDDLE_CAND_OOM;
                    } else if (t == 0) {
                        // the whole cluster is free: n, T and B are the standalone ones
                        T = sl.T[c];
                        B = sl.B[c];
                        st = HEDDLE_CAND_OK;
                        if (n != (int64_t)sl.ndp[c]) atomicOr(a.err, kErrInternal);
                    } else {
                        // Evaluate with this n: T = (M-1) max t_s + sum t_s + max g_s
                        int64_t tmax = 0, tsum = 0;
                        uint64_t bestG = 0, bestD = 1;
                        int sg = -1;
                        int hi = sl.bounds[c];
                        for (int s = 0; s < S; ++s) {
                            const int b = sl.code[(int64_t)s * sl.stride + c];
                            const int g = b & 7, j = (b >> 3) & 3;
                            const int lo = hi;
                            hi = sl.bounds[(int64_t)(s + 1) * sl.bstride + c];
                            int64_t cs = 0;
                            if (s + 1 < S) {
                                const int bn = sl.code[(int64_t)(s + 1) * sl.stride + c];
                                const int h = bn & 7, jn = (bn >> 3) & 3;
                                const int same = (g == h) && ((1 << j) + (1 << jn) <= maxn[g]);
                                cs = p2p[(g * 8 + h) * 2 + same];
                            }
                            const int64_t* row = P + (g * 4 + j) * (L + 1);
                            const int64_t ts = row[hi] - row[lo] + cs;
                            tmax = max(tmax, ts);
                            tsum += ts;
                            const uint64_t G = (uint64_t)(PB[hi] - PB[lo]);
                            const uint64_t D = (uint64_t)inter[g] << j;
                            if (sg < 0 || (u128)G * bestD > (u128)bestG * D) {
                                sg = s;
                                bestG = G;
                                bestD = D;
                            }
                        }
                        int64_t gmax = 0;
                        if (n > 1) {
                            const u128 num = (u128)(2 * (uint64_t)(n - 1) * 1000000000ull) * bestG;
                            bool ok = true;
                            gmax = (int64_t)ceil_div_u128(num, (uint64_t)n * bestD, &ok);
                            if (!ok) atomicOr(a.err, kErrInternal);
                        }
                        T = (int64_t)(M - 1) * tmax + tsum + gmax;
                        B = tmax;
                        st = HEDDLE_CAND_OK;
                    }
                    if (st == HEDDLE_CAND_OK) {
                        thr = __dadd_rn(thr, __ddiv_rn(__dmul_rn((double)(n * (int64_t)M), 1e9), (double)T));
                        placed = t + 1;
                        // place n copies of the groups, largest first
                        for (int e = 3; e >= 0; --e) {
                            const int w = 1 << e;
                            for (uint32_t pm = present; pm; pm &= pm - 1) {
                                const int g = __ffs(pm) - 1;
                                int64_t left = (int64_t)(((my_dem[g * kPlanBlock] >> (16 * e)) & 0xffffu) >> e) * n;
                                while (left > 0) {
                                    if (w <= V && H(g, w) > 0) {
                                        // nodes with exactly w free: m of them filled
                                        const int64_t m = min(left, (int64_t)H(g, w));
                                        H(g, w) -= (uint16_t)m;
                                        H(g, 0) += (uint16_t)m;
                                        left -= m;
                                        continue;
                                    }
                                    int v = w + 1;
                                    while (v <= V && H(g, v) == 0) ++v;
                                    if (v > V) {
                                        atomicOr(a.err, kErrInternal);  // n came from these nodes
                                        break;
                                    }
                                    H(g, v) -= 1;
                                    H(g, v - w) += 1;
                                    left -= 1;
                                }
                            }
                        }
                    }
                }
                if (st != HEDDLE_CAND_OK) ended = true;
            }
            if (t > 0) {  // the first template keeps its standalone results
                sl.T[c] = T;
                sl.B[c] = B;
                sl.ndp[c] = (uint16_t)(st == HEDDLE_CAND_OK || st == HEDDLE_CAND_OOM ? n : 0);
                sl.status[c] = st;
                // an OK template keeps its standalone split; any other
                // status clears the planes
                if (st != HEDDLE_CAND_OK && !sl.bounds_scratch)
                    for (int s = 0; s <= kMaxStages; ++s) sl.bounds[(int64_t)s * sl.bstride + c] = 0;
            }
        }
        a.placed[c] = (uint8_t)placed;
        a.thr[c] = thr;
    };
    // ---- one warp a plan
    auto walk = [&](int64_t c) {
        for (int i = lane; i < kMaxTypes * (V + 1); i += 32) hist[i / (V + 1)][i % (V + 1)] = init[i / (V + 1)][i % (V + 1)];
        __syncwarp();
        const int nt = min((int)a.n_tmpl[c], a.slots);
        bool ended = false;
        int placed = 0;
        double thr = 0.0;  // lane 0's
        // (the slots past the plan's templates were priced SKIPPED)
        for (int t = 0; t < nt; ++t) {
            const PlanSlot& sl = a.slot[t];
            uint8_t st = HEDDLE_CAND_SKIPPED;
            int64_t T = -1, B = -1;
            uint32_t n = 0;
            const int S = sl.S[c];
            const int M = sl.M[c];
            const uint8_t st0 = ended ? (uint8_t)HEDDLE_CAND_SKIPPED : sl.status[c];
            if (!ended && st0 == HEDDLE_CAND_INVALID) {
                st = HEDDLE_CAND_INVALID;
            } else if (!ended) {
                // this lane's stage
                const bool live = lane < S;
                const int b = live ? sl.code[(int64_t)lane * sl.stride + c] : 0;
                const int g = b & 7, j = (b >> 3) & 3;
                dem[lane] = 0;
                __syncwarp();
                if (live) {
                    const int unit = (1 << j) <= maxn[g] ? (1 << j) : pow2[g];
                    atomicAdd(&dem[4 * g + 31 - __clz(unit)], 1u << j);
                }
                __syncwarp();
                // this lane's (type, class e): n = min over those with groups
                // of floor(cap / demand), demand in classes e and above, cap =
                // sum over nodes of floor(free / 2^e) 2^e (a class without
                // groups is dominated by the one above)
                {
                    const int gt = lane >> 2, e = lane & 3;
                    const uint32_t f = dem[lane];
                    const uint32_t d1 = __shfl_down_sync(kFull, f, 1), d2 = __shfl_down_sync(kFull, f, 2),
                                   d3 = __shfl_down_sync(kFull, f, 3);
                    const uint32_t d = f + (e < 3 ? d1 : 0) + (e < 2 ? d2 : 0) + (e < 1 ? d3 : 0);
                    uint32_t cap = 0;
                    for (int v = 1; v <= V; ++v) cap += (uint32_t)hist[gt][v] * (uint32_t)((v >> e) << e);
                    n = __reduce_min_sync(kFull, f ? cap / d : 0xffffffffu);
                    if (n == 0xffffffffu) n = 0;
                }
                if (n == 0) {
                    st = HEDDLE_CAND_NO_FIT;
                } else if (st0 == HEDDLE_CAND_OOM) {
                    st = HEDDLE_CAND_OOM;
                } else if (t == 0) {
                    // the whole cluster is free: n, T and B are the standalone ones
                    T = sl.T[c];
                    B = sl.B[c];
                    st = HEDDLE_CAND_OK;
                    if (n != (uint32_t)sl.ndp[c] && lane == 0) atomicOr(a.err, kErrInternal);
                } else {
                    // Evaluate with this n: T = (M-1) max t_s + sum t_s + max g_s
                    const int lo = live ? sl.bounds[(int64_t)lane * sl.bstride + c] : 0;
                    const int hi = live ? sl.bounds[(int64_t)(lane + 1) * sl.bstride + c] : 0;
                    const int bn = __shfl_down_sync(kFull, b, 1);
                    int64_t ts = 0;
                    uint64_t G = 0, D = 1;
                    if (live) {
                        if (lane + 1 < S) {
                            const int h = bn & 7, jn = (bn >> 3) & 3;
                            const int same = (g == h) && ((1 << j) + (1 << jn) <= maxn[g]);
                            ts = p2p[(g * 8 + h) * 2 + same];
                        }
                        const int64_t* row = P + (g * 4 + j) * (L + 1);
                        ts += row[hi] - row[lo];
                        G = (uint64_t)(PB[hi] - PB[lo]);
                        D = (uint64_t)inter[g] << j;
                    }
                    const int64_t tmax = wp::wmax64(ts), tsum = wp::wsum64(ts);
                    // the largest G / (k bw), compared exactly
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) {
                        const uint64_t G2 = __shfl_xor_sync(kFull, G, o), D2 = __shfl_xor_sync(kFull, D, o);
                        if ((u128)G2 * D > (u128)G * D2) {
                            G = G2;
                            D = D2;
                        }
                    }
                    int64_t gmax = 0;
                    if (n > 1) {
                        const u128 num = (u128)(2 * (uint64_t)(n - 1) * 1000000000ull) * G;
                        bool ok = true;
                        gmax = (int64_t)ceil_div_u128(num, (uint64_t)n * D, &ok);
                        if (!ok) atomicOr(a.err, kErrInternal);
                    }
                    T = (int64_t)(M - 1) * tmax + tsum + gmax;
                    B = tmax;
                    st = HEDDLE_CAND_OK;
                }
                if (st == HEDDLE_CAND_OK) {
                    if (lane == 0)
                        thr = __dadd_rn(thr, __ddiv_rn(__dmul_rn((double)((int64_t)n * M), 1e9), (double)T));
                    placed = t + 1;
                    // place n copies of the groups, largest first, a type per lane
                    if (lane < NT) {
                        uint16_t* H = hist[lane];
                        for (int e = 3; e >= 0; --e) {
                            const int w = 1 << e;
                            int64_t left = (int64_t)(dem[4 * lane + e] >> e) * n;
                            while (left > 0) {
                                if (w <= V && H[w] > 0) {
                                    // nodes with exactly w free: m of them filled
                                    const int64_t m = min(left, (int64_t)H[w]);
                                    H[w] -= (uint16_t)m;
                                    H[0] += (uint16_t)m;
                                    left -= m;
                                    continue;
                                }
                                int v = w + 1;
                                while (v <= V && H[v] == 0) ++v;
                                if (v > V) {
                                    atomicOr(a.err, kErrInternal);  // n came from these nodes
                                    break;
                                }
                                H[v] -= 1;
                                H[v - w] += 1;
                                left -= 1;
                            }
                        }
                    }
                    __syncwarp();
                }
            }
            if (st != HEDDLE_CAND_OK) ended = true;
            if (t > 0) {  // the first template keeps its standalone results
                if (lane == 0) {
                    sl.T[c] = T;
                    sl.B[c] = B;
                    sl.ndp[c] = (uint16_t)(st == HEDDLE_CAND_OK || st == HEDDLE_CAND_OOM ? n : 0);
                    sl.status[c] = st;
                }
                // an OK template keeps its standalone split; any other
                // status clears the planes
                if (st != HEDDLE_CAND_OK && !sl.bounds_scratch)
                    for (int s = lane; s <= kMaxStages; s += 32) sl.bounds[(int64_t)s * sl.bstride + c] = 0;
            }
        }
        if (lane == 0) {
            a.placed[c] = (uint8_t)placed;
            a.thr[c] = thr;
        }
        __syncwarp();  // the warp's histogram and demand are reused
    };
    const int64_t stride = (int64_t)gridDim.x * a.per_pass;
    int64_t c0 = (int64_t)blockIdx.x * a.per_pass;
    while (true) {
        const bool more = c0 < a.n;  // uniform over the CTA
        if (more) {
            const int64_t c = c0 + threadIdx.x;
            bool walks = false;
            if ((int)threadIdx.x < a.per_pass && c < a.n) {
                // a plan walks from its second template on; the others keep
                // their slots as priced (templates past the first OK-alone
                // prefix were priced SKIPPED) and take the first template's
                // throughput if it is OK
                const int nt = min((int)a.n_tmpl[c], a.slots);
                const bool ok0 = nt >= 1 && a.slot[0].status[c] == HEDDLE_CAND_OK;
                walks = ok0 && nt >= 2;
                if (!walks) {
                    double thr = 0.0;
                    if (ok0) {
                        const PlanSlot& s0 = a.slot[0];
                        const int64_t n0 = s0.ndp[c];
                        thr = __ddiv_rn(__dmul_rn((double)(n0 * (int64_t)s0.M[c]), 1e9), (double)s0.T[c]);
                    }
                    a.placed[c] = ok0 ? 1 : 0;
                    a.thr[c] = thr;
                }
            }
            const unsigned wm = __ballot_sync(0xffffffffu, walks);
            if (wm) {
                int q0 = 0;
                if (lane == __ffs(wm) - 1) q0 = atomicAdd(&queued, __popc(wm));
                q0 = __shfl_sync(0xffffffffu, q0, __ffs(wm) - 1);
                if (walks) queue[q0 + __popc(wm & ((1u << lane) - 1))] = (int32_t)(c0 + threadIdx.x);
            }
        }
        __syncthreads();
        const int have = queued;
        __syncthreads();
        if (have >= kPlanBlock || !more) {
            int alone_min = a.alone_min;
            if (alone_min == 0) {  // by the depth of the queued plans
                alone_min = kAloneMin;
                if (have >= alone_min) {
                    unsigned depth = 0;
                    for (int i = threadIdx.x; i < have; i += kPlanBlock) {
                        const int64_t c = queue[i];
                        const int nt = min((int)a.n_tmpl[c], a.slots);
                        for (int t = 0; t < nt; ++t) depth = max(depth, min((unsigned)a.slot[t].S[c], (unsigned)kMaxStages));
                    }
                    depth = __reduce_max_sync(kFull, depth);
                    if (lane == 0) sh.deep[warp] = (int)depth;
                    __syncthreads();
                    int deepest = 0;
                    for (int w = 0; w < kPlanWarps; ++w) deepest = max(deepest, sh.deep[w]);
                    alone_min += kAlonePerStage * deepest;
                }
            }
            if (have >= alone_min) {  // 128 at a time, a thread each, while that many are left
                const int n1 = min(have, kPlanBlock);
                if (threadIdx.x < n1) walk_alone(queue[have - n1 + threadIdx.x]);
                if (threadIdx.x == 0) queued = have - n1;
            } else {  // a warp each
                for (int i = warp; i < have; i += kPlanWarps) walk(queue[i]);
                if (threadIdx.x == 0) queued = 0;
            }
        }
        __syncthreads();
        if (!more && queued == 0) break;
        if (more) c0 += stride;
    }
}

}  // namespace

cudaError_t launch_plans(const PlanArgs& a, int num_sms, cudaStream_t st) {
    if (a.n <= 0) return cudaSuccess;
    if (a.vmax < 1 || a.vmax > kPlanMaxNode) return cudaErrorInvalidValue;
    const size_t smem = plan_smem(a.lay.NT, a.vmax);
    int per_sm = 0;
    const cudaError_t e = resident_blocks(reinterpret_cast<const void*>(&plan_kernel), kPlanBlock, smem, &per_sm);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    const int64_t most = (int64_t)num_sms * per_sm;
    PlanArgs b = a;
    b.per_pass = (int32_t)std::min<int64_t>(std::max<int64_t>((a.n + most - 1) / most, kPlanWarps), kPlanBlock);
    const int grid = (int)std::min<int64_t>((a.n + b.per_pass - 1) / b.per_pass, most);
    plan_kernel<<<grid, kPlanBlock, smem, st>>>(b);
    return cudaGetLastError();
}

}  // namespace hd
