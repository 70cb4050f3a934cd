// heddle_gsearch.cu -- general PartitionLayers + Evaluate (§3.1 listing,
// §5.2 memory validation, §5.3 iteration time) for models whose layers
// differ, one thread per worklist entry.
//
// Stage s "holds" [i, j) at a bound B when the interval's time plus the
// stage's P2P is at most B and its state plus in-flight activations fit the
// stage's memory; both grow with the interval, so a stage that holds an
// interval holds every part of it.
//
// Probe of a bound B.  U_0 = 0, and U_{s+1} bounds every feasible end of
// stage s from above: the furthest end stage s reaches from U_s (a later
// start reaches no less far), or, when it does not hold layer U_s at all
// (every longer interval from a start up to U_s contains that layer), the
// largest end j <= U_s whose last layer j - 1 it holds.
//   * U_s runs out, or the last stage does not hold [U_{S-1}, L): no split
//     exists, whatever the holes below U_s;
//   * every stage advanced: the chain itself is a split, so B is feasible;
//   * some stage stepped back: a split is built from the end, a_s the
//     largest start at most U_s and below a_{s+1} whose last layer a_s - 1
//     the stage before holds; if every stage holds its part, B is feasible.
//     If not, the probe cannot decide: the entry goes to the warp kernel
//     (heddle_wsearch.cu), which runs the set-based probe.
// The answers are exact without any condition on the layers.  (A rule that
// takes only entries whose stages hold any one layer of the model sends 45%
// of the entries of an 80-layer profile with a heavy first and last layer to
// the warp kernel: 1.41 ms there per 300,007 candidates beside 0.12 ms here;
// this one 0.0 to 0.8%, 0.16 and 0.35 ms.)
//
// The split at B*.  Symmetrically V_S = L and V_s bounds every feasible start
// of stage s from below; the smallest boundary is at least
// max(a_s + 1, V_{s+1}), and past that the next one whose first layer stage
// s + 1 holds.  If every stage holds the part this gives it, no smaller
// split exists; if not, the entry goes to the warp kernel.
//
// The search: a memory-only probe where the screen could not decide memory,
// the saturating balance as first guess, each probe snapping the bracket to
// its largest accepted or smallest rejected stage time (every bound in
// [hi, B] has that split, every bound in [B, lo) meets the same rejections),
// galloping, then bisecting.  The
// kernel runs only when the depth buckets hold at least
// PriceArgs::thread_min entries (a few entries would leave it as long as its
// longest serial chain); each warp takes 32 entries at a time, deepest first.

#include <algorithm>

#include "heddle_wprobe.cuh"

namespace hd {
namespace {

constexpr int kGBlock = 128;
constexpr int kGWarps = kGBlock / 32;
constexpr unsigned kFull = 0xffffffffu;
constexpr int kGMaxIters = 256;
constexpr int kStepShift = 7;
// Undecided probes after which an entry goes to the warp kernel: they do not
// snap the bracket, so closing it takes a bisection down to 1 ns, and a warp
// waits for its slowest lane.
constexpr int kMaxDoubts = 3;
constexpr int64_t kNoBound = (int64_t)1 << 61;  // above every stage time
constexpr int kGZeroP2P = 128;  // index of a zero after the 8 x 8 x 2 P2P table

struct GTabs {
    const int64_t* P;      // [NT][4][L+1] prefix ns per (type, degree)
    const longlong2* SA;   // [L+1] prefix of (state bytes, activation bytes)
    const int64_t* PB;     // [L+1] prefix of gradient bytes
    const int64_t* p2p;    // [8][8][2] (index 128: no next stage, P2P 0)
    const int64_t* mem;    // [8]
    const int64_t* inter;  // [8]
    const float* rqavg;    // [NT * 4] 1 / the average layer time
    const int64_t* minmid; // [NT * 4] the cheapest layer besides the first and the last
    const uint8_t* win;    // [8 * 4][33] the longest run of layers within memory, per in-flight count
    int L;
};

// Stage word (per thread, in shared memory): bits 0-4 the stage byte's type
// and degree, bits 5-12 the P2P index, bits 13-18 the in-flight count f,
// bits 19-26 the memory run during the guess, then U_s during a probe and
// V_s during the split.
constexpr int kVShift = 19;
constexpr uint32_t kNoV = (1u << kVShift) - 1;

struct GStage {
    int row;       // offset of the prefix row
    int64_t c;     // P2P to the next stage
    int64_t capk;  // memory per GPU x devices
    int64_t f;     // in-flight micro-batches
};

__device__ __forceinline__ GStage unpack(uint32_t w, const GTabs& t) {
    GStage st;
    const int g = w & 7, j = (w >> 3) & 3;
    st.row = (g * 4 + j) * (t.L + 1);
    const int pidx = (w >> 5) & 255;
    st.c = pidx < kGZeroP2P ? t.p2p[pidx] : 0;  // the image's table has 128 entries
    st.capk = t.mem[g] << j;
    st.f = (w >> 13) & 63;
    return st;
}

// Stage s holding layers [i, j): fits memory?  Its time in *cost.
__device__ __forceinline__ bool fits_mem(const GTabs& t, const GStage& st, int i, int j) {
    const longlong2 si = t.SA[i], sj = t.SA[j];
    return (int64_t)(sj.x - si.x) + st.f * (int64_t)(sj.y - si.y) <= st.capk;
}
__device__ __forceinline__ int64_t cost(const GTabs& t, const GStage& st, int i, int j) {
    return t.P[st.row + j] - t.P[st.row + i] + st.c;
}

// The largest x in [lo, hi] with ok(x), for a test that holds up to some
// point and fails beyond it (ok(lo) taken as true), searched from an
// estimate x0: gallop away from x0 (1, 2, 4, ... positions) until the
// boundary is bracketed, then bisect.  With a good estimate -- the prefix
// sums are nearly linear, exactly so for equal layers -- that is two tests
// instead of a bisection's eight.
template <class F>
__device__ __forceinline__ int last_ok(int lo, int hi, int x0, F ok) {
    x0 = min(max(x0, lo), hi);
    int a, b;
    if (x0 == lo || ok(x0)) {
        int good = x0, step = 1;
        b = hi;
        while (true) {
            const int k = good + step;
            if (k > hi) break;
            if (!ok(k)) {
                b = k - 1;
                break;
            }
            good = k;
            step <<= 1;
        }
        a = good;
    } else {
        int fail = x0, step = 1;
        a = lo;
        while (true) {
            const int k = fail - step;
            if (k <= lo) break;
            if (ok(k)) {
                a = k;
                break;
            }
            fail = k;
            step <<= 1;
        }
        b = fail - 1;
    }
    while (a < b) {
        const int mid = (a + b + 1) >> 1;
        if (ok(mid)) a = mid;
        else b = mid - 1;
    }
    return a;
}

// Layers of stage st that a bound and its memory admit, estimated from the
// average layer time and the longest run of layers its memory holds anywhere
// (for the searches' first guesses).
__device__ __forceinline__ float layers_est(const GTabs& t, const GStage& st, int row_idx, int64_t room) {
    const float by_time = room > 0 ? u64_to_float((uint64_t)room) * t.rqavg[row_idx] : 0.f;
    return fminf(by_time, (float)t.win[row_idx * 33 + (int)st.f]);
}

// The furthest end j in (u, lim] of a stage starting at u within B and its
// memory (u if none; for the last stage only L counts).  acc: the stage time
// at that end (-1 if none); rej: the stage time at the next end (the last
// stage: at L) if memory admits it there and its time is above B (kInf
// otherwise).
//
// The terms of u move to the other side once (the memory sums stay below
// 2^57, B - c + P[u] below 2^62), so a test is two loads, one multiplication
// and two comparisons.  Four consecutive ends around the estimate are tested
// side by side, whatever they say, and only a boundary outside them is
// searched for: a warp's lanes stay together, where a gallop from the
// estimate left 8.2 of 32 lanes active.
__device__ __forceinline__ int reach_of(const GTabs& t, const GStage& st, int row_idx, int u, int lim, bool last,
                                        int64_t B, int64_t& acc, int64_t& rej) {
    const int64_t* P = t.P + st.row;
    const longlong2 su = t.SA[u];
    const int64_t Pu = P[u];
    const int64_t time_lim = B - st.c + Pu, mem_lim = st.capk + su.x + st.f * (int64_t)su.y;
    auto ok = [&](int j) {
        const longlong2 sj = t.SA[j];
        return P[j] <= time_lim && (int64_t)sj.x + st.f * (int64_t)sj.y <= mem_lim;
    };
    const int est = (int)layers_est(t, st, row_idx, B - st.c);
    const int x0 = min(max(last ? lim : u + est - 1, u), max(lim - 3, u));
    const bool o0 = x0 == u || ok(x0);
    const bool o1 = ok(min(x0 + 1, lim)), o2 = ok(min(x0 + 2, lim)), o3 = ok(min(x0 + 3, lim));
    int r = min(x0 - 1 + (int)o0 + (int)o1 + (int)o2 + (int)o3, lim);
    if (!last) {
        if (!o0) r = last_ok(u, x0 - 1, x0 - 1, ok);
        else if (o3 && x0 + 3 < lim) r = last_ok(x0 + 3, lim, x0 + 4, ok);
    }
    acc = r > u ? P[r] - Pu + st.c : -1;
    rej = kInf;
    const int q = last ? lim : r + 1;
    if (q > r && q <= lim && P[q] > time_lim) {
        const longlong2 sq = t.SA[q];
        if ((int64_t)sq.x + st.f * (int64_t)sq.y <= mem_lim) rej = P[q] - Pu + st.c;
    }
    return r;
}

// The smallest start i in [s, v) from which a stage reaches v within B and
// its memory; v if it does not hold layer v - 1.
__device__ __forceinline__ int start_of(const GTabs& t, const GStage& st, int row_idx, int s, int v, int64_t B) {
    const int64_t* P = t.P + st.row;
    const longlong2 sv = t.SA[v];
    const int64_t time_lim = P[v] + st.c - B, mem_lim = (int64_t)sv.x + st.f * (int64_t)sv.y - st.capk;
    auto ok = [&](int i) {
        const longlong2 si = t.SA[i];
        return P[i] >= time_lim && (int64_t)si.x + st.f * (int64_t)si.y >= mem_lim;
    };
    const int est = (int)layers_est(t, st, row_idx, B - st.c);
    const int x0 = max(min(v - est - 1, v - 4), s);
    const int held = (int)ok(x0) + (int)ok(min(x0 + 1, v - 1)) + (int)ok(min(x0 + 2, v - 1)) +
                     (int)ok(min(x0 + 3, v - 1));
    if (held == 4 && x0 > s) return x0 - last_ok(0, x0 - s, 1, [&](int y) { return ok(x0 - y); });
    if (held == 0) {
        if (x0 + 4 >= v || !ok(v - 1)) return v;
        return v - 1 - last_ok(0, v - 1 - (x0 + 4), v - 1 - (x0 + 4), [&](int y) { return ok(v - 1 - y); });
    }
    return x0 + 4 - held;
}

// Stage holds [i, j) within B and its memory?
__device__ __forceinline__ bool holds(const GTabs& t, const GStage& st, int i, int j, int64_t B) {
    return cost(t, st, i, j) <= B && fits_mem(t, st, i, j);
}

__device__ __forceinline__ int pos_of(uint32_t w) { return (int)(w >> kVShift) & 255; }

// The split of a probe in which some stage stepped back, built from the end
// (see the head of this file); the U_s are in the stage words.  Its largest
// stage time, or -1 if a stage does not hold its part.
__device__ __noinline__ int64_t split_below(const GTabs& t, const uint32_t* sw, int S, int64_t B) {
    int end = t.L;
    int64_t hi = -1;
    GStage st = unpack(sw[(S - 1) * kGBlock], t);
    for (int s = S - 1; s >= 1; --s) {
        const GStage before = unpack(sw[(s - 1) * kGBlock], t);
        int x = min(end - 1, pos_of(sw[s * kGBlock]));
        while (x >= s && !holds(t, before, x - 1, x, B)) --x;
        if (x < s || !holds(t, st, x, end, B)) return -1;
        hi = max(hi, cost(t, st, x, end));
        end = x;
        st = before;
    }
    return holds(t, st, 0, end, B) ? max(hi, cost(t, st, 0, end)) : -1;
}

// Appends entry p to the list the warp kernel finishes, with the bracket
// [lo, hi] of B* (hi a feasible bound, -1: memory is undecided; probed: a
// probe found the split of hi).
__device__ __forceinline__ void defer(const PriceArgs& a, int64_t p, int64_t hi, int64_t lo, bool probed) {
    const int pos = atomicAdd(a.wl_count + kWlGeneral, 1);
    if (in_range(pos, a.wl_cap, a.err)) {
        a.sv_idx[pos] = (int32_t)p;
        a.sv_T[pos] = hi;
        a.sv_nM[pos] = probed ? 1 : 0;
        a.wl_T[p] = lo;
    }
}

// Below a.thread_min bucketed entries the kernel returns at once and the
// warp kernel prices the whole worklist.  Five CTAs per SM at 90 registers a
// thread: a cap that lets in six or eight measured 0.38 and 0.43 ms beside
// 0.35 ms (profiled 80-layer model, 300,007 candidates).
//
// kMemOnly: only the probe of memory, ahead of the tiled search: an entry
// without a split within memory is OOM, the others go on that search's list
// with sv_T 0 (memory known) or -1 (undecided).
template <bool kCount, bool kMemOnly>
__global__ void __launch_bounds__(kGBlock, 4) gsearch_kernel(PriceArgs a) {
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ uint64_t bar;
    __shared__ float rqavg[4 * kMaxTypes], cfl[129];
    __shared__ int64_t minmid[4 * kMaxTypes];
    __shared__ int end_of[kMaxStages + 2];
    const Layout& y = a.lay;
    const int L = y.L;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    allow_dependents();
    await_previous();
    if (threadIdx.x < 32) {
        // end_of[S] = entries of depths >= S (see eq_search_kernel)
        int x = a.wl_count[1 + (kMaxStages - lane)];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y2 = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y2;
        }
        end_of[kMaxStages - lane] = x;
        if (lane == 0) end_of[kMaxStages + 1] = 0;
    }
    __syncthreads();
    if (end_of[1] < a.thread_min) return;
    if (!wp::load_image(smem, a.img, y.searchBytes, &bar, a.err)) return;
    {
        const int64_t* P = reinterpret_cast<const int64_t*>(smem + y.offP);
        // per (type, degree) 1 / the average layer time and the cheapest
        // layer besides the first and the last
        for (int r = warp; r < 4 * y.NT; r += kGWarps) {
            int64_t m = kInf;
            for (int l = 1 + lane; l + 1 < L; l += 32) m = min(m, P[r * (L + 1) + l + 1] - P[r * (L + 1) + l]);
            m = wp::wmin64(m);
            if (lane == 0) {
                minmid[r] = m;
                const int64_t all = P[r * (L + 1) + L];
                rqavg[r] = all > 0 ? (float)L / u64_to_float((uint64_t)all) : 0.f;
            }
        }
        const int64_t* p2p = reinterpret_cast<const int64_t*>(smem + y.offP2P);
        for (int i = threadIdx.x; i < 129; i += blockDim.x) cfl[i] = i < 128 ? u64_to_float((uint64_t)p2p[i]) : 0.f;
        __syncthreads();
    }
    GTabs t;
    t.P = reinterpret_cast<const int64_t*>(smem + y.offP);
    t.SA = reinterpret_cast<const longlong2*>(smem + y.offSA);
    t.PB = reinterpret_cast<const int64_t*>(smem + y.offPB);
    t.p2p = reinterpret_cast<const int64_t*>(smem + y.offP2P);
    t.mem = reinterpret_cast<const int64_t*>(smem + y.offMem);
    t.inter = reinterpret_cast<const int64_t*>(smem + y.offInter);
    t.rqavg = rqavg;
    t.minmid = minmid;
    t.win = smem + y.offWin;
    t.L = L;
    const int32_t* maxn = reinterpret_cast<const int32_t*>(smem + y.offMaxN);
    uint32_t* sw = reinterpret_cast<uint32_t*>(smem + ((y.searchBytes + 127u) & ~127u)) + threadIdx.x;

    unsigned long long checks = 0, probes = 0, priced = 0;
    // the entries filed in the depth buckets (every worklist entry)
    const int64_t entries = min((int64_t)*a.wl_count, (int64_t)a.wl_cap);
    const int64_t count = min((int64_t)end_of[1], entries);
    // each warp prices 32 entries (deepest first): its own first, then the
    // next untaken ones whenever it is free
    const int64_t first = (int64_t)gridDim.x * kGBlock;
    auto take = [&]() {
        int b = 0;
        if (lane == 0) b = atomicAdd(a.wl_count + kWlTakeThread, 32);
        return first + __shfl_sync(0xffffffffu, b, 0);
    };
    for (int64_t base = ((int64_t)blockIdx.x * kGWarps + warp) * 32; base < count; base = take()) {
        const int64_t g = base + lane;
        bool have = g < count;
        int64_t p = 0;
        if (have) {
            int lo_d = 1, hi_d = kMaxStages;
            while (lo_d < hi_d) {
                const int mid = (lo_d + hi_d + 1) >> 1;
                if (end_of[mid] > g) lo_d = mid; else hi_d = mid - 1;
            }
            const int64_t off = g - end_of[lo_d + 1];
            have = in_range(off, end_of[lo_d] - end_of[lo_d + 1], a.err);
            if (have) p = a.wl_bucket[(int64_t)(lo_d - 1) * a.wl_cap + off];
            have = have && in_range(p, entries, a.err);
        }
        const int64_t c = have ? a.wl_idx[p] : 0;
        const int S = have ? a.wl_S[p] : 1, M = have ? a.wl_M[p] : 1;
        const int64_t n = have ? a.wl_n[p] : 1;
        const bool memok = have && a.wl_memok[p] != 0;
        have = have && in_range(c, a.n, a.err) && in_range(S - 1, kMaxStages, a.err);
        int64_t hiB = 0, LB = 0, B = 0;
        if (have) {
            if (kCount) ++priced;
            // pack the stages; a bound no split beats and a bound feasible
            // whenever memory is (the entry's 32-byte row of stage bytes, read a byte
            // per stage: an array indexed by the stage would live in local memory;
            // ordinary loads: the screen may have written it while this kernel
            // already ran)
            const uint8_t* row = a.wl_code + p * kMaxStages;
            int next = row[0];
            for (int s = 0; s < S; ++s) {
                const int code = next;
                next = s + 1 < S ? row[s + 1] : 0;
                const int gg = code & 7, jj = (code >> 3) & 3;
                int pidx = kGZeroP2P;
                if (s + 1 < S) {
                    const int h = next & 7, jn = (next >> 3) & 3;
                    pidx = (gg * 8 + h) * 2 + ((gg == h) && ((1 << jj) + (1 << jn) <= maxn[gg]));
                }
                const int f = min(S - s, M);
                const uint32_t w = (uint32_t)(code & 31) | ((uint32_t)pidx << 5) | ((uint32_t)f << 13);
                const GStage st = unpack(w, t);
                // the first stage holds layer 0, the last one layer L - 1, the
                // others at least one layer besides these
                const int64_t least = s == 0       ? t.P[st.row + 1] - t.P[st.row]
                                      : s + 1 == S ? t.P[st.row + L] - t.P[st.row + L - 1]
                                                   : t.minmid[gg * 4 + jj];
                LB = max(LB, least + st.c);
                hiB = max(hiB, t.P[st.row + L] + st.c);
                sw[s * kGBlock] = w;
            }
            // first guess: the saturating continuous balance with each stage's
            // average layer time and memory run from layer 0
            if (!kMemOnly) {
                float inv = 0.f, cw = 0.f, flo = 0.f;
                for (int s = 0; s < S; ++s) {
                    const uint32_t w = sw[s * kGBlock];
                    const int ri = (w & 7) * 4 + ((w >> 3) & 3);
                    const float rq = rqavg[ri], cf = cfl[(w >> 5) & 255];
                    // the longest run of layers memory admits
                    sw[s * kGBlock] = (w & kNoV) | ((uint32_t)t.win[ri * 33 + ((w >> 13) & 63)] << kVShift);
                    inv += rq;
                    cw += cf * rq;
                    if (rq > 0.f) flo = fmaxf(flo, cf + 1.0f / rq);
                }
                const float fhi = u64_to_float((uint64_t)hiB);
                float Bf = fmaxf(flo, inv > 0.f ? ((float)L + 0.5f * (float)S + cw) / inv : flo);
                for (int it = 0; it < 3; ++it) {
                    Bf = fminf(Bf, fhi);
                    float cnt = 0.f, sl = 0.f, nb = 0.f;
                    for (int s = 0; s < S; ++s) {
                        const uint32_t w = sw[s * kGBlock];
                        const float rq = rqavg[(w & 7) * 4 + ((w >> 3) & 3)], cf = cfl[(w >> 5) & 255];
                        const float mr = (float)((w >> kVShift) & 255);
                        const float x = (Bf - cf) * rq;
                        if (rq <= 0.f || x >= mr) {
                            cnt += mr;
                        } else {
                            cnt += x;
                            sl += rq;
                            nb += 1.f;
                        }
                    }
                    const float tgt = (float)L + 0.5f * nb;
                    if (cnt >= tgt - 0.25f || sl <= 0.f) break;
                    Bf += (tgt - cnt) / sl;
                }
                B = (int64_t)float_to_u64(fmaxf(fminf(Bf, fhi), 0.f));
            }
        }
        // The threshold search on [lo, hi]; where the screen could not decide
        // memory it begins with a probe of memory alone.  One pass of the
        // loop is one stage of the lane's current probe: a lane whose probe
        // ends starts its next one in the next pass, so the lanes of a warp
        // wait for one another once per entry and not once per probe.
        //
        // An undecided bound moves lo like an infeasible one, but not
        // lo_proven: the bracket left at the end goes to the warp kernel.
        // The gallop's first step is the next breakpoint, then 2^-7 of the
        // bound and doubling: with layers that differ the breakpoints lie too
        // close for steps that start from 1 ns (at most 14 probes on the
        // ragged 80-layer profile, not 32).
        int64_t lo = LB, hi = hiB, lo_proven = LB, step = 1, shi = -1, slo = kInf;
        bool lo_known = false, hi_known = false, oom = false, undecided = false, back = false;
        int it = 0, s = 0, u = 0, doubts = 0;
        const int64_t guess = min(max(B, lo), hi - 1);
        B = memok ? guess : kNoBound;
        bool run = have && !(memok && (kMemOnly || lo >= hi));
        while (__any_sync(kFull, run)) {
            if (!run) continue;
            const uint32_t w = sw[s * kGBlock];
            sw[s * kGBlock] = (w & kNoV) | ((uint32_t)u << kVShift);
            const GStage st = unpack(w, t);
            const bool last = s + 1 == S;
            int64_t acc, rej;
            int r = reach_of(t, st, (w & 7) * 4 + ((w >> 3) & 3), u, L - (S - 1 - s), last, B, acc, rej);
            slo = min(slo, rej);
            if (kCount) checks += 2;
            if (r == u && !last) {
                // layer u alone does not fit: the largest end at or below u
                back = true;
                for (; r > s; --r) {
                    if (kCount) ++checks;
                    if (fits_mem(t, st, r - 1, r)) {
                        const int64_t v = cost(t, st, r - 1, r);
                        if (v <= B) break;
                        slo = min(slo, v);
                    }
                }
            }
            const bool fails = last ? r < L : r < s + 1;
            if (!fails) shi = max(shi, acc);
            u = r;
            ++s;
            if (!fails && !last) continue;
            // ---- the probe's answer moves the bracket
            if (kCount) ++probes;
            bool feasible = !fails, unsure = false;
            if (feasible && back) {
                shi = split_below(t, sw, S, B);
                feasible = shi >= 0;
                unsure = !feasible;
            }
            if (B == kNoBound) {
                // memory only: OOM, else a tighter feasible bound
                run = !kMemOnly && feasible && lo < shi;
                oom = fails;
                undecided = unsure;
                hi = feasible ? shi : hi;
                if (lo >= hi) lo_proven = hi;
                B = min(guess, hi - 1);
            } else {
                if (feasible) {
                    hi = shi;
                    hi_known = true;
                } else {
                    lo = unsure ? B + 1 : min(slo, hi);
                    if (!unsure) lo_proven = lo;
                    lo_known = true;
                }
                if (!lo_known) {
                    B = hi - step;
                    step = max(2 * step, hi >> kStepShift);
                } else if (!hi_known) {
                    B = lo + step - 1;
                    step = max(2 * step, lo >> kStepShift);
                } else {
                    B = lo + (hi - lo) / 2;
                }
                if (unsure) ++doubts;
                run = lo < hi && doubts < kMaxDoubts;
                if (++it > kGMaxIters) {
                    atomicOr(a.err, kErrSearchBound);
                    run = false;
                }
                B = min(max(B, lo), hi - 1);
            }
            s = u = 0;
            shi = -1;
            slo = kInf;
            back = false;
        }
        if (!have) continue;
        if (oom) {
            a.T[c] = -1;
            a.B[c] = -1;
            a.ndp[c] = (uint16_t)n;
            a.status[c] = HEDDLE_CAND_OOM;
            a.wl_T[p] = -1;
            if (a.bounds)
                for (int q = 0; q <= kMaxStages; ++q) a.bounds[(int64_t)q * a.bstride + c] = 0;
            continue;
        }
        if (kMemOnly) {
            defer(a, p, undecided ? -1 : 0, 0, false);
            continue;
        }
        const int64_t Bstar = hi;
        if (undecided || lo_proven < hi) {
            defer(a, p, undecided ? -1 : hi, lo_proven, hi_known);
            continue;
        }
        // the split: the smallest start V_s from which stage s reaches
        // V_{s+1} -- or, when it does not hold layer V_{s+1} - 1, the first
        // start from V_{s+1} on whose layer it holds -- into bits 19-26 of
        // the stage words
        {
            int v = L;
            for (int s = S - 1; s >= 1; --s) {
                const uint32_t w = sw[s * kGBlock];
                const GStage st = unpack(w, t);
                if (kCount) checks += 2;
                const int from = start_of(t, st, (w & 7) * 4 + ((w >> 3) & 3), s, v, Bstar);
                if (from < v) {
                    v = from;
                } else {
                    while (v < L - (S - s) && !holds(t, st, v, v + 1, Bstar)) ++v;
                    v = min(v, L - (S - s));
                }
                sw[s * kGBlock] = (w & kNoV) | ((uint32_t)v << kVShift);
            }
        }
        // Evaluate: T = (M-1) max t_s + sum t_s + max g_s
        int64_t tmax = 0, tsum = 0;
        uint64_t bestG = 0, bestD = 1;
        int at = 0;
        bool bad = false;
        for (int s = 0; s < S; ++s) {
            const uint32_t w = sw[s * kGBlock];
            const GStage st = unpack(w, t);
            int nxt = L;
            if (s + 1 < S) {
                // the first boundary whose first layer the next stage holds
                const uint32_t wn = sw[(s + 1) * kGBlock];
                const GStage sn = unpack(wn, t);
                nxt = max(at + 1, pos_of(wn));
                while (nxt < L - (S - 1 - s) && !holds(t, sn, nxt, nxt + 1, Bstar)) ++nxt;
            }
            bad |= !holds(t, st, at, nxt, Bstar);
            if (a.bounds) a.bounds[(int64_t)(s + 1) * a.bstride + c] = (uint8_t)nxt;
            const int64_t ts = cost(t, st, at, nxt);
            tmax = max(tmax, ts);
            tsum += ts;
            if (n > 1) {
                const uint64_t G = (uint64_t)(t.PB[nxt] - t.PB[at]);
                const uint64_t D = (uint64_t)t.inter[w & 7] << ((w >> 3) & 3);
                if (s == 0 || (u128)G * bestD > (u128)bestG * D) {
                    bestG = G;
                    bestD = D;
                }
            }
            at = nxt;
        }
        if (a.bounds) {
            a.bounds[c] = 0;
            for (int s = S + 1; s <= kMaxStages; ++s) a.bounds[(int64_t)s * a.bstride + c] = 0;
        }
        if (bad) {
            defer(a, p, Bstar, Bstar, true);  // the warp kernel writes the whole row
            continue;
        }
        if (tmax != Bstar) atomicOr(a.err, kErrInternal);
        int64_t gmax = 0;
        if (n > 1) {
            // ring all-reduce over n replicas: ceil(2(n-1) G 1e9 / (n k bw))
            const u128 num = (u128)(2 * (uint64_t)(n - 1) * 1000000000ull) * bestG;
            bool ok = true;
            gmax = (int64_t)ceil_div_u128(num, (uint64_t)n * bestD, &ok);
            if (!ok) atomicOr(a.err, kErrInternal);
        }
        const int64_t T = (int64_t)(M - 1) * Bstar + tsum + gmax;
        a.T[c] = T;
        a.wl_T[p] = T;
        a.wl_nM[p] = (uint32_t)n * (uint32_t)M;
        a.B[c] = Bstar;
        a.ndp[c] = (uint16_t)n;
        a.status[c] = HEDDLE_CAND_OK;
    }
    if (kCount) {
        unsigned long long v0 = checks, v1 = probes, v2 = priced;
#pragma unroll
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

template <bool kCount, bool kMemOnly>
cudaError_t launch(const PriceArgs& a, int num_sms, cudaStream_t st) {
    const size_t smem = ((a.lay.searchBytes + 127u) & ~127u) + sizeof(uint32_t) * kMaxStages * kGBlock;
    int per_sm = 0;
    const cudaError_t e = resident_blocks(reinterpret_cast<const void*>(&gsearch_kernel<kCount, kMemOnly>), kGBlock, smem, &per_sm);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    // the worklist length is only known on the device: one wave at most
    const int64_t need = (a.n + kGBlock - 1) / kGBlock;
    const int grid = (int)std::min<int64_t>(need, (int64_t)num_sms * per_sm);
    return launch_after(a.chained, gsearch_kernel<kCount, kMemOnly>, grid, kGBlock, smem, st, a);
}

}  // namespace

cudaError_t launch_thread_search(const PriceArgs& a, int num_sms, cudaStream_t st) {
    return a.counters ? launch<true, false>(a, num_sms, st) : launch<false, false>(a, num_sms, st);
}

cudaError_t launch_memory_probe(const PriceArgs& a, int num_sms, cudaStream_t st) {
    return launch<false, true>(a, num_sms, st);
}

}  // namespace hd
