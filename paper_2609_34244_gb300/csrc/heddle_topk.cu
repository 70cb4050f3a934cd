// heddle_topk.cu -- rank and top-k of priced candidates.
//
// The rank order and the warp-level lists are in heddle_rank.cuh.
//
// One launch.  A CTA's share of the entries (the batch's results, or the
// worklist of a priced chunk) is read twice.  First every thread keeps its
// best entry; the best of 64 groups of four threads (128 pairs for k > 32)
// are ranked against each other, and the k-th of them is a bar: k entries
// rank no lower, so none below it can enter the top-k.  Then the entries not
// below the bar (the incoming state's k-th, once it holds k) are gathered
// unsorted: little more than k of them, several times k in a sorted order or
// among ties.  The rank order is strict, ties in throughput going to the smaller
// index, so many equal throughputs -- a small structure space drawn many times --
// overflow no gather.  Over a large batch's results the CTAs also post their bars,
// and each drops what falls below the best posted so far.  The CTA that draws the
// last ticket does the same once more over all CTAs' gathered entries and the
// incoming state, ranks what is left exactly against each other, and writes the
// state.  No CTA waits on another.  Where a gather overflows its buffer the CTA
// falls back on sorted warp lists and their tree merge (heddle_rank.cuh).
//
// What bounds it is latency: two passes over a few entries a thread and one
// hand-over.  Top-k phase of a pricing call into an empty
// state (events, launch included): 1,000 candidates of the 32-layer workload
// 12.2 us, 1e5 of them 18.1, 1e6 of the 80-layer one 22 (18.2, 30.3 and 35 with a
// bitonic merge per 32 entries for a floor on float keys, sorted warp lists and
// two levels of tree merges, three launches in the separate call).

#include <algorithm>

#include "heddle_rank.cuh"

namespace hd {
namespace {

constexpr int kSelBlock = 256;
constexpr int kSelWarps = kSelBlock / 32;
// entries gathered per CTA (a list of the scratch); by the last CTA
constexpr int kCandCap = kTopkListCap;
constexpr int kFinalCap = 256;
constexpr int kDirect = 96;  // at most this many are ranked without a bar
static_assert(kCandCap >= kMaxTopK, "a fallback list of k entries fits a CTA's list");
// each CTA takes at least this many entries (four a thread): fewer only add
// hand-overs
constexpr int kPerCta = 4 * kSelBlock;
// Above so many CTAs times k, the CTAs of a batch's top-k post their bars and drop
// what falls below another's (a worklist's entries lie in no such order, and fused
// calls have a running threshold).  Without it the last CTA reads all that they gather, several times k
// entries each in a sorted order or among ties: 3e5 results, k = 64, random 74 us
// a call, sorted 89, all equal 98; so 64, 35 and 37.  (Below, the exchange itself
// costs one or two microseconds: 1.4e5 random results at k = 16 21 -> 22.)
constexpr int kPostMin = 4096;
constexpr float kMargin = 1.0f - 1.0f / 65536.0f;

// One candidate entry: from a batch's results, or from the worklist of a
// priced chunk (only the searched candidates, T = -1 unless OK).  Every
// field is loaded whether or not the entry turns out valid, so the loads of
// several entries are independent and can be in flight together.
template <bool kWorklist>
__device__ __forceinline__ bool fetch(const TopkArgs& a, int64_t i, TopkEntry& e) {
    e.pad = 0;
    if (kWorklist) {
        e.T = a.wl_T[i];
        e.idx = a.base_index + a.wl_idx[i];
        e.nM = a.wl_nM[i];
        return e.T >= 0;
    }
    const bool ok = a.status[i] == HEDDLE_CAND_OK;
    e.idx = a.base_index + i;
    e.T = a.T[i];
    e.nM = (uint32_t)a.ndp[i] * (uint32_t)a.M[i];
    return ok;
}

__device__ __forceinline__ float key_of(const TopkEntry& e) { return (float)e.nM / (float)e.T; }

// No entry: ranks below every entry that processes something.
__device__ __forceinline__ TopkEntry no_entry(int at) {
    TopkEntry e;
    e.idx = INT64_MAX - at;
    e.T = 1;
    e.nM = e.pad = 0;
    return e;
}

struct Groups {
    TopkEntry best[kSelBlock / 2];
    int rank[kSelBlock / 2];
    TopkEntry kth;
};

// The k-th of the group bests of the CTA's threads' entries (no_entry where
// a thread has none): 64 groups of four threads, or 128 of two for k > 32.
// Every thread of the CTA calls it; false: fewer than k groups hold an entry.
__device__ __forceinline__ bool cta_kth(TopkEntry e, int k, Groups& g, TopkEntry& kth) {
    const int shift = k <= 32 ? 2 : 1;
    const int ngroups = kSelBlock >> shift;
    for (int o = 1; o < (1 << shift); o <<= 1) {
        TopkEntry x;
        x.idx = __shfl_xor_sync(0xffffffffu, e.idx, o);
        x.T = __shfl_xor_sync(0xffffffffu, e.T, o);
        x.nM = __shfl_xor_sync(0xffffffffu, e.nM, o);
        x.pad = 0;
        if (better(x, e)) e = x;
    }
    if ((threadIdx.x & ((1 << shift) - 1)) == 0) {
        g.best[threadIdx.x >> shift] = e;
        g.rank[threadIdx.x >> shift] = 0;
    }
    __syncthreads();
    // group i against a 1 / 2^shift share of the groups
    const int i = threadIdx.x & (ngroups - 1);
    const int part = (threadIdx.x / ngroups) * (ngroups >> shift);
    const TopkEntry mine = g.best[i];
    int r = 0;
#pragma unroll 4
    for (int j = part; j < part + (ngroups >> shift); ++j) r += better(g.best[j], mine) ? 1 : 0;
    if (r) atomicAdd(&g.rank[i], r);
    __syncthreads();
    if (threadIdx.x < ngroups && g.rank[threadIdx.x] == k - 1) g.kth = mine;
    __syncthreads();
    kth = g.kth;
    return kth.idx <= INT64_MAX - kSelBlock;
}

// The best of the CTA's threads' entries (in every thread); tmp: one per warp.
__device__ __forceinline__ TopkEntry cta_best(TopkEntry e, TopkEntry* tmp) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        TopkEntry x;
        x.idx = __shfl_xor_sync(0xffffffffu, e.idx, o);
        x.T = __shfl_xor_sync(0xffffffffu, e.T, o);
        x.nM = __shfl_xor_sync(0xffffffffu, e.nM, o);
        x.pad = 0;
        if (better(x, e)) e = x;
    }
    if ((threadIdx.x & 31) == 0) tmp[threadIdx.x >> 5] = e;
    __syncthreads();
    e = tmp[0];
    for (int w = 1; w < kSelWarps; ++w)
        if (better(tmp[w], e)) e = tmp[w];
    __syncthreads();
    return e;
}

__device__ __forceinline__ int32_t load_acquire(const int32_t* p) {
    int32_t v;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void store_release(int32_t* p, int32_t v) {
    asm volatile("st.release.gpu.global.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Append one entry per lane (want) to a list in shared memory; every lane
// of the warp calls it.  Entries past the capacity are counted only.
__device__ __forceinline__ void gather(TopkEntry* list, int* count, int cap, bool want, const TopkEntry& e) {
    const unsigned m = __ballot_sync(0xffffffffu, want);
    if (!m) return;
    const int lane = threadIdx.x & 31, lead = __ffs(m) - 1;
    int base = 0;
    if (lane == lead) base = atomicAdd(count, __popc(m));
    const int pos = __shfl_sync(0xffffffffu, base, lead) + __popc(m & ((1u << lane) - 1));
    if (want && pos < cap) list[pos] = e;
}

__device__ __forceinline__ TopkEntry state_entry(const heddle_topk_state* s, int i) {
    TopkEntry e;
    e.idx = s->idx[i];
    e.T = s->T[i];
    e.nM = s->nM[i];
    e.pad = 0;
    return e;
}

// An entry another CTA wrote: read past L1.
__device__ __forceinline__ TopkEntry far_entry(const TopkEntry* p) {
    TopkEntry e;
    e.idx = __ldcg(&p->idx);
    e.T = __ldcg(&p->T);
    e.nM = __ldcg(&p->nM);
    e.pad = 0;
    return e;
}

template <bool kWorklist>
__global__ void __launch_bounds__(kSelBlock) topk_select_kernel(TopkArgs a) {
    __shared__ Groups groups;
    __shared__ TopkEntry cand[kCandCap], fin[kFinalCap];
    __shared__ int ranks[kFinalCap];
    __shared__ TopkEntry lists[kSelWarps * kMaxTopK];
    __shared__ TopkEntry tmp[(kSelWarps / 2) * kMaxTopK];
    __shared__ int counts[kSelWarps], tmp_counts[kSelWarps / 2];
    __shared__ int n_cand, last_flag, first;
    await_previous();
    const int k = state_k(a.state);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t n = kWorklist ? min((int64_t)*a.wl_count, (int64_t)a.wl_cap) : a.n;
    const int ncta = (int)min((int64_t)gridDim.x, max((n + kPerCta - 1) / kPerCta, (int64_t)1));
    TopkEntry* bars = a.meet->bars();
    int32_t* posted = a.meet->posted(a.max_blocks);
    const bool posts = !kWorklist && ncta * k > kPostMin;
    if ((int)blockIdx.x >= ncta) return;
    const int held = min(max(a.state->count, 0), k);  // entries of the incoming state
    const bool full = held >= k;
    // entries that rank below the bar cannot enter the top-k
    TopkEntry bar = no_entry(0);
    bool have_bar = full;
    if (full) bar = state_entry(a.state, k - 1);
    // the running threshold of the call (a float lower bound, lowered by the
    // margin, on the k-th key of the candidates priced so far): an entry
    // whose key, computed the same way, falls below it has k entries of the
    // call that rank before it
    const float floor_key = a.thr ? __uint_as_float(__ldcg(a.thr)) : 0.0f;
    if (n <= 32) {
        // at most one entry per lane: warp 0 ranks them against each other
        // (the order is strict, so the ranks are distinct), places them,
        // and merges them with the state -- no CTA barrier
        if (warp != 0) return;
        TopkEntry e;
        e.idx = e.T = 0;
        e.nM = e.pad = 0;
        bool valid = lane < n && fetch<kWorklist>(a, lane, e);
        if (valid && full) valid = better(e, bar);
        const unsigned live = __ballot_sync(0xffffffffu, valid);
        int rank = 0;
        for (unsigned m = live; m; m &= m - 1) {
            const int j = __ffs(m) - 1;
            TopkEntry o;
            o.idx = __shfl_sync(0xffffffffu, e.idx, j);
            o.T = __shfl_sync(0xffffffffu, e.T, j);
            o.nM = __shfl_sync(0xffffffffu, e.nM, j);
            o.pad = 0;
            rank += better(o, e) ? 1 : 0;
        }
        const int nv = min(__popc(live), k);
        TopkEntry* mine = lists + kMaxTopK;
        if (valid && rank < k) mine[rank] = e;
        for (int i = lane; i < held; i += 32) lists[i] = state_entry(a.state, i);
        __syncwarp();
        const int total = warp_merge(lists, held, mine, nv, tmp, k);
        for (int i = lane; i < kMaxTopK; i += 32) {
            const bool on = i < total;
            a.state->idx[i] = on ? tmp[i].idx : -1;
            a.state->T[i] = on ? tmp[i].T : -1;
            a.state->nM[i] = on ? tmp[i].nM : 0;
        }
        if (lane == 0) {
            a.state->count = total;
            // the new k-th key, lowered by the margin (see TopkArgs::thr)
            if (a.thr && total >= k) atomicMax(a.thr, __float_as_uint(key_of(tmp[k - 1]) * kMargin));
        }
        return;
    }
    constexpr int U = 4;
    const int64_t step = (int64_t)ncta * kSelBlock;
    const int64_t start = (int64_t)blockIdx.x * kSelBlock;
    auto scan = [&](auto&& take) {
        for (int64_t base = start + warp * 32; base < n; base += step * U) {
            TopkEntry e[U];
            bool valid[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int64_t i = base + u * step + lane;
                valid[u] = false;
                e[u] = no_entry(0);
                if (i < n) valid[u] = fetch<kWorklist>(a, i, e[u]);
            }
#pragma unroll
            for (int u = 0; u < U; ++u)
                take(valid[u] && (floor_key <= 0.0f || key_of(e[u]) >= floor_key) &&
                         (!have_bar || !better(bar, e[u])),
                     e[u]);
        }
    };
    // ---- two passes: the CTA's bar, then the entries not below it; while the
    //      state is full its k-th entry stops almost every entry, and the
    //      first pass is left out unless the gather overflows
    int mine = 0;
    for (int attempt = full ? 1 : 0; attempt < 3; ++attempt) {
        if (attempt != 1) {
            TopkEntry best = no_entry(threadIdx.x);
            scan([&](bool want, const TopkEntry& e) {
                if (want && better(e, best)) best = e;
            });
            TopkEntry kth;
            if (cta_kth(best, k, groups, kth)) {
                bar = kth;
                have_bar = true;
                // it raises the call's threshold for the other CTAs
                if (threadIdx.x == 0 && a.thr) atomicMax(a.thr, __float_as_uint(key_of(kth) * kMargin));
                if (threadIdx.x == 0 && posts) {
                    bars[blockIdx.x] = kth;
                    store_release(posted + blockIdx.x, 1);
                }
            }
            if (attempt == 0) attempt = 1;
        }
        if (threadIdx.x == 0) n_cand = 0;
        __syncthreads();
        scan([&](bool want, const TopkEntry& e) { gather(cand, &n_cand, kCandCap, want, e); });
        __syncthreads();
        mine = n_cand;
        __syncthreads();
        if (mine <= kCandCap || !full) break;
    }
    if (mine > kCandCap) {  // uniform over the CTA
        int cnt = 0;
        scan([&](bool want, const TopkEntry& e) { warp_offer(lists + warp * kMaxTopK, cnt, k, want, e); });
        if (lane == 0) counts[warp] = cnt;
        cta_tree_merge(lists, counts, tmp, tmp_counts, kSelWarps, k);
        mine = counts[0];
        for (int p = threadIdx.x; p < mine; p += kSelBlock) cand[p] = lists[p];
        __syncthreads();
    }
    // ---- drop what falls below the best of the bars posted so far: in a sorted
    //      order, and among ties, every CTA gathers several times k entries,
    //      and most of them stop here instead of at the last CTA
    if (posts && mine > 0) {
        TopkEntry best = have_bar ? bar : no_entry(threadIdx.x);
        for (int i = threadIdx.x; i < ncta; i += kSelBlock)
            if (load_acquire(posted + i)) {
                const TopkEntry b = far_entry(bars + i);
                if (better(b, best)) best = b;
            }
        best = cta_best(best, tmp);
        if (best.idx <= INT64_MAX - kSelBlock) {
            bar = best;
            have_bar = true;
        }
        TopkEntry e = no_entry(0);
        bool want = (int)threadIdx.x < mine;
        if (want) e = cand[threadIdx.x];
        if (want) want = !better(best, e);
        if (threadIdx.x == 0) n_cand = 0;
        __syncthreads();
        gather(cand, &n_cand, kCandCap, want, e);
        __syncthreads();
        mine = n_cand;
    }
    // ---- hand over: the CTA reserves its places in the scratch list; the
    //      barrier gathers its stores, thread 0 fences them (fences are
    //      cumulative) before its ticket, and the CTA that draws the last one
    //      fences again before it reads the others' entries
    if (ncta > 1) {
        if (threadIdx.x == 0) first = mine ? atomicAdd(&a.meet->entries, mine) : 0;
        __syncthreads();
        for (int p = threadIdx.x; p < mine; p += kSelBlock) a.scratch[first + p] = cand[p];
        __syncthreads();
        if (threadIdx.x == 0) {
            __threadfence();
            const bool last = atomicAdd(&a.meet->tickets, 1) == ncta - 1;
            if (last) __threadfence();
            last_flag = last;
        }
        __syncthreads();
        if (!last_flag) return;
    }
    // ---- once more over the gathered entries and the state
    const int got = ncta > 1 ? __ldcg(&a.meet->entries) : mine;
    const int all = got + held;
    auto each = [&](auto&& take) {
        for (int base = warp * 32; base < all; base += kSelBlock * U) {
            TopkEntry e[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int i = base + u * kSelBlock + lane;
                e[u] = no_entry(0);
                if (i < got) e[u] = ncta > 1 ? far_entry(a.scratch + i) : cand[i];
                else if (i < all) e[u] = state_entry(a.state, i - got);
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const bool valid = base + u * kSelBlock + lane < all;
                take(valid && (!have_bar || !better(bar, e[u])), e[u]);
            }
        }
    };
    if (all > kDirect) {
        TopkEntry best = no_entry(threadIdx.x), kth;
        each([&](bool want, const TopkEntry& e) {
            if (want && better(e, best)) best = e;
        });
        if (cta_kth(best, k, groups, kth)) {
            bar = kth;
            have_bar = true;
        }
    }
    if (threadIdx.x == 0) n_cand = 0;
    __syncthreads();
    each([&](bool want, const TopkEntry& e) { gather(fin, &n_cand, kFinalCap, want, e); });
    __syncthreads();
    int m = n_cand;
    if (m > kFinalCap) {
        int cnt = 0;
        each([&](bool want, const TopkEntry& e) { warp_offer(lists + warp * kMaxTopK, cnt, k, want, e); });
        if (lane == 0) counts[warp] = cnt;
        cta_tree_merge(lists, counts, tmp, tmp_counts, kSelWarps, k);
        m = counts[0];
        for (int p = threadIdx.x; p < m; p += kSelBlock) fin[p] = lists[p];
    }
    // ---- exact ranks: warp w counts the entries of its eighth that rank
    //      before entry i (lane), 32 entries i at a time
    for (int p = threadIdx.x; p < m; p += kSelBlock) ranks[p] = 0;
    __syncthreads();
    const int part = (m + kSelWarps - 1) / kSelWarps;
    const int j0 = warp * part, j1 = min(m, j0 + part);
    for (int i = lane; i < m; i += 32) {
        const TopkEntry e = fin[i];
        int r = 0;
        for (int j = j0; j < j1; ++j) r += better(fin[j], e) ? 1 : 0;
        if (r) atomicAdd(&ranks[i], r);
    }
    __syncthreads();
    const int total = min(m, k);
    for (int p = threadIdx.x; p < m; p += kSelBlock) {
        const int r = ranks[p];
        if (r >= k) continue;
        const TopkEntry e = fin[p];
        a.state->idx[r] = e.idx;
        a.state->T[r] = e.T;
        a.state->nM[r] = e.nM;
        // the new k-th key, lowered by the margin (see TopkArgs::thr)
        if (a.thr && r == k - 1) atomicMax(a.thr, __float_as_uint(key_of(e) * kMargin));
    }
    for (int p = total + threadIdx.x; p < kMaxTopK; p += kSelBlock) {
        a.state->idx[p] = -1;
        a.state->T[p] = -1;
        a.state->nM[p] = 0;
    }
    if (threadIdx.x == 0) {
        a.state->count = total;
        if (ncta > 1) {  // every ticket is drawn: ready for the next launch
            a.meet->tickets = 0;
            a.meet->entries = 0;
        }
    }
    if (posts)
        for (int i = threadIdx.x; i < ncta; i += kSelBlock) posted[i] = 0;
}

template <bool kWorklist>
cudaError_t launch_select(const TopkArgs& a, int64_t n, int num_sms, cudaStream_t st, int64_t* launches) {
    if (n <= 0) return cudaSuccess;
    // two CTAs per SM: 3e5 results are one round of four loads a thread; the
    // survivors of a threshold are few after a call's first chunk, and a
    // small launch finds room sooner beside the next chunks' searches
    const int most = std::min(a.survivors ? 64 : 2 * num_sms, a.max_blocks);
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>((n + kPerCta - 1) / kPerCta, most));
    if (launches) *launches += 1;
    return launch_after(a.chained, topk_select_kernel<kWorklist>, grid, kSelBlock, 0, st, a);
}

__global__ void topk_reset_kernel(heddle_topk_state* s, int k) {
    for (int p = threadIdx.x; p < kMaxTopK; p += blockDim.x) {
        s->idx[p] = -1;
        s->T[p] = -1;
        s->nM[p] = 0;
    }
    if (threadIdx.x == 0) {
        s->k = k;
        s->count = 0;
    }
}

}  // namespace

cudaError_t launch_topk(const TopkArgs& a, int num_sms, cudaStream_t st, int64_t* launches) {
    return launch_select<false>(a, a.n, num_sms, st, launches);
}

cudaError_t launch_topk_worklist(const TopkArgs& a, int64_t n, int num_sms, cudaStream_t st,
                                 int64_t* launches) {
    return launch_select<true>(a, n, num_sms, st, launches);
}

cudaError_t launch_topk_reset(heddle_topk_state* state, int32_t k, cudaStream_t st) {
    topk_reset_kernel<<<1, 64, 0, st>>>(state, k);
    return cudaGetLastError();
}

}  // namespace hd
