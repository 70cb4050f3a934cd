// heddle_price.cu -- the screen kernel (decode + validate, §5.1 masks; DP
// degree, §5.3 packing; the memory screen of §5.2) and the dispatch of the
// search over its worklist.
//
// Two launches per chunk.  The screen kernel (one thread per candidate,
// coalesced) decodes and validates every candidate, computes its DP degree
// and decides memory feasibility from a table of the longest run of layers
// each (type, degree, in-flight count) can hold: if the runs of the stages
// sum below L no split fits (OOM); when every layer has the same state and
// activation bytes, runs summing to at least L (each at least one layer)
// also guarantee a split that fits, so no memory-only probe is needed.
// Candidates that still need PartitionLayers are compacted into a worklist,
// which one of the searches then prices: the equal-layer closed form
// (heddle_eqsearch.cu) when every layer costs the same, the paper's split
// rule in that mode (heddle_distribute.cu), else the general exact
// threshold search: one thread per entry (heddle_gsearch.cu), and one warp
// per entry for what that leaves (heddle_wsearch.cu).

#include <algorithm>
#include <mutex>

#include "heddle_tiled.cuh"

namespace hd {
namespace {

constexpr int kScreenBlock = 256;

// 1 / x to 1 ulp (infinity for zero)
__device__ __forceinline__ float rcp(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// A small count as float: its bits under 2^23's exponent, less 2^23 (two
// full-rate instructions; a conversion runs at a quarter of the rate).
__device__ __forceinline__ float small_float(uint32_t n) { return __uint_as_float(n | 0x4b000000u) - 8388608.0f; }

// min over the classes of (capacity + 1/2) / demand for one type, whose floor
// is min floor(capacity / demand): the exact ratio lies at least
// 1 / (2 demand) from a whole number, and capacities (at most 65,535) times
// the rounding of two operations (2^-22) stay below 1/2.  A class without
// demand gives infinity.
template <int kClasses>
__device__ __forceinline__ float type_ratio(uint32_t v, const float4& cap) {
    float r = cap.x * rcp(small_float(v & 0x1ffu));
    if (kClasses >= 2) r = fminf(r, cap.y * rcp(small_float((v >> 9) & 0xffu)));
    if (kClasses >= 1) r = fminf(r, cap.z * rcp(small_float((v >> 17) & 0x7fu)));
    return fminf(r, cap.w * rcp(small_float(v >> 24)));
}

template <int kClasses>
__device__ __forceinline__ float min_ratio(const uint32_t* dem, const float4* cap, int NT) {
    float r = __int_as_float(0x7f800000);
    for (int g0 = 0; g0 < NT; g0 += 4)  // types past NT hold no demand
#pragma unroll
        for (int g = g0; g < g0 + 4; ++g) r = fminf(r, type_ratio<kClasses>(dem[g * kScreenBlock], cap[g]));
    return r;
}

__device__ __forceinline__ void copy_async16(void* to, const void* from) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(to)), "l"(from)
                 : "memory");
}

constexpr int kRow = kScreenBlock + 16;  // bytes of a tile row: 256 candidates and a block's offset

// Steps 1-2 and the memory screen for every candidate of the batch.  Each
// CTA takes 256 consecutive candidates at a time: their code planes are
// copied to shared memory while their S and M arrive, the candidates are
// counting-sorted by S, and thread i screens the i-th of that order, so the
// lanes of a warp run stage loops of nearly equal length.
//
// The planes are copied in aligned blocks of 16 bytes.  A plane stride that
// is no multiple of 16 (any batch of odd size) puts plane s of the slice at
// its own offset, (code + s stride + c0) mod 16, in a row of 272 bytes; only a
// block that reaches past the arrays is read byte by byte.  (999,983
// candidates, byte copies after the sort: 55.9 us on the 80-layer workload,
// 53.6 on the largest, 33.5 on the expert one; these: 52.7, 50.0 and 30.3;
// with the rows written as below: 50.3, 50.1 and 29.2.)
//
// Instructions bound it (and the search that overlaps it), so the tables are
// kept in the form in which a stage adds them up: one word that adds the
// stage to every class of its type's demand, one run length that marks "no
// layer fits" in its size; the DP degree is one minimum of float ratios over
// the classes that can decide on this cluster.  1e6 candidates of the largest
// workload: 33.3M warp instructions and 50 us alone (40.0M and 65 with tables
// built by every CTA, integer quotients and rejections written in sorted order);
// of the 80-layer one 50 us (61), of the expert one 29 (39).
__global__ void __launch_bounds__(kScreenBlock) screen_kernel(PriceArgs a) {
    __shared__ ScreenTabs tab;
    __shared__ uint32_t dem[8 * kScreenBlock];  // per-thread demand word (see stage_desc), per type
    __shared__ __align__(16) uint8_t tile[kMaxStages * kRow];  // [stage][candidate of the slice, past its offset]
    __shared__ uint8_t sS[kScreenBlock];
    __shared__ uint16_t sM[kScreenBlock];
    __shared__ uint8_t order[kScreenBlock];
    __shared__ uint16_t sn[kScreenBlock];  // OOM: the DP degree
    __shared__ uint8_t sstatus[kScreenBlock];
    __shared__ uint16_t sel[kScreenBlock];  // per warp: the candidates taken and their depths
    __shared__ int bins[kMaxStages + 3];
    const Layout& y = a.lay;
    const int L = y.L;
    allow_dependents();
    {
        const uint4* from = reinterpret_cast<const uint4*>(a.img + y.offScreen);
        uint4* to = reinterpret_cast<uint4*>(&tab);
        for (int i = threadIdx.x; i < (int)(sizeof(ScreenTabs) / 16); i += kScreenBlock) to[i] = __ldg(from + i);
    }
    const bool memuni = reinterpret_cast<const ModelInfo*>(a.img + y.offModel)->mem_uniform != 0;
    const int s_lim = min(min(kMaxStages, a.s_max), L);
    const uint8_t* code_end = a.code + (int64_t)(a.s_max - 1) * a.stride + a.n;
    const int skew = (int)(a.stride & 15);  // each plane's offset against the one before
    uint32_t* mydem = dem + threadIdx.x;
    const int lane = threadIdx.x & 31;
    for (int64_t c0 = (int64_t)blockIdx.x * kScreenBlock; c0 < a.n; c0 += (int64_t)gridDim.x * kScreenBlock) {
        const int nloc = (int)min((int64_t)kScreenBlock, a.n - c0);
        // ---- code planes of the slice into the tile
        const int off0 = (int)(reinterpret_cast<uintptr_t>(a.code + c0) & 15);
        for (int i = threadIdx.x; i < s_lim * (kRow / 16); i += kScreenBlock) {
            const int s = i / (kRow / 16), o = (i % (kRow / 16)) * 16;
            const uint8_t* from = a.code + (int64_t)s * a.stride + c0 + o - ((off0 + s * skew) & 15);
            uint8_t* to = tile + s * kRow + o;
            if (from >= a.code && from + 16 <= code_end) {
                copy_async16(to, from);
            } else {
                for (int b = 0; b < 16; ++b)
                    if (from + b >= a.code && from + b < code_end) to[b] = __ldg(from + b);
            }
        }
        // ---- S and M of the slice; S = 0 marks a depth or M outside range,
        //      bin kMaxStages + 1 the padding past the batch
        int key = kMaxStages + 1;
        if (threadIdx.x < nloc) {
            const int S = a.S[c0 + threadIdx.x];
            // at micro-batch size 2^shift a replica runs M / 2^shift
            // micro-batches; a size that does not divide M is not priced
            const int Mraw = a.M[c0 + threadIdx.x];
            const int M = Mraw >> a.mbs_shift;
            const bool whole = (Mraw & ((1 << a.mbs_shift) - 1)) == 0;
            key = (S >= 1 && S <= s_lim && M >= 1 && whole) ? S : 0;
            // a plan's template that the plan cannot reach is priced SKIPPED
            // (bit 7 of its S byte; it sorts with the invalid ones)
            const bool skipped =
                a.n_tmpl && !(min((int)a.n_tmpl[c0 + threadIdx.x], a.plan_slots) > a.plan_slot &&
                              (!a.prev_status || a.prev_status[c0 + threadIdx.x] == HEDDLE_CAND_OK));
            if (skipped) key = 0;
            sS[threadIdx.x] = (uint8_t)(key | (skipped ? 0x80 : 0));
            sM[threadIdx.x] = (uint16_t)M;
        }
        if (threadIdx.x < kMaxStages + 3) bins[threadIdx.x] = 0;
        __syncthreads();
        atomicAdd(&bins[key], 1);
        __syncthreads();
        if (threadIdx.x < 32) {
            // exclusive scan of bins 0..33 by one warp (lane l: bin l, lane
            // 31 also bins 32 and 33)
            const int v = bins[lane];
            int x = v;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y2 = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o) x += y2;
            }
            const int b32 = bins[32], b33 = bins[33];
            __syncwarp();
            bins[lane] = x - v;
            if (lane == 31) {
                bins[32] = x;
                bins[33] = x + b32;
            }
            (void)b33;
        }
        __syncthreads();
        order[atomicAdd(&bins[key], 1)] = (uint8_t)threadIdx.x;
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
        const int ci = order[threadIdx.x];
        const bool live = threadIdx.x < nloc;  // padding sorts last
        const int64_t c = c0 + ci;
        int S = 0, M = 0, status = HEDDLE_CAND_INVALID;
        int n = 0;
        if (live) {
            S = sS[ci] & 0x3f;
            M = sM[ci];
            if (sS[ci] & 0x80) status = HEDDLE_CAND_SKIPPED;
            if (S > 0) {
#pragma unroll
                for (int g = 0; g < 8; ++g) mydem[g * kScreenBlock] = 0;
                uint32_t bad = 0;
                int run_sum = 0;
                const uint8_t* col = tile + ci;
                int off = off0;
                const int f_lim = min(M, kMaxStages) * 32;
                int f = S * 32;
#pragma unroll 4
                for (int s = 0; s < S; ++s) {
                    const int b = col[s * kRow + (off & 15)];
                    off += skew;
                    const uint32_t d = tab.desc[b];
                    bad |= d;
                    mydem[(b & 7) * kScreenBlock] += d;
                    run_sum += tab.run[min(f, f_lim) + b];
                    f -= 32;
                }
                if (!(bad >> 31)) {
                    const int cls = tab.classes;
                    n = (int)(cls == 0   ? min_ratio<0>(mydem, tab.cap, y.NT)
                              : cls == 1 ? min_ratio<1>(mydem, tab.cap, y.NT)
                                         : min_ratio<2>(mydem, tab.cap, y.NT));
                    status = n == 0                                  ? HEDDLE_CAND_NO_FIT
                             : run_sum >= kNoRun || run_sum < L ? HEDDLE_CAND_OOM
                                                                     : HEDDLE_CAND_OK;
                }
            }
            sstatus[ci] = (uint8_t)status;
            sn[ci] = (uint16_t)(status == HEDDLE_CAND_OOM ? n : 0);
        }
        // compact the candidates that need the search (one atomic per warp)
        const bool take = live && status == HEDDLE_CAND_OK;
        const unsigned mask = __ballot_sync(0xffffffffu, take);
        if (mask) {
            int base = 0;
            if (lane == 0) base = atomicAdd(a.wl_count, __popc(mask));
            base = __shfl_sync(0xffffffffu, base, 0);
            const int p = base + __popc(mask & ((1u << lane) - 1));
            if (take) {
                if (p < a.wl_cap) {
                    a.wl_idx[p] = (int32_t)c;
                    a.wl_n[p] = (uint16_t)n;
                    a.wl_M[p] = (uint16_t)M;
                    a.wl_S[p] = (uint8_t)S;
                    a.wl_memok[p] = memuni ? 1 : 0;
                } else {
                    atomicOr(a.err, kErrInternal);
                }
            }
            // the entry in its depth's bucket, for the searches' order by
            // decreasing depth
            if (take) {
                const unsigned same = __match_any_sync(mask, S);
                const int leader = __ffs(same) - 1;
                int b0 = 0;
                if (lane == leader) b0 = atomicAdd(a.wl_count + 1 + S, __popc(same));
                const int bpos = __shfl_sync(same, b0, leader) + __popc(same & ((1u << lane) - 1));
                if (p < a.wl_cap && bpos < a.wl_cap) a.wl_bucket[(int64_t)(S - 1) * a.wl_cap + bpos] = p;
            }
            // the taken candidates' rows of 32 stage bytes (zero past S): a
            // word a lane, four lanes a row and eight rows at once while no
            // candidate of the warp is deeper than 16, else eight lanes a row
            // (1e6 candidates of up to 8 stages, nine tenths taken: a row a
            // warp store 66.9 us, so 57.2; of up to 16 stages, a third to two
            // thirds taken: 53.1 and 65.3 -> 50.3 and 57.6; two lanes a row
            // where they do: 56.8 with part of a row unwritten, 66.3 with the
            // rest zeroed; always eight: 58.9)
            uint16_t* mine = sel + (threadIdx.x & ~31);
            if (take) mine[__popc(mask & ((1u << lane) - 1))] = (uint16_t)(ci | (S << 8));
            __syncwarp();
            const int lw = __any_sync(0xffffffffu, take && S > 16) ? 3 : 2;
            const int s0 = 4 * (lane & ((1 << lw) - 1));  // this lane's first stage
            const uint8_t* planes = tile + s0 * kRow;
            const int o0 = (off0 + s0 * skew) & 15, o1 = (off0 + (s0 + 1) * skew) & 15,
                      o2 = (off0 + (s0 + 2) * skew) & 15, o3 = (off0 + (s0 + 3) * skew) & 15;
            const int taken = __popc(mask);
            for (int k = lane >> lw; k < taken; k += 32 >> lw) {
                if (base + k >= a.wl_cap) continue;
                const int from = mine[k], left = (from >> 8) - s0;  // stages from s0 on
                const uint8_t* at = planes + (from & 0xff);
                uint32_t word = 0;
                if (left > 0) word = at[o0];
                if (left > 1) word |= (uint32_t)at[kRow + o1] << 8;
                if (left > 2) word |= (uint32_t)at[2 * kRow + o2] << 16;
                if (left > 3) word |= (uint32_t)at[3 * kRow + o3] << 24;
                uint32_t* out = reinterpret_cast<uint32_t*>(a.wl_code + (int64_t)(base + k) * kMaxStages + s0);
                *out = word;
                if (lw == 2) out[4] = 0;  // stages 16 on
            }
        }
        __syncthreads();  // the tile, S, M and order are reused by the next slice
        // the rejected candidates' results, in candidate order (coalesced;
        // sn and sstatus are next written three barriers on)
        if (threadIdx.x < nloc && sstatus[threadIdx.x] != HEDDLE_CAND_OK) {
            const int64_t r = c0 + threadIdx.x;
            a.T[r] = -1;
            a.B[r] = -1;
            a.ndp[r] = sn[threadIdx.x];
            a.status[r] = sstatus[threadIdx.x];
            if (a.bounds && !a.bounds_scratch)
                for (int s = 0; s <= kMaxStages; ++s) a.bounds[(int64_t)s * a.bstride + r] = 0;
        }
    }
}

}  // namespace

// The general search: one thread per entry (heddle_gsearch.cu), then one warp
// per entry it left (heddle_wsearch.cu).
cudaError_t launch_thread_search(const PriceArgs& a, int num_sms, cudaStream_t st);
cudaError_t launch_warp_search(const PriceArgs& a, int num_sms, cudaStream_t st, bool listed);

cudaError_t launch_screen(const PriceArgs& a, int num_sms, cudaStream_t st, cudaEvent_t mid, int64_t* launches) {
    if (a.n <= 0) return cudaSuccess;
    if (a.n > a.wl_cap) return cudaErrorInvalidValue;
    cudaError_t e = cudaMemsetAsync(a.wl_count, 0, sizeof(int32_t) * a.wl_clear, st);
    if (e != cudaSuccess) return e;
    // one wave of resident CTAs, each looping over slices
    int screen_per_sm = 0;
    e = resident_blocks(reinterpret_cast<const void*>(&screen_kernel), kScreenBlock, 0, &screen_per_sm);
    if (e != cudaSuccess) return e;
    // (six of the eight CTAs that fit an SM beside other chunks' searches:
    // 1e7 candidates of the largest workload 668 -> 645 us; five 650, four 653)
    const int most = std::max(a.beside ? std::min(screen_per_sm, 6) : screen_per_sm, 1);
    const int grid = (int)std::min<int64_t>((a.n + kScreenBlock - 1) / kScreenBlock, (int64_t)num_sms * most);
    screen_kernel<<<grid, kScreenBlock, 0, st>>>(a);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if (launches) launches[0] += 1;
    if (mid && (e = cudaEventRecord(mid, st)) != cudaSuccess) return e;
    return cudaSuccess;
}

cudaError_t resident_blocks(const void* func, int block, size_t smem, int* per_sm) {
    struct Limit {  // the largest dynamic shared memory a kernel was allowed so far
        const void* func;
        int device;
        size_t smem;
    };
    struct Answer {
        const void* func;
        int device, block;
        size_t smem;
        int per_sm;
    };
    static std::mutex mu;
    static Limit limits[32];
    static Answer answers[128];
    static int n_limits = 0, n_answers = 0;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lock(mu);
    for (int i = 0; i < n_answers; ++i) {
        const Answer& x = answers[i];
        if (x.func == func && x.device == dev && x.block == block && x.smem == smem) {
            *per_sm = x.per_sm;
            return cudaSuccess;
        }
    }
    // raise (never lower) the kernel's limit: cached launches of larger
    // sizes rely on it.  Past the tables' capacity nothing is cached and
    // the limit is set on every call.
    int li = -1;
    for (int i = 0; i < n_limits; ++i)
        if (limits[i].func == func && limits[i].device == dev) li = i;
    if (li < 0 && n_limits < 32) {
        li = n_limits++;
        limits[li] = Limit{func, dev, 0};
    }
    if (li < 0 || limits[li].smem < smem) {
        e = cudaFuncSetAttribute(func, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        if (li >= 0) limits[li].smem = smem;
    }
    int v = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, func, block, smem);
    if (e != cudaSuccess) return e;
    if (li >= 0 && n_answers < 128) answers[n_answers++] = Answer{func, dev, block, smem, v};
    *per_sm = v;
    return cudaSuccess;
}

cudaError_t launch_price(const PriceArgs& a, int num_sms, cudaStream_t st, cudaEvent_t mid, int64_t* launches) {
    if (a.n <= 0) return cudaSuccess;
    cudaError_t e = launch_screen(a, num_sms, st, mid, launches);
    if (e != cudaSuccess) return e;
    if (launches) launches[1] += 1;
    if (a.split_mode) return launch_distribute(a, num_sms, st);
    if (a.uniform) return launch_eq_search(a, num_sms, st);
    // a batch smaller than the thread search's threshold cannot fill its
    // buckets up to it: that kernel would return at once, so it is not launched
    if (a.n >= a.thread_min && (e = launch_thread_search(a, num_sms, st)) != cudaSuccess) return e;
    return launch_warp_search(a, num_sms, st, true);
}

}  // namespace hd
