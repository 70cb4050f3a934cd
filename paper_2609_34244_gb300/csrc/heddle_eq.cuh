// heddle_eq.cuh -- pieces shared by the two searches that run one thread per
// worklist entry on a model whose layers all cost the same: the min-max
// search (heddle_eqsearch.cu) and the paper's split rule
// (heddle_distribute.cu).
#pragma once

#include <cstddef>

#include "heddle_internal.cuh"

namespace hd {
namespace {

constexpr int kEqBlock = 128;
constexpr int kEqWarps = kEqBlock / 32;

struct EqShared {
    EqTabs tab;
    uint16_t run[32 * 33 + 256];  // ScreenTabs::run
    uint32_t sw[kMaxStages * kEqBlock];  // stage words, [s][thread]
};

// Stage word: bits 0-4 cost index (the stage byte's type | degree bits),
// bits 5-12 P2P index, bits 13-20 memory run m, bits 21-28 the cap.
constexpr int kCapShift = 21;
constexpr uint32_t kNoCap = 0x1fffffu;

__device__ __forceinline__ int cap_of(uint32_t w) { return (int)(w >> kCapShift) & 255; }
__device__ __forceinline__ int run_of(uint32_t w) { return (int)(w >> 13) & 255; }
__device__ __forceinline__ int p2p_of(uint32_t w) { return (int)(w >> 5) & 255; }
// a count below 2^23 as float (two full-rate instructions)
__device__ __forceinline__ float count_float(uint32_t n) { return __uint_as_float(n | 0x4b000000u) - 8388608.0f; }

// The tables, as the image holds them (the caller synchronises the CTA).
__device__ __forceinline__ void load_eq_tables(const PriceArgs& a, EqTabs& tab, uint16_t (&run)[32 * 33 + 256]) {
    const uint4* from = reinterpret_cast<const uint4*>(a.img + a.lay.offEq);
    uint4* to = reinterpret_cast<uint4*>(&tab);
    for (int i = threadIdx.x; i < (int)(sizeof(EqTabs) / 16); i += kEqBlock) to[i] = __ldg(from + i);
    const uint4* from2 = reinterpret_cast<const uint4*>(a.img + a.lay.offScreen + offsetof(ScreenTabs, run));
    uint4* to2 = reinterpret_cast<uint4*>(run);
    static_assert(sizeof(run) % 16 == 0 && offsetof(ScreenTabs, run) % 16 == 0, "copied 16 bytes at a time");
    for (int i = threadIdx.x; i < (int)(sizeof(run) / 16); i += kEqBlock) to2[i] = __ldg(from2 + i);
}

// end_of[S] = bucketed entries of depths >= S: an inclusive scan of depths
// 32 .. 1 in lanes 0 .. 31 of the first warp.
__device__ __forceinline__ void depth_ends(const int32_t* wl_count, int* end_of) {
    if (threadIdx.x >= 32) return;
    const int lane = threadIdx.x;
    int x = wl_count[1 + (kMaxStages - lane)];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y2 = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y2;
    }
    end_of[kMaxStages - lane] = x;
    if (lane == 0) end_of[kMaxStages + 1] = 0;
}

// Entry g of the buckets read in order of decreasing depth.
__device__ __forceinline__ bool deepest_first(const PriceArgs& a, const int* end_of, int64_t g, int64_t entries,
                                              int64_t& p) {
    // its depth: the largest S with end_of[S] > g (end_of falls with S)
    int lo = 1, hi = kMaxStages;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (end_of[mid] > g) lo = mid; else hi = mid - 1;
    }
    const int64_t off = g - end_of[lo + 1];
    if (!in_range(off, end_of[lo] - end_of[lo + 1], a.err)) return false;
    p = a.wl_bucket[(int64_t)(lo - 1) * a.wl_cap + off];
    return in_range(p, entries, a.err);
}

// f(s, stage byte, P2P index, memory run) for the stages of entry p.
template <class F>
__device__ __forceinline__ void for_stages(const PriceArgs& a, const EqTabs& t, const uint16_t* run, int64_t p, int S,
                                           int M, F f) {
    // the entry's row of stage bytes (zero past S), 16 at a time (ordinary
    // loads: the screen may have written it while this kernel already ran)
    uint32_t cw4[8];
    {
        const uint4* row = reinterpret_cast<const uint4*>(a.wl_code + p * kMaxStages);
        const uint4 v0 = row[0];
        const uint4 v1 = S > 16 ? row[1] : make_uint4(0, 0, 0, 0);
        cw4[0] = v0.x; cw4[1] = v0.y; cw4[2] = v0.z; cw4[3] = v0.w;
        cw4[4] = v1.x; cw4[5] = v1.y; cw4[6] = v1.z; cw4[7] = v1.w;
    }
    const int f_lim = min(M, kMaxStages) * 32;
    int fl = S * 32;
#pragma unroll
    for (int s = 0; s < kMaxStages; ++s) {
        if (s >= S) break;
        const int code = (cw4[s >> 2] >> ((s & 3) * 8)) & 0x1f;
        const int next = s + 1 < kMaxStages ? (cw4[(s + 1) >> 2] >> (((s + 1) & 3) * 8)) & 0x1f : 0;
        f(s, code, (int)t.pair[(s + 1 == S ? 32 : next) * 32 + code], (uint32_t)run[min(fl, f_lim) + code]);
        fl -= 32;
    }
}

// The stage with the largest G_s / (k_s bw_s): with equal gradient bytes per
// layer that is the largest layers / D, found in float (three roundings,
// 2^-22) and compared exactly (layers < 2^8 times D < 2^43) where two come
// within 2^-20 of each other.
struct GradMax {
    uint64_t G = 0, D = 1;
    float f = -1.f;

    // the stage [at, nxt); pbytes: gradient bytes of every layer when they
    // are all equal, else -1 (PB: their prefix)
    __device__ __forceinline__ void add(const EqTabs& t, const int64_t* PB, int64_t pbytes, int code, int at,
                                        int nxt) {
        constexpr float kNear = 1.0f / 1048576.0f;
        if (pbytes >= 0) {
            const uint64_t len = (uint64_t)(nxt - at);
            const float x = count_float((uint32_t)len) * t.rD[code];
            if (x > f * (1.0f - kNear)) {
                const uint64_t d = t.D[code];
                if (x > f * (1.0f + kNear) || len * D > G * d) {
                    f = x;
                    G = len;
                    D = d;
                }
            }
        } else {
            const uint64_t g = (uint64_t)(PB[nxt] - PB[at]), d = t.D[code];
            if (f < 0.f || (u128)g * D > (u128)G * d) {
                f = 0.f;
                G = g;
                D = d;
            }
        }
    }

    // ring all-reduce over n > 1 replicas: ceil(2(n-1) G 1e9 / (n k bw))
    // (G < 2^50 and bandwidths < 2^40 keep n k bw below 2^64)
    __device__ __forceinline__ int64_t sync_ns(int64_t n, int64_t pbytes, uint32_t* err) const {
        const uint64_t bytes = pbytes >= 0 ? G * (uint64_t)pbytes : G;
        const u128 num = (u128)(2 * (uint64_t)(n - 1) * 1000000000ull) * bytes;
        bool ok = true;
        const int64_t ns = (int64_t)ceil_div_u128(num, (uint64_t)n * D, &ok);
        if (!ok) atomicOr(err, kErrInternal);
        return ns;
    }
};

}  // namespace
}  // namespace hd
