// heddle_internal.cuh -- definitions shared by the library's translation
// units (never installed, never included by the oracle).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <utility>

#include "heddle.h"

namespace hd {

constexpr int kMaxTypes = HEDDLE_MAX_TYPES;
constexpr int kMaxStages = HEDDLE_MAX_STAGES;
static_assert(kMaxStages == 32, "the searches hold one stage (or one depth) per lane");
constexpr int kMaxLayers = HEDDLE_MAX_LAYERS;
constexpr int kMaxTopK = HEDDLE_MAX_TOPK;
constexpr int64_t kInf = INT64_MAX;

typedef unsigned __int128 u128;

// Device error flags (heddle_device_errors).
constexpr uint32_t kErrStageWait = 1u;
constexpr uint32_t kErrSearchBound = 2u;
constexpr uint32_t kErrInternal = 4u;
constexpr uint32_t kErrBounds = 8u;  // a bounds check of the checked build failed

// The bounds-checked build (HEDDLE_CHECKED) tests the data-dependent
// indices -- worklist entries, candidate indices, table rows -- before it
// uses them; a failed test raises kErrBounds and the access is skipped (no
// trap, no out-of-range access).  The product build compiles the tests away.
#ifdef HEDDLE_CHECKED
constexpr bool kChecked = true;
#else
constexpr bool kChecked = false;
#endif
__device__ __forceinline__ bool in_range(int64_t i, int64_t n, uint32_t* err) {
    if (!kChecked) return true;
    if (i >= 0 && i < n) return true;
    atomicOr(err, kErrBounds);
    return false;
}
// Table-build flags (checked by the host at load time).
constexpr uint32_t kTabBadValue = 1u;   // non-finite or negative per-layer cost
constexpr uint32_t kTabTooLarge = 2u;   // a table total or P2P term above its limit

// What the screen looks up per stage byte and per type, in the form in which
// it adds it up (see screen_kernel); one 16-byte-aligned section of the image.
struct ScreenTabs {
    float4 cap[kMaxTypes];      // capacity of class e in units of 2^e, plus 1/2
    uint32_t desc[256];         // per stage byte: bit 31 inadmissible, else its demand per class
    uint16_t run[32 * 33 + 256];  // [f * 32 + byte] the longest run of layers, kNoRun for none
                                // (bytes above 31 are inadmissible and read on)
    int32_t classes;            // 0: classes 0 and 3 decide, 1: 0, 2 and 3, 2: all four
    int32_t pad[3];
};
static_assert(sizeof(ScreenTabs) % 16 == 0, "copied 16 bytes at a time");
constexpr int kNoRun = 8192;  // above 32 runs of 255 layers
// first bit of class e in a type's demand word (9, 8, 7 and 6 bits)
__host__ __device__ constexpr int demand_shift(int e) { return e == 0 ? 0 : e == 1 ? 9 : e == 2 ? 17 : 24; }

// What the equal-layer search looks up per stage: by stage byte (type and
// degree, 0 .. 31), by P2P index (kZeroP2P: no next stage) and by pair of
// consecutive stage bytes.
constexpr int kZeroP2P = 128;  // a zero entry after the 8 x 8 x 2 P2P table
struct EqTabs {
    int64_t q[32];          // one layer's time
    int64_t p2p[130];       // P2P per index
    uint64_t D[32];         // slowest NIC times degree
    float rq[32];           // 1 / q (0 for a free layer)
    float qf[32];
    float cf[132];
    float rD[32];           // 1 / D
    uint8_t pair[33 * 32];  // [next byte, 32: none][byte] P2P index
};
static_assert(sizeof(EqTabs) % 16 == 0, "copied 16 bytes at a time");

// CTAs of the table build: one per (type, degree), one per type, one more.
__host__ __device__ constexpr int table_ctas(int NT) { return 4 * NT + kMaxTypes + 1; }

// What the build found out about the model; the host reads it back.
struct ModelInfo {
    int32_t mem_uniform;   // every layer has the same state and activation bytes
    int32_t grad_uniform;  // every layer has the same gradient bytes
    int32_t row_uniform[4 * kMaxTypes];  // every layer costs the same on this (type, degree)
    uint32_t flags[table_ctas(kMaxTypes)];  // kTab* per CTA
};

// Byte layout of the cost-table image.  The search kernels copy its first
// searchBytes into shared memory with bulk (TMA) copies, so every section
// starts on a 16-byte boundary and the totals are multiples of 16.
struct Layout {
    int32_t L, NT;
    uint32_t offP;      // int64 [NT][4][L+1]   prefix of per-layer ns per (type, degree)
    uint32_t offSA;     // int64x2 [L+1]         prefix of (state bytes, activation bytes)
    uint32_t offPB;     // int64 [L+1]           prefix of gradient bytes
    uint32_t offP2P;    // int64 [8][8][2]       P2P ns (from, to, same-node)
    uint32_t offMem;    // int64 [8]             memory per GPU
    uint32_t offInter;  // int64 [8]             slowest NIC of the type
    uint32_t offMaxN;   // int32 [8]             largest node of the type
    uint32_t offPow2;   // int32 [8]             largest power of two <= largest node (<= 8)
    uint32_t offGpus;   // int32 [8]             GPUs of the type
    uint32_t offWin;    // uint8 [8][4][33]      longest run of layers that fits memory per
                        //                       (type, degree, in-flight microbatches f)
    uint32_t offModel;  // ModelInfo
    uint32_t searchBytes;
    uint32_t offScreen; // ScreenTabs
    uint32_t offEq;     // EqTabs (of the first layer's costs)
    uint32_t bytes;
};

inline uint32_t align16(uint32_t x) { return (x + 15u) & ~15u; }

inline Layout make_layout(int L, int NT) {
    Layout y{};
    y.L = L;
    y.NT = NT;
    uint32_t o = 0;
    y.offP = o;     o = align16(o + 8u * NT * 4 * (L + 1));
    y.offSA = o;    o = align16(o + 16u * (L + 1));
    y.offPB = o;    o = align16(o + 8u * (L + 1));
    y.offP2P = o;   o = align16(o + 8u * 8 * 8 * 2);
    y.offMem = o;   o = align16(o + 8u * 8);
    y.offInter = o; o = align16(o + 8u * 8);
    y.offMaxN = o;  o = align16(o + 4u * 8);
    y.offPow2 = o;  o = align16(o + 4u * 8);
    y.offGpus = o;  o = align16(o + 4u * 8);
    y.offWin = o;   o = align16(o + 8u * 4 * 33);
    y.offModel = o; o = align16(o + (uint32_t)sizeof(ModelInfo));
    y.searchBytes = o;
    y.offScreen = o; o = align16(o + (uint32_t)sizeof(ScreenTabs));
    y.offEq = o;    o = align16(o + (uint32_t)sizeof(EqTabs));
    y.bytes = o;
    return y;
}

struct TopkEntry {
    int64_t idx;
    int64_t T;
    uint32_t nM;
    uint32_t pad;
};

struct TableArgs {
    Layout lay;
    const heddle_gpu_type* types;
    const heddle_node* nodes;
    int32_t n_nodes;
    const heddle_layer* layers;
    const double* profile;   // nullable
    int64_t boundary_bytes;
    int32_t moe;
    unsigned char* img;      // out
    int64_t* q;              // out [NT][4][L]
};
cudaError_t launch_tables(const TableArgs& a, cudaStream_t st);

// Blocks of `func` (a kernel) resident per SM at `block` threads and `smem`
// bytes of dynamic shared memory, after raising the kernel's dynamic
// shared-memory limit to smem.  The answer is cached per (kernel, block,
// smem, device): the two runtime queries cost microseconds of host time,
// which a small pricing call would otherwise pay on every launch.
cudaError_t resident_blocks(const void* func, int block, size_t smem, int* per_sm);

// Programmatic dependent launch: a kernel launched by launch_after may start
// while the previous kernel of its stream still runs, once every CTA of that
// one has called allow_dependents (or exited); await_previous returns when
// the previous kernel has completed and its writes are visible (at once when
// the kernel was launched the ordinary way).  What the previous kernels write
// is read by ordinary loads only: the wait does not order the read-only path
// (__ldg).  A call of one chunk chains its
// kernels so: with a thousand candidates each runs for little longer than a
// launch takes.
__device__ __forceinline__ void allow_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void await_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <class... P, class... A>
cudaError_t launch_after(bool chained, void (*kernel)(P...), int grid, int block, size_t smem, cudaStream_t st,
                         A&&... args) {
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = chained ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...);
}

struct PriceArgs {
    Layout lay;
    const unsigned char* img;
    int32_t moe;
    const uint8_t* S;
    const uint16_t* M;
    const uint8_t* code;
    // one template slot of a plan batch (n_tmpl nullable: none): a candidate is
    // priced SKIPPED unless its plan reaches the slot on its templates' own
    // prices -- it has more than plan_slot templates and, past the first
    // slot, the previous one's status is OK (a SKIPPED one is not)
    const uint8_t* n_tmpl;
    int32_t plan_slots, plan_slot;
    const uint8_t* prev_status;  // nullable: the first slot
    int32_t bounds_scratch;      // only the planes 0 .. S of OK candidates are read: the others stay as they are
    int64_t n;
    int64_t stride;
    int32_t s_max;
    int64_t* T;
    int64_t* B;
    uint16_t* ndp;
    uint8_t* status;
    uint8_t* bounds;
    int64_t bstride;  // plane stride of bounds (>= n)
    uint32_t* err;
    unsigned long long* counters;  // non-null selects the counting variant
    // worklist of the candidates that need the threshold search (device
    // scratch owned by the context, capacity wl_cap candidates)
    int32_t* wl_count;   // [kWlMeta]: entries, the general list, per depth S the entries
                         // of that depth, two take counters, survivors (cleared per chunk)
    int32_t* wl_idx;
    uint16_t* wl_n;
    uint16_t* wl_M;
    uint8_t* wl_S;
    uint8_t* wl_memok;   // 1: memory feasibility already decided by the screen
    uint8_t* wl_code;    // [wl_cap][kMaxStages] stage bytes, a 32-byte row per entry (zero past S)
    int32_t* wl_bucket;  // [kMaxStages][wl_cap]: per depth S (row S - 1) the entries of
                         // that depth, in any order (equal-layer search)
    int32_t wl_cap;
    int32_t wl_clear;    // ints of wl_count the screen's launch clears (kWlMeta, or one more with the threshold)
    int32_t beside;      // other chunks are searched meanwhile
    int32_t chained;     // the search may start while the screen still runs (see launch_after)
    int32_t uniform;     // search with the equal-layer closed form (model flags [0] and [1])
    int32_t mbs_shift;   // micro-batch size 2^shift: M >> shift micro-batches (invalid unless 2^shift | M)
    int32_t equal_layers;  // every layer has the same time per (type, degree) and the same memory
    int32_t split_mode;  // 1: the paper's own split rule (distribute_kernel) instead of PartitionLayers
    int32_t thread_min;  // general search: the bucketed entries below which only the warp search runs
    int32_t split_min, split_per_stage;  // split rule of equal layers: see split_by_threads
    // per worklist entry, written by the search: T (-1 unless OK) and n * M,
    // so a top-k can run over the searched candidates only
    int64_t* wl_T;
    uint32_t* wl_nM;
    // survivors of the top-k threshold (equal-layer search inside a top-k
    // pricing; sv_count null otherwise): OK entries whose n*M / T, in
    // float, is at least the float threshold *thr are appended as (chunk
    // index, T, n*M).  *thr never exceeds the running top-k's k-th key
    // (see TopkArgs::thr), so no entry that can enter the top-k is left out.
    int32_t* sv_count;
    int32_t* sv_idx;
    int64_t* sv_T;
    uint32_t* sv_nM;
    uint32_t* thr;
    const int32_t* topk_k;  // the state's k (device)
};
// Prices candidates [0, a.n) with a.n <= a.wl_cap: screen, then search.
// `mid` (nullable) is recorded on st between the two; `launches` (nullable)
// gains the kernels launched: [0] screen, [1] search.
cudaError_t launch_price(const PriceArgs& a, int num_sms, cudaStream_t st, cudaEvent_t mid = nullptr,
                         int64_t* launches = nullptr);
// The equal-layer search over the worklist the screen produced.
cudaError_t launch_eq_search(const PriceArgs& a, int num_sms, cudaStream_t st);
// Multi-template plans (Algorithm 1): per template slot the plans' arrays,
// already priced standalone (bounds required), overwritten with the plan's
// prices; per plan the templates placed and the summed throughput.
constexpr int kMaxTemplates = HEDDLE_MAX_TEMPLATES;
constexpr int kPlanMaxNode = HEDDLE_PLAN_MAX_NODE;
struct PlanSlot {
    const uint8_t* S;
    const uint16_t* M;
    const uint8_t* code;  // [s][stride]
    int64_t stride;
    int64_t* T;
    int64_t* B;
    uint16_t* ndp;
    uint8_t* status;
    uint8_t* bounds;  // [33][bstride]
    int64_t bstride;
    int32_t bounds_scratch;  // the caller passed none: nothing reads them afterwards
};
struct PlanArgs {
    Layout lay;
    const unsigned char* img;
    int64_t n;
    int32_t slots;
    const uint8_t* n_tmpl;
    PlanSlot slot[kMaxTemplates];
    const int32_t* node_type;
    const int32_t* node_gpus;
    int32_t n_nodes;
    int32_t vmax;  // largest node (GPUs), <= kPlanMaxNode
    int32_t per_pass;   // plans a CTA looks at in one pass (at most 128): batches of few spread over all SMs
    int32_t alone_min;  // queued plans of a CTA from which a thread walks each (0: by their depth)
    uint8_t* placed;
    double* thr;
    uint32_t* err;
};
cudaError_t launch_plans(const PlanArgs& a, int num_sms, cudaStream_t st);
// Ahead of the tiled search (heddle_gsearch.cu): the entries no split fits
// are priced OOM, the others listed at a.sv_idx (count at
// wl_count[kWlGeneral]); does nothing below a.thread_min bucketed entries.
cudaError_t launch_memory_probe(const PriceArgs& a, int num_sms, cudaStream_t st);

// The paper's own layer split over the worklist (comparison mode).  On a model
// of equal layers a thread prices each entry when the depth buckets hold at
// least PriceArgs::split_min plus split_per_stage entries for each stage of the
// deepest one, else a warp does (the device decides: few of a large batch may
// reach the search).  A warp's entries take 1.8 to 2.2 us per thousand, a
// thread's chain 5, 9, 18 or 41 us more than a warp's at 3, 8, 16 or 32 stages:
// measured, they meet at some 6,800, 9,500, 14,500 and 22,000 entries.
constexpr int32_t kSplitThreadMin = 5000, kSplitThreadPerStage = 550;
cudaError_t launch_distribute(const PriceArgs& a, int num_sms, cudaStream_t st);
constexpr int32_t kWorklistCap = 1 << 20;
constexpr int kWlMeta = 1 + kMaxStages + 1 + 2 + 1;  // ints of a.wl_count
constexpr int kWlGeneral = 1;  // entries the thread-per-entry general search left to the warp search
// the next entries the general searches take (each warp of the thread
// search takes 32 at a time, each warp of the warp search one)
constexpr int kWlTakeThread = kWlMeta - 3;
constexpr int kWlTakeWarp = kWlMeta - 2;
// The thread-per-entry general search runs when the depth buckets hold at
// least one warp of entries per SM; with fewer it would run one warp or less
// per SM, its time the latency of its longest serial chain, and the warp
// search (whose probes spread over 32 lanes) prices every entry instead.
inline int thread_search_min(int num_sms) { return num_sms * 32; }
constexpr int kWlSurv = kWlMeta - 1;             // the survivor count (see PriceArgs::sv_count)


// Entries a CTA of the top-k hands to the last one.
constexpr int kTopkListCap = 128;
// What the CTAs of one top-k launch share; behind it, for each of the max_blocks
// CTAs, the bar that it posts and whether it has.
struct alignas(16) TopkMeet {
    int32_t tickets;  // CTAs that have handed over
    int32_t entries;  // entries in the scratch list
    __host__ __device__ TopkEntry* bars() { return reinterpret_cast<TopkEntry*>(this + 1); }
    __host__ __device__ int32_t* posted(int max_blocks) { return reinterpret_cast<int32_t*>(bars() + max_blocks); }
    static size_t bytes(int max_blocks) { return sizeof(TopkMeet) + (sizeof(TopkEntry) + sizeof(int32_t)) * max_blocks; }
};

struct TopkArgs {
    // results of a batch (heddle_topk) ...
    const uint16_t* M;
    const int64_t* T;
    const uint16_t* ndp;
    const uint8_t* status;
    int64_t n;
    int64_t base_index;
    heddle_topk_state* state;  // device, in/out
    TopkEntry* scratch;        // [max_blocks * kTopkListCap]
    int32_t max_blocks;
    TopkMeet* meet;            // all zero between launches
    // ... or the worklist of a priced chunk (heddle_price_topk)
    const int32_t* wl_count;
    const int32_t* wl_idx;
    const int64_t* wl_T;
    const uint32_t* wl_nM;
    int32_t wl_cap;
    int32_t chained;    // launched behind its search (see launch_after)
    int32_t survivors;  // the worklist holds a threshold's survivors only
    // nullable: raised (atomicMax on the bits of a positive float) to the
    // new state's k-th key n*M / T in float times (1 - 2^-16) once the state
    // holds k entries.  Float conversions and the division are each within
    // 2^-24 relative, so the stored value stays below every key at least
    // the k-th's, exactly compared, by more than the rounding of a key
    // computed the same way.
    uint32_t* thr;
};
// `launches` (nullable) gains the number of kernels launched.
cudaError_t launch_topk(const TopkArgs& a, int num_sms, cudaStream_t st, int64_t* launches = nullptr);
// Top-k of the searched candidates of a priced chunk (a.wl_*), merged into
// *a.state; `n` bounds the worklist length (the chunk size).
cudaError_t launch_topk_worklist(const TopkArgs& a, int64_t n, int num_sms, cudaStream_t st,
                                 int64_t* launches = nullptr);
cudaError_t launch_topk_reset(heddle_topk_state* state, int32_t k, cudaStream_t st);

// Micro-batch-size fill: fold the results of the larger sizes (levels 1 ..
// levels - 1) into the base size's (smaller T wins, ties keep the smaller
// size).
struct MbsLevel {
    const int64_t* T;
    const int64_t* B;
    const uint16_t* ndp;
    const uint8_t* status;
    const uint8_t* bounds;  // nullable, plane stride MbsMergeArgs::bstride_l
};
struct MbsMergeArgs {
    int64_t n;
    int32_t levels;
    MbsLevel level[HEDDLE_MAX_MBS_LEVELS];  // [0] unused
    int64_t bstride_l;
    int64_t* T;
    int64_t* B;
    uint16_t* ndp;
    uint8_t* status;
    uint8_t* bounds;  // nullable, plane stride bstride
    int64_t bstride;
    uint8_t* mbs;     // nullable: the chosen level, 0 where none is OK
};
cudaError_t launch_mbs_merge(const MbsMergeArgs& a, int num_sms, cudaStream_t st);

// Conversions between non-negative 64-bit integers and float through their
// 32-bit halves: the 32-bit conversions run on the fast pipes, while a
// 64-bit conversion instruction runs on the (narrow) FP64 pipe.
// u64_to_float: relative error below 2^-23.
__device__ __forceinline__ float u64_to_float(uint64_t x) {
    return __fmaf_rn((float)(uint32_t)(x >> 32), 4294967296.0f, (float)(uint32_t)x);
}

// Truncation of a float in [0, 2^63) to an integer (exact: the low part
// f - hi 2^32 is representable).
__device__ __forceinline__ uint64_t float_to_u64(float f) {
    const float hi = floorf(f * 2.3283064365386963e-10f);
    const float lo = __fmaf_rn(-hi, 4294967296.0f, f);
    return ((uint64_t)(uint32_t)hi << 32) + (uint64_t)(uint32_t)fmaxf(lo, 0.f);
}

// ceil(A / C) for a 128-bit A and 1 <= C < 2^64 whose quotient is below
// 2^62: a float estimate of the quotient refined with exact 128-bit
// remainders (each refinement leaves about 2^-22 of the error), then exact
// unit steps.  *ok is cleared if the steps did not settle (never expected).
__device__ __forceinline__ float u128_to_float(u128 v) {
    return __fmaf_rn(u64_to_float((uint64_t)(v >> 64)), 18446744073709551616.0f, u64_to_float((uint64_t)v));
}

//
// The usual sizes (a quotient below 2^31, C below 2^50) need 64 bits only:
// the estimate is off by at most 2^-20 of the quotient, so the remainder
// stays below 2^62 and is exact modulo 2^64, and the second estimate is off
// by at most one.
__device__ inline uint64_t ceil_div_u128(u128 A, uint64_t C, bool* ok) {
    const float rc = 1.0f / u64_to_float(C);
    const float e = u128_to_float(A) * rc;
    if (e < 2147483648.0f && C < ((uint64_t)1 << 50)) {
        uint64_t q = (uint32_t)e;
        int64_t r = (int64_t)((uint64_t)A - q * C);
        const int d = (int)(u64_to_float((uint64_t)(r < 0 ? -r : r)) * rc);
        q += (int64_t)(r < 0 ? -d : d);
        r -= (int64_t)(r < 0 ? -d : d) * (int64_t)C;
        for (int it = 0; it < 3 && r < 0; ++it) {
            --q;
            r += (int64_t)C;
        }
        for (int it = 0; it < 3 && r >= (int64_t)C; ++it) {
            ++q;
            r -= (int64_t)C;
        }
        if (r < 0 || r >= (int64_t)C) *ok = false;
        return q + (r != 0 ? 1 : 0);
    }
    uint64_t q = e < 4.0e18f ? float_to_u64(e) : 4000000000000000000ull;
    for (int it = 0; it < 6; ++it) {
        const u128 qc = (u128)q * C;
        if (qc > A) {
            const uint64_t d = float_to_u64(u128_to_float(qc - A) * rc);
            q -= d == 0 ? 1 : (d < q ? d : q);
        } else {
            const u128 r = A - qc;
            if (r < C) break;
            const uint64_t d = float_to_u64(u128_to_float(r) * rc);
            q += d == 0 ? 1 : d;
        }
    }
    const u128 qc = (u128)q * C;
    if (qc > A || A - qc >= C) *ok = false;
    return q + (qc != A ? 1 : 0);
}

}  // namespace hd
