// heddle_tables.cu -- cost-table build (step 0 of the pricing path).
//
// One launch turns the cluster and model descriptions into the integer image
// the pricing kernels read:
//   * per (GPU type g, degree 2^j, layer l) the layer's time in whole ns --
//     the profile entry of the paper's cost model (§5.2: computation plus
//     communication of one layer per GPU type and TP degree), synthesised
//     from FLOPs and link bandwidths or taken from an explicit profile --
//     and its prefix sums over layers;
//   * prefix sums of state, activation and gradient bytes (memory validation
//     of §5.2, gradient synchronisation);
//   * per-type node statistics for the DP packing of §5.1/§5.3;
//   * the P2P constants between consecutive stages.
// One CTA per (type, degree) row, one per type for its memory runs, one for
// the rest; every CTA reads the nodes for itself (a few hundred, 256 at a
// time) and every prefix is a block scan, so no part of the build is a chain
// of L loads.  One CTA doing all of it, type by type and prefix by prefix in
// single threads, took 12 us for 8 layers, 35 us for 32 and 266 us for 128 of
// a 1,024-GPU cluster; this takes 7 us for any of them (18 us for 80 layers
// that all differ).
//
// Double arithmetic uses explicitly rounded intrinsics (no contraction into
// fused multiply-add) in the order the header documents.

#include <math.h>

#include "heddle_internal.cuh"

namespace hd {
namespace {

typedef unsigned __int128 u128;

constexpr int kThreads = 256;
constexpr int64_t kTableLimit = (int64_t)1 << 40;

// Nearest integer of v >= 0, halves away from zero.  v - trunc(v) is exact
// for every double below 2^52 (and zero above).
__device__ int64_t round_half_away(double v) {
    double r = trunc(v);
    if (__dsub_rn(v, r) >= 0.5) r = __dadd_rn(r, 1.0);
    return (int64_t)r;
}

// ceil(a / b), at most 2^63 - 1 (a P2P term at 1 byte/s needs 73 bits)
__device__ int64_t ceil_div(u128 a, u128 b) {
    const u128 q = (a + b - 1) / b;
    return q > (u128)kInf ? kInf : (int64_t)q;
}

// Per stage byte: inadmissible (bit 31), or what the stage adds to its
// type's demand word -- per class e the GPUs of groups placed in units of at
// least 2^e GPUs, in units of 2^e (a stage of 2^j GPUs is placed whole, or, on
// a type whose nodes are smaller, in the largest power of two a node holds).
__device__ uint32_t stage_desc(int b, int NT, int moe, const int32_t* gpus, const int32_t* maxn,
                               const int32_t* pow2) {
    const int g = b & 7, j = (b >> 3) & 3;
    if ((b >> 5) != 0 || g >= NT || gpus[g] <= 0 || (!moe && (1 << j) > maxn[g])) return 1u << 31;
    const int unit = (1 << j) <= maxn[g] ? (1 << j) : pow2[g];
    uint32_t d = 0;
    for (int e = 0; (1 << e) <= unit && e < 4; ++e) d += (uint32_t)((1 << j) >> e) << demand_shift(e);
    return d;
}

// The cluster's nodes per type, gathered by the CTA.
struct NodeStats {
    unsigned long long nic[kMaxTypes];  // slowest NIC
    int32_t gpus[kMaxTypes], maxn[kMaxTypes], pow2[kMaxTypes];
    int32_t cap[kMaxTypes * 4];
};

__device__ void gather_nodes(const TableArgs& a, NodeStats& n) {
    const int tid = threadIdx.x;
    if (tid < kMaxTypes) {
        n.nic[tid] = (unsigned long long)kInf;
        n.gpus[tid] = n.maxn[tid] = 0;
    }
    if (tid < kMaxTypes * 4) n.cap[tid] = 0;
    __syncthreads();
    for (int b = tid; b < a.n_nodes; b += kThreads) {
        const heddle_node nd = a.nodes[b];
        atomicAdd(&n.gpus[nd.type], nd.gpus);
        atomicMax(&n.maxn[nd.type], nd.gpus);
        atomicMin(&n.nic[nd.type], (unsigned long long)nd.nic_bw);
        for (int e = 0; e < 4; ++e) atomicAdd(&n.cap[nd.type * 4 + e], (nd.gpus >> e) << e);
    }
    __syncthreads();
    if (tid < kMaxTypes) {
        int p = 1;
        while (p * 2 <= n.maxn[tid] && p < 8) p *= 2;
        n.pow2[tid] = n.gpus[tid] ? p : 0;
        if (!n.gpus[tid]) n.nic[tid] = 0;
    }
    __syncthreads();
}

// Inclusive sum over the CTA's threads (L <= 255 values, one a thread).
__device__ int64_t block_scan(int64_t v, int64_t* warp_sums) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int64_t u = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += u;
    }
    __syncthreads();  // an earlier scan's sums are read
    if (lane == 31) warp_sums[warp] = v;
    __syncthreads();
    for (int w = 0; w < warp; ++w) v += warp_sums[w];
    return v;
}
static_assert(kThreads > kMaxLayers, "one layer per thread, and one thread past them");

__global__ void __launch_bounds__(kThreads) build_tables_kernel(TableArgs a) {
    __shared__ NodeStats nodes;
    __shared__ int64_t warp_sums[kThreads / 32];
    __shared__ int64_t pre[2][kThreads];
    __shared__ uint32_t flags;
    const Layout& y = a.lay;
    const int L = y.L, NT = y.NT;
    const int tid = threadIdx.x;
    ModelInfo* info = reinterpret_cast<ModelInfo*>(a.img + y.offModel);
    ScreenTabs* sc = reinterpret_cast<ScreenTabs*>(a.img + y.offScreen);
    EqTabs* eq = reinterpret_cast<EqTabs*>(a.img + y.offEq);
    if (tid == 0) flags = 0;
    gather_nodes(a, nodes);

    if ((int)blockIdx.x < 4 * NT) {
        // ---- one (type, degree) row: per-layer cost entries and prefix
        const int g = blockIdx.x >> 2, j = blockIdx.x & 3, l = tid;
        const bool on = l < L;
        int64_t q = 0;
        if (on && nodes.gpus[g] > 0) {
            double s;
            if (a.profile) {
                s = a.profile[(g * 4 + j) * L + l];
            } else {
                const heddle_layer ly = a.layers[l];
                const double k = (double)(1 << j);
                s = __ddiv_rn(ly.flops, __dmul_rn(__dmul_rn(k, a.types[g].tflops), 1e12));
                if (j > 0) {
                    const double bw = (1 << j) <= nodes.maxn[g] ? __ll2double_rn(a.types[g].intra_bw)
                                                                : __ll2double_rn((int64_t)nodes.nic[g]);
                    const double ring = __ddiv_rn(__dmul_rn(2.0, __dsub_rn(k, 1.0)), k);
                    double u = __dmul_rn(4.0, ring);
                    u = __dmul_rn(u, __ll2double_rn(ly.ar_bytes));
                    u = __ddiv_rn(u, bw);
                    s = __dadd_rn(s, u);
                    const double part = __ddiv_rn(__dsub_rn(k, 1.0), k);
                    u = __dmul_rn(4.0, part);
                    u = __dmul_rn(u, __ll2double_rn(ly.a2a_bytes));
                    u = __ddiv_rn(u, bw);
                    s = __dadd_rn(s, u);
                }
            }
            const double ns = __dmul_rn(s, 1e9);
            if (!(ns >= 0.0) || !(ns < 4.0e18)) {
                atomicOr(&flags, kTabBadValue);
            } else {
                q = round_half_away(ns);
            }
        }
        if (on) a.q[(g * 4 + j) * L + l] = q;
        // (an entry above the limit makes the total exceed it too)
        const int64_t sum = block_scan(min(q, kTableLimit + 1), warp_sums);
        int64_t* row = reinterpret_cast<int64_t*>(a.img + y.offP) + (size_t)(g * 4 + j) * (L + 1);
        if (tid == 0) {
            row[0] = 0;
            pre[0][0] = q;
            const int b = j * 8 + g;
            eq->q[b] = q;
            eq->rq[b] = q > 0 ? 1.0f / (float)q : 0.0f;
            eq->qf[b] = (float)q;
        }
        if (on) row[l + 1] = sum;
        if (on && sum > kTableLimit) atomicOr(&flags, kTabTooLarge);
        __syncthreads();
        const int uniform = __syncthreads_and(!on || q == pre[0][0]);
        if (tid == 0) info->row_uniform[blockIdx.x] = uniform;
    } else if ((int)blockIdx.x < 4 * NT + kMaxTypes) {
        // ---- one type's memory runs: the longest run of consecutive layers
        // whose state plus f in-flight activations fit one group of degree
        // 2^j; a candidate whose stages' runs sum below L cannot fit
        const int g = blockIdx.x - 4 * NT;
        const bool there = g < NT && nodes.gpus[g] > 0;
        const int64_t st = tid < L ? a.layers[tid].state_bytes : 0, ac = tid < L ? a.layers[tid].act_bytes : 0;
        const int64_t s_to = block_scan(st, warp_sums), a_to = block_scan(ac, warp_sums);
        if (tid < L) {
            pre[0][tid + 1] = s_to;
            pre[1][tid + 1] = a_to;
        }
        if (tid == 0) pre[0][0] = pre[1][0] = 0;
        __syncthreads();
        const int64_t st0 = pre[0][1], ac0 = pre[1][1];
        const int uniform = __syncthreads_and(tid >= L || (st == st0 && ac == ac0));
        uint8_t* win = a.img + y.offWin + g * 4 * 33;
        if (tid < 4 * 33) {
            const int f = tid % 33, j = tid / 33;
            int best = 0;
            if (there && f > 0) {
                const int64_t capk = a.types[g].mem_bytes << j;
                if (uniform) {
                    const int64_t per = st0 + f * ac0;
                    best = per <= 0 ? L : (int)min(capk / per, (int64_t)L);
                } else {
                    // two pointers: the furthest end grows with the start
                    int e = 0;
                    for (int i = 0; i < L; ++i) {
                        e = max(e, i);
                        while (e < L && (pre[0][e + 1] - pre[0][i]) + f * (pre[1][e + 1] - pre[1][i]) <= capk) ++e;
                        best = max(best, e - i);
                    }
                }
            }
            win[tid] = (uint8_t)best;
            if (f > 0) sc->run[f * 32 + j * 8 + g] = (uint16_t)(best ? best : kNoRun);
            else sc->run[j * 8 + g] = kNoRun;
        }
    } else {
        // ---- byte prefixes, the types' constants, P2P, the screen's and the
        // equal-layer search's remaining tables
        int64_t* SA = reinterpret_cast<int64_t*>(a.img + y.offSA);
        int64_t* PB = reinterpret_cast<int64_t*>(a.img + y.offPB);
        int64_t* p2p = reinterpret_cast<int64_t*>(a.img + y.offP2P);
        const heddle_layer first = a.layers[0];
        heddle_layer ly = first;
        if (tid < L) ly = a.layers[tid];
        const int64_t st = block_scan(tid < L ? ly.state_bytes : 0, warp_sums);
        const int64_t ac = block_scan(tid < L ? ly.act_bytes : 0, warp_sums);
        const int64_t pb = block_scan(tid < L ? ly.param_bytes : 0, warp_sums);
        if (tid < L) {
            SA[2 * (tid + 1)] = st;
            SA[2 * (tid + 1) + 1] = ac;
            PB[tid + 1] = pb;
        }
        if (tid == 0) SA[0] = SA[1] = PB[0] = 0;
        const int uni = __syncthreads_and(ly.state_bytes == first.state_bytes && ly.act_bytes == first.act_bytes);
        const int puni = __syncthreads_and(ly.param_bytes == first.param_bytes);
        if (tid == 0) {
            info->mem_uniform = uni;
            info->grad_uniform = puni;
            // a class whose capacity equals the class below's is dominated by
            // it (no less demand on the same GPUs)
            int need = 0;
            for (int g = 0; g < NT; ++g)
                for (int e = 1; e < 4; ++e)
                    if (nodes.cap[g * 4 + e] != nodes.cap[g * 4 + e - 1]) need |= 1 << e;
            sc->classes = (need & 2) ? 2 : (need & 4) ? 1 : 0;
        }
        if (tid < kMaxTypes) {
            const int g = tid;
            reinterpret_cast<int32_t*>(a.img + y.offGpus)[g] = nodes.gpus[g];
            reinterpret_cast<int32_t*>(a.img + y.offMaxN)[g] = nodes.maxn[g];
            reinterpret_cast<int32_t*>(a.img + y.offPow2)[g] = nodes.pow2[g];
            reinterpret_cast<int64_t*>(a.img + y.offInter)[g] = (int64_t)nodes.nic[g];
            reinterpret_cast<int64_t*>(a.img + y.offMem)[g] = g < NT ? a.types[g].mem_bytes : 0;
            const int32_t* cap = nodes.cap + g * 4;
            sc->cap[g] = make_float4((float)cap[0] + 0.5f, (float)(cap[1] >> 1) + 0.5f, (float)(cap[2] >> 2) + 0.5f,
                                     (float)(cap[3] >> 3) + 0.5f);
        }
        for (int b = tid; b < 256; b += kThreads)
            sc->desc[b] = stage_desc(b, NT, a.moe, nodes.gpus, nodes.maxn, nodes.pow2);
        for (int t = 32 * 33 + tid; t < 32 * 33 + 256; t += kThreads) sc->run[t] = kNoRun;
        if (tid < 32) {
            const uint64_t D = (uint64_t)nodes.nic[tid & 7] << (tid >> 3);
            eq->D[tid] = D;
            eq->rD[tid] = D > 0 ? 1.0f / (float)D : 0.0f;
            if ((tid & 7) >= NT) {  // (the row CTAs write the others)
                eq->q[tid] = 0;
                eq->rq[tid] = eq->qf[tid] = 0.0f;
            }
        }
        // P2P: forward activation plus backward gradient (2 x boundary bytes)
        // over the intra-node link when the two consecutive groups share a
        // node, else over the slower NIC of the two types
        for (int t = tid; t < 130; t += kThreads) {
            int64_t c = 0;
            if (t < kZeroP2P) {
                const int same = t & 1;
                const int h = (t >> 1) & 7;
                const int g = t >> 4;
                int64_t bw = 0;
                if (g < NT && h < NT && nodes.gpus[g] > 0 && nodes.gpus[h] > 0)
                    bw = same ? a.types[g].intra_bw : (int64_t)min(nodes.nic[g], nodes.nic[h]);
                if (bw > 0) {
                    c = ceil_div((u128)2 * (u128)a.boundary_bytes * 1000000000u, (u128)bw);
                    if (c > kTableLimit) atomicOr(&flags, kTabTooLarge);
                }
                p2p[t] = c;
            }
            eq->p2p[t] = c;
            eq->cf[t] = (float)c;
        }
        for (int t = tid; t < 33 * 32; t += kThreads) {
            const int b = t & 31, nx = t >> 5;
            const int g = b & 7, h = nx & 7;
            const int same = g == h && (1 << (b >> 3)) + (1 << (nx >> 3)) <= nodes.maxn[g];
            eq->pair[t] = (uint8_t)(nx == 32 ? kZeroP2P : (g * 8 + h) * 2 + same);
        }
    }
    __syncthreads();
    if (tid == 0) info->flags[blockIdx.x] = flags;
}

}  // namespace

cudaError_t launch_tables(const TableArgs& a, cudaStream_t st) {
    build_tables_kernel<<<table_ctas(a.lay.NT), kThreads, 0, st>>>(a);
    return cudaGetLastError();
}

}  // namespace hd
