// heddle_mbs.cu -- the micro-batch-size fill (§5.3 "Micro-batch size"):
// the library prices a batch once per power-of-two micro-batch size (the
// same screen and search kernels, with that size's cost tables and M / 2^i
// micro-batches), and this kernel folds the larger sizes' results into the
// base size's: a size replaces the choice so far when it is OK and its
// iteration time is strictly shorter (or the choice is not OK), so equal
// times keep the smaller size.

#include <algorithm>

#include "heddle_internal.cuh"

namespace hd {
namespace {

// One pass over the candidates for all sizes: a thread reads each size's status
// and, where it is OK, its T, and copies the winner's results once.  (One
// pass per size, three launches for four sizes, and a memset of the choices:
// 250,000 candidates at four sizes 104 -> 91 us a call.)
__global__ void __launch_bounds__(256) mbs_merge_kernel(MbsMergeArgs a) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < a.n; c += stride) {
        uint8_t st[HEDDLE_MAX_MBS_LEVELS];
#pragma unroll
        for (int i = 0; i < HEDDLE_MAX_MBS_LEVELS; ++i)
            st[i] = i == 0 ? a.status[c] : i < a.levels ? a.level[i].status[c] : (uint8_t)HEDDLE_CAND_INVALID;
        int best = 0;
        int64_t T = st[0] == HEDDLE_CAND_OK ? a.T[c] : kInf;
#pragma unroll
        for (int i = 1; i < HEDDLE_MAX_MBS_LEVELS; ++i) {
            if (st[i] != HEDDLE_CAND_OK) continue;
            const int64_t t = a.level[i].T[c];
            if (t < T) {
                T = t;
                best = i;
            }
        }
        if (a.mbs) a.mbs[c] = (uint8_t)best;
        if (best == 0) continue;
        const MbsLevel& l = a.level[best];
        a.T[c] = T;
        a.B[c] = l.B[c];
        a.ndp[c] = l.ndp[c];
        a.status[c] = HEDDLE_CAND_OK;
        if (a.bounds && l.bounds)
            for (int s = 0; s <= kMaxStages; ++s) a.bounds[(int64_t)s * a.bstride + c] = l.bounds[(int64_t)s * a.bstride_l + c];
    }
}

}  // namespace

cudaError_t launch_mbs_merge(const MbsMergeArgs& a, int num_sms, cudaStream_t st) {
    if (a.n <= 0) return cudaSuccess;
    const int grid = (int)std::min<int64_t>((a.n + 255) / 256, (int64_t)num_sms * 8);
    mbs_merge_kernel<<<grid, 256, 0, st>>>(a);
    return cudaGetLastError();
}

}  // namespace hd
