// Several solves on one cost matrix in one launch (sk_multi.cuh).
#include <cuda_runtime.h>

#include "sk_kernels.cuh"
#include "sk_multi.cuh"

namespace ota {

// Several solves sharing one cost matrix (sk_multi.cuh): the same launch structure.
template <int TW, int VPT, int NS, bool RC>
__global__ void __launch_bounds__(Cons<TW>::NT, 1) sk_solve_multi(MultiParams M, StreamCfg S) {
    constexpr int NCW = Cons<TW>::NCW;
    extern __shared__ __align__(128) unsigned char dyn[];
    __shared__ SkShared sh;
    uint64_t* full = reinterpret_cast<uint64_t*>(dyn);
    uint64_t* empty = full + MAX_STAGES;
    float* ring = reinterpret_cast<float*>(dyn + S.off_ring);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const SolveParams& P0 = M.P[0];
    int64_t r0, r1;
    cta_rows(P0.I, S.rows_per_stage, P0.V, blockIdx.x, gridDim.x, &r0, &r1);
    if (threadIdx.x == 0) {
        for (int s = 0; s < S.stages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], NCW);
        }
        sh.s_stop = 0;
        sh.s_bad = 0;
        sh.s_dec = 0;
        mbar_fence_init();
    }
    __syncthreads();
    if (warp == NCW) {
        if (lane == 0)
            stream_rows_producer(P0.C, P0.ld, r0, r1, S, ring, full, empty, &sh.s_stop, &M.grp->status, P0.spin);
        return;
    }
    GroupCtx g{(int)gridDim.x, (int)blockIdx.x, &M.grp->bar, 0u, &M.grp->status, &M.grp->status};
    ms_consumers<TW, VPT, NS, RC>(M, S, g, &sh, dyn, r0, r1);
}

// Kernels of the multi-solve launch.  Up to 128 float4 chunks a row, one-warp teams keep
// three solves' accumulators with the row (4 chunks a lane).  Wider rows: two solves on
// one-warp teams with the cell values computed twice (the row stays with the one-warp
// team of a single solve), three solves on wider teams (4 chunks a lane).
template <int TW, int VPT, int NS, bool RC>
static Kernels multi_for() {
    return Kernels{(const void*)sk_solve_multi<TW, VPT, NS, RC>, TW, VPT, Cons<TW>::NCW, Cons<TW>::NT};
}
bool pick_multi(int J, int n, Kernels* k) {
    const int J4 = (J + 3) / 4;
    if (J4 <= 32) *k = multi_for<1, 1, 3, false>();
    else if (J4 <= 64) *k = multi_for<1, 2, 3, false>();
    else if (J4 <= 96) *k = multi_for<1, 3, 3, false>();
    else if (J4 <= 128) *k = multi_for<1, 4, 3, false>();
    else if (n <= 2 && J4 <= 160) *k = multi_for<1, 5, 2, true>();
    else if (n <= 2 && J4 <= 192) *k = multi_for<1, 6, 2, true>();
    else if (n <= 2 && J4 <= 224) *k = multi_for<1, 7, 2, true>();
    else if (n <= 2 && J4 <= 256) *k = multi_for<1, 8, 2, true>();
    else if (J4 <= 256) *k = multi_for<2, 4, 3, false>();
    else if (J4 <= 512) *k = multi_for<4, 4, 3, false>();
    else if (J4 <= 1024) *k = multi_for<8, 4, 3, false>();
    else return false;
    return true;
}

}  // namespace ota
