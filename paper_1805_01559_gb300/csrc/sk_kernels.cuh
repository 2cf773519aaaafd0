// Kernels of the persistent FP32 solver and their choice by row length.  The instantiations
// live in several translation units so that they compile side by side.
#pragma once

#include "sk_core.cuh"

namespace ota {

struct Kernels {
    const void* solve;
    int tw, vpt, ncw;
    int nthreads;  // block size: the consumer warps, plus the producer warp where C is streamed
};

// The solver of C read from memory: teams of one warp up to 1024 columns (k_sinkhorn_narrow.cu),
// of 2, 4 and 8 warps up to 8192 (k_sinkhorn_wide.cu).  A lane holds VPT = ceil(J4 / (32 TW))
// chunks of four columns exactly; chunk_inside() relies on it.
bool pick_narrow(int J, Kernels* k);
bool pick_wide(int J, Kernels* k);
inline bool pick_kernels(int J, Kernels* k) { return J <= 1024 ? pick_narrow(J, k) : pick_wide(J, k); }
// The solver that forms the Euclidean cost in its sweeps (k_sinkhorn_euclid.cu).
bool pick_euclid(int J, Kernels* k);
// Up to three solves of one C in a launch (k_sinkhorn_multi.cu).
bool pick_multi(int J, int n, Kernels* k);

template <int TW, int VPT>
__global__ void __launch_bounds__(Cons<TW>::NT, 1) sk_solve(SolveParams P, StreamCfg S) {
    constexpr int NCW = Cons<TW>::NCW;
    extern __shared__ __align__(128) unsigned char dyn[];
    __shared__ SkShared sh;
    uint64_t* full = reinterpret_cast<uint64_t*>(dyn);
    uint64_t* empty = full + MAX_STAGES;
    float* ring = reinterpret_cast<float*>(dyn + S.off_ring);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int64_t r0, r1;
    cta_rows(P.I, S.rows_per_stage, P.V, blockIdx.x, gridDim.x, &r0, &r1);
    if (threadIdx.x == 0) {
        for (int s = 0; s < S.stages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], NCW);
        }
        sh.s_stop = 0;
        sh.s_bad = 0;
        mbar_fence_init();
    }
    if (warp == 0) tmem_alloc(&sh.tmem, tmem_cols<TW, VPT>());
    __syncthreads();
    if (warp == NCW) {
        if (lane == 0)
            stream_rows_producer(P.C, P.ld, r0, r1, S, ring, full, empty, &sh.s_stop, &P.st->status, P.spin);
        return;
    }
    GroupCtx g{(int)gridDim.x, (int)blockIdx.x, &P.st->bar, 0u, &P.st->status, &P.st->status};
    int par = 0;
    sk_consumers<TW, VPT>(P, S, g, &sh, dyn, r0, r1, &par);
    bar_named(CONS_BAR, NCW * 32);
    if (warp == 0) tmem_free(sh.tmem, tmem_cols<TW, VPT>());
}

// VPT by row length for teams of one warp, and for wider ones.
template <template <int, int> class K>
bool pick_one_warp(int J, Kernels* k) {
    switch ((J + 127) / 128) {
        case 1: *k = K<1, 1>::get(); return true;
        case 2: *k = K<1, 2>::get(); return true;
        case 3: *k = K<1, 3>::get(); return true;
        case 4: *k = K<1, 4>::get(); return true;
        case 5: *k = K<1, 5>::get(); return true;
        case 6: *k = K<1, 6>::get(); return true;
        case 7: *k = K<1, 7>::get(); return true;
        case 8: *k = K<1, 8>::get(); return true;
        default: return false;
    }
}
template <template <int, int> class K, int TW>
bool pick_team(int J, Kernels* k) {
    switch ((J + 128 * TW - 1) / (128 * TW)) {
        case 5: *k = K<TW, 5>::get(); return true;
        case 6: *k = K<TW, 6>::get(); return true;
        case 7: *k = K<TW, 7>::get(); return true;
        case 8: *k = K<TW, 8>::get(); return true;
        default: return false;
    }
}
template <template <int, int> class K>
bool pick_teams(int J, Kernels* k) {
    if (J <= 2048) return pick_team<K, 2>(J, k);
    if (J <= 4096) return pick_team<K, 4>(J, k);
    return pick_team<K, 8>(J, k);
}

}  // namespace ota
