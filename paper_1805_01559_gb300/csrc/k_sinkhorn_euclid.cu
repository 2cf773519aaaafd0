// The persistent FP32 solver with the Euclidean cost formed in its sweeps.
#include <cuda_runtime.h>

#include "sk_kernels.cuh"

namespace ota {

// Euclidean cost formed on the fly (Sec. IV cost choice (i)): no matrix is read, so there is
// no producer warp (the block is the consumer warps alone, which leaves each thread more
// registers); the RRH coordinates are staged once in the ring's space and every sweep forms
// C_ij = ||x_i - x_j|| from them and the device's coordinates.
template <int TW, int VPT>
__global__ void __launch_bounds__(Cons<TW>::NCW * 32, 1) sk_solve_euclid(SolveParams P, StreamCfg S) {
    extern __shared__ __align__(128) unsigned char dyn[];
    __shared__ SkShared sh;
    float* rx = reinterpret_cast<float*>(dyn + S.off_ring);
    for (int j = threadIdx.x; j < P.Jp; j += blockDim.x) {
        const float2 r = j < P.J ? P.rrh_xy[j] : make_float2(0.f, 0.f);
        rx[j] = r.x;
        rx[P.Jp + j] = r.y;
    }
    if (threadIdx.x == 0) {
        sh.s_stop = 0;
        sh.s_bad = 0;
    }
    if (threadIdx.x < 32) tmem_alloc(&sh.tmem, tmem_cols<TW, VPT>());
    __syncthreads();
    int64_t r0, r1;
    cta_rows(P.I, S.rows_per_stage, P.V, blockIdx.x, gridDim.x, &r0, &r1);
    GroupCtx g{(int)gridDim.x, (int)blockIdx.x, &P.st->bar, 0u, &P.st->status, &P.st->status};
    int par = 0;
    sk_consumers<TW, VPT, true>(P, S, g, &sh, dyn, r0, r1, &par);
    __syncthreads();
    if (threadIdx.x < 32) tmem_free(sh.tmem, tmem_cols<TW, VPT>());
}

namespace {
template <int TW, int VPT>
struct Euclid {
    static Kernels get() {
        return Kernels{(const void*)sk_solve_euclid<TW, VPT>, TW, VPT, Cons<TW>::NCW, Cons<TW>::NCW * 32};
    }
};
}  // namespace

bool pick_euclid(int J, Kernels* k) { return J <= 1024 ? pick_one_warp<Euclid>(J, k) : pick_teams<Euclid>(J, k); }

}  // namespace ota
