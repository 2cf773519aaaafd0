// The persistent FP32 solver for rows of up to 1024 columns (one-warp teams).
#include <cuda_runtime.h>

#include "sk_kernels.cuh"

namespace ota {

namespace {
template <int TW, int VPT>
struct Plain {
    static Kernels get() { return Kernels{(const void*)sk_solve<TW, VPT>, TW, VPT, Cons<TW>::NCW, Cons<TW>::NT}; }
};
}  // namespace

bool pick_narrow(int J, Kernels* k) { return pick_one_warp<Plain>(J, k); }

}  // namespace ota
