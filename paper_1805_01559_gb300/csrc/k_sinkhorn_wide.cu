// The persistent FP32 solver for rows of 1025 to 8192 columns (teams of 2, 4 and 8 warps).
#include <cuda_runtime.h>

#include "sk_kernels.cuh"

namespace ota {

namespace {
template <int TW, int VPT>
struct Plain {
    static Kernels get() { return Kernels{(const void*)sk_solve<TW, VPT>, TW, VPT, Cons<TW>::NCW, Cons<TW>::NT}; }
};
}  // namespace

bool pick_wide(int J, Kernels* k) { return pick_teams<Plain>(J, k); }

}  // namespace ota
