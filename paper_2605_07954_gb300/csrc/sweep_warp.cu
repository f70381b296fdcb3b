// sweep_warp.cu -- one-warp streaming kernels for whole grids: radius 1, 8 steps per launch.
#include "sweep_warp.cuh"

namespace gbst {

template <typename TS>
static const void* warp_kernel_for(int star, int nc) {
    if (!star) return nc == 4 ? (const void*)sweep_warp_kernel<false, 8, TS, 4> : nullptr;
    return nc == 4 ? (const void*)sweep_warp_kernel<true, 8, TS, 4> : (const void*)sweep_warp_kernel<true, 8, TS, 8>;
}

// Kernel advancing 8 steps with nc (4, or 8 for the 5-point star) columns per lane.
const void* get_warp_kernel(int star, int dtype, int nc) {
    switch (dtype) {
        case DT_F32: return warp_kernel_for<float>(star, nc);
        case DT_BF16: return warp_kernel_for<__nv_bfloat16>(star, nc);
        case DT_F16: return warp_kernel_for<__half>(star, nc);
        default: return nullptr;
    }
}

// The 5-point star's, storing every level (FP32, 4 columns per lane, nx % 4 == 0).
const void* get_warp_states_kernel() { return (const void*)sweep_warp_kernel<true, 8, float, 4, true>; }

}  // namespace gbst
