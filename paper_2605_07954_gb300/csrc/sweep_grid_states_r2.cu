// sweep_grid_states_r2.cu -- chip-resident register-tile kernels that store every step: radius 2.
#include "sweep_grid.cuh"

namespace gbst {

// Kernel with rb rows per warp ({nullptr, 0} if not instantiated).
GridKernelRef get_grid_states_kernel_r2(int star, int rb) {
    switch (rb) {
        case 4:
            return {star ? (const void*)sweep_grid_kernel<2, true, 4, true> : (const void*)sweep_grid_kernel<2, false, 4, true>,
                    grid_max_threads(2, 4)};
        case 8:
            return {star ? (const void*)sweep_grid_kernel<2, true, 8, true> : (const void*)sweep_grid_kernel<2, false, 8, true>,
                    grid_max_threads(2, 8)};
        default: return {nullptr, 0};
    }
}

}  // namespace gbst
