// sweep_grid_states_r3.cu -- chip-resident register-tile kernels that store every step: radius 3.
#include "sweep_grid.cuh"

namespace gbst {

// Kernel with rb rows per warp ({nullptr, 0} if not instantiated).
GridKernelRef get_grid_states_kernel_r3(int star, int rb) {
    switch (rb) {
        case 4:
            return {star ? (const void*)sweep_grid_kernel<3, true, 4, true> : (const void*)sweep_grid_kernel<3, false, 4, true>,
                    grid_max_threads(3, 4)};
        case 8:
            return {star ? (const void*)sweep_grid_kernel<3, true, 8, true> : (const void*)sweep_grid_kernel<3, false, 8, true>,
                    grid_max_threads(3, 8)};
        default: return {nullptr, 0};
    }
}

}  // namespace gbst
