// sweep_grid_plain_r3.cu -- chip-resident register-tile kernels in the plain summation order: radius 3.
#include "sweep_grid.cuh"

namespace gbst {

// Kernel with rb rows per warp ({nullptr, 0} if not instantiated).
GridKernelRef get_grid_plain_kernel_r3(int star, int rb) {
    switch (rb) {
        case 4:
            return {star ? (const void*)sweep_grid_kernel<3, true, 4, false, true> : (const void*)sweep_grid_kernel<3, false, 4, false, true>,
                    grid_max_threads(3, 4)};
        case 8:
            return {star ? (const void*)sweep_grid_kernel<3, true, 8, false, true> : (const void*)sweep_grid_kernel<3, false, 8, false, true>,
                    grid_max_threads(3, 8)};
        default: return {nullptr, 0};
    }
}

}  // namespace gbst
