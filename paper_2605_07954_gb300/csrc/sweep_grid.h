// sweep_grid.h -- host interface of the chip-resident register-tile kernel (sweep_grid.cuh).
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>

namespace gbst {

struct Weights;

// How a grid is cut into one register tile per SM.
struct GridConfig {
    int rb = 0;       // rows per warp
    int warps = 0;    // warps per CTA
    int k = 0;        // steps per exchange
    int H = 0, Hy = 0;  // halo columns and rows
    int bx = 0, by = 0, strips = 0, tiles_y = 0;
    int plain = 0;    // the cluster-resident kernel's summation order
    double cycles = 0;  // estimated SM cycles per step
};

// Cheapest configuration by the cost model; k > 0 or rb > 0 fixes that choice.
// False where no configuration fits `sms` tiles.
bool grid_config(int ny, int nx, int R, int star, int periodic, int sms, int k, int rb, GridConfig* out);

// The same kernel as k-step launches over any number of tiles (no exchange, so no
// waits): cheapest configuration with at least kmin steps per launch.
bool tiles_config(int ny, int nx, int R, int star, int periodic, int sms, int kmin, GridConfig* out);

// Whether the kernel can be launched with this configuration on the current device.
bool grid_fits(const GridConfig& c, int R, int star, int sms);

// Device scratch of a plan: two exchange grids and the control words (zeroed by the caller).
size_t grid_scratch_bytes(int ny, int nx);

// T steps, in one cooperative launch.  k <= c.k: steps per exchange of this launch.
// states (FP32 runs): the results of steps state_first .. T-1 as well, state_stride floats apart.
cudaError_t launch_grid(const GridConfig& c, int R, int star, int dtype, int periodic, const void* in, void* out,
                        int ny, int nx, int vec, int T, int k, void* scratch, unsigned* status, long long wait_ns,
                        int withhold, const Weights& w, cudaStream_t st, float* states = nullptr,
                        long long state_stride = 0, int state_first = 1);

// T <= c.k steps as an ordinary launch over a tiles_config (in and out distinct).
cudaError_t launch_tiles(const GridConfig& c, int R, int star, int dtype, int periodic, const void* in, void* out,
                         int ny, int nx, int vec, int T, const Weights& w, cudaStream_t st);

}  // namespace gbst
