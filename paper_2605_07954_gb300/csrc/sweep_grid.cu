// sweep_grid.cu -- host side of the chip-resident register-tile kernel:
// configuration (cost model) and launch.
#include <algorithm>

#include "sweep_grid.cuh"
#include "sweep_grid.h"

namespace gbst {

GridKernelRef get_grid_kernel_r1(int star, int rb);
GridKernelRef get_grid_kernel_r2(int star, int rb);
GridKernelRef get_grid_kernel_r3(int star, int rb);

GridKernelRef get_grid_states_kernel_r1(int star, int rb);
GridKernelRef get_grid_states_kernel_r2(int star, int rb);
GridKernelRef get_grid_states_kernel_r3(int star, int rb);

GridKernelRef get_grid_plain_kernel_r1(int star, int rb);
GridKernelRef get_grid_plain_kernel_r2(int star, int rb);
GridKernelRef get_grid_plain_kernel_r3(int star, int rb);

static GridKernelRef grid_states_kernel(int R, int star, int rb) {
    switch (R) {
        case 1: return get_grid_states_kernel_r1(star, rb);
        case 2: return get_grid_states_kernel_r2(star, rb);
        case 3: return get_grid_states_kernel_r3(star, rb);
        default: return {nullptr, 0};
    }
}

static GridKernelRef grid_kernel(int R, int star, int rb, int plain = 0) {
    if (plain) switch (R) {
            case 1: return get_grid_plain_kernel_r1(star, rb);
            case 2: return get_grid_plain_kernel_r2(star, rb);
            case 3: return get_grid_plain_kernel_r3(star, rb);
            default: return {nullptr, 0};
        }
    switch (R) {
        case 1: return get_grid_kernel_r1(star, rb);
        case 2: return get_grid_kernel_r2(star, rb);
        case 3: return get_grid_kernel_r3(star, rb);
        default: return {nullptr, 0};
    }
}

static int up(int a, int b) { return (a + b - 1) / b; }

static const int kGridRows[2] = {4, 8};  // rows per warp
constexpr int kGridMaxK = 16;
constexpr int kGridMaxSmem = 200 * 1024;
// Cost model, in SM cycles, fitted to probes on GB300 (512^2 to 1400^2, radius 1
// and 3, k = 1..12): within 15 % of the measured step times, and its choice
// within 6 % of the best configuration timed.
constexpr double kGridExchange = 3000.0;  // one exchange: store and load through L2, skew between tiles
constexpr double kGridStep = 300.0;       // one step's barrier and exchange latency
static double grid_row_cycles(int taps, int R) { return 6.8 * taps + 10.0 * R; }  // one row of one warp

bool grid_config(int ny, int nx, int R, int star, int periodic, int sms, int k, int rb, GridConfig* out) {
    const int taps = star ? 4 * R + 1 : (2 * R + 1) * (2 * R + 1);
    bool found = false;
    for (int rows : kGridRows) {
        if (rb > 0 && rows != rb) continue;
        const GridKernelRef ref = grid_kernel(R, star, rows);
        if (!ref.fn) continue;
        for (int kk = 1; kk <= kGridMaxK; ++kk) {
            if (k > 0 && kk != k) continue;
            GridConfig c;
            c.rb = rows;
            c.k = kk;
            c.Hy = R * kk;
            c.H = up(R * kk, 4) * 4;
            c.bx = kGridCols - 2 * c.H;
            if (c.bx < 8) break;
            // Zero rule: the strips at the grid's edges own a halo depth more (see the kernel).
            const int ex = periodic ? 0 : 2 * c.H, ey = periodic ? 0 : 2 * c.Hy;
            c.strips = std::max(1, up(nx - ex, c.bx));
            if (c.strips > sms) continue;
            // As many tile rows as SMs: the fewer rows a tile has, the less each SM computes.
            c.by = std::max(1, up(ny - ey, std::max(1, sms / c.strips)));
            c.tiles_y = std::max(1, up(ny - ey, c.by));
            c.warps = up(std::min(c.by + 2 * c.Hy, periodic ? 1 << 30 : ny), rows);
            if (c.warps * 32 > ref.max_threads || grid_smem_bytes(R, c.warps) > kGridMaxSmem) continue;
            c.cycles = kGridStep + up(c.warps, 4) * rows * grid_row_cycles(taps, R) + kGridExchange / kk;
            if (!found || c.cycles < out->cycles) *out = c;
            found = true;
        }
    }
    return found;
}

constexpr double kTilesWave = 8000.0;  // launches of tiles: a wave's loads, stores, start and end

bool tiles_config(int ny, int nx, int R, int star, int periodic, int sms, int kmin, GridConfig* out) {
    const int taps = star ? 4 * R + 1 : (2 * R + 1) * (2 * R + 1);
    bool found = false;
    for (int rows : kGridRows) {
        const GridKernelRef ref = grid_kernel(R, star, rows);
        if (!ref.fn) continue;
        for (int kk = kmin; kk <= kGridMaxK; ++kk) {
            GridConfig c;
            c.rb = rows;
            c.k = kk;
            c.Hy = R * kk;
            c.H = up(R * kk, 4) * 4;
            c.bx = kGridCols - 2 * c.H;
            if (c.bx < 8) break;
            const int ex = periodic ? 0 : 2 * c.H, ey = periodic ? 0 : 2 * c.Hy;
            c.strips = std::max(1, up(nx - ex, c.bx));
            const int max_warps = std::min(ref.max_threads / 32, (kGridMaxSmem / (R * 32 * 16) - 1) / 4);
            const int by_max = max_warps * rows - 2 * c.Hy;
            if (by_max < 1) break;
            // the fewest tile rows, and up to three times as many (more CTAs per SM, fuller last waves)
            const int fewest = std::max(1, up(ny - ey, by_max));
            for (int ty = fewest; ty <= std::min(3 * fewest, fewest + 64); ++ty) {
                c.by = std::max(1, up(ny - ey, ty));
                c.tiles_y = std::max(1, up(ny - ey, c.by));
                c.warps = up(std::min(c.by + 2 * c.Hy, periodic ? 1 << 30 : ny), rows);
                if (c.warps > max_warps || c.warps < 4) continue;
                const int per_sm = std::max(1, max_warps / c.warps);
                const long long waves = ((long long)c.strips * c.tiles_y + (long long)sms * per_sm - 1) /
                                        ((long long)sms * per_sm);
                const double wave = kk * (kGridStep + up(per_sm * c.warps, 4) * rows * grid_row_cycles(taps, R)) + kTilesWave;
                c.cycles = (double)waves * wave / kk;
                if (!found || c.cycles < out->cycles) *out = c;
                found = true;
            }
        }
    }
    return found;
}

bool grid_fits(const GridConfig& c, int R, int star, int sms) {
    const GridKernelRef ref = grid_kernel(R, star, c.rb, c.plain);
    if (!ref.fn || (sms > 0 && c.strips * c.tiles_y > sms)) return false;
    const int smem = grid_smem_bytes(R, c.warps);
    int per_sm = 0;
    if (cudaFuncSetAttribute(ref.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kGridMaxSmem) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, ref.fn, c.warps * 32, (size_t)smem) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return per_sm >= 1;
}

size_t grid_scratch_bytes(int ny, int nx) {
    const size_t grid = (size_t)ny * (size_t)(up(nx, 4) * 4) * sizeof(uint2);
    return 2 * ((grid + 255) / 256 * 256) + sizeof(int) * kGridCtlInts;
}

cudaError_t launch_grid(const GridConfig& c, int R, int star, int dtype, int periodic, const void* in, void* out,
                        int ny, int nx, int vec, int T, int k, void* scratch, unsigned* status, long long wait_ns,
                        int withhold, const Weights& w, cudaStream_t st, float* states,
                        long long state_stride, int state_first) {
    const GridKernelRef ref = states ? grid_states_kernel(R, star, c.rb) : grid_kernel(R, star, c.rb, c.plain);
    if (!ref.fn) return cudaErrorInvalidValue;
    if (states) {  // (plain kernels: set when the plan is made, by grid_fits)
        const cudaError_t e =
            cudaFuncSetAttribute(ref.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kGridMaxSmem);
        if (e != cudaSuccess) return e;
    }
    GridParams p{};
    p.in = in;
    p.out = out;
    p.ny = ny;
    p.nx = nx;
    p.ld = nx;
    p.xld = up(nx, 4) * 4;
    const size_t grid = ((size_t)ny * p.xld * sizeof(uint2) + 255) / 256 * 256;
    p.xbuf[0] = static_cast<uint2*>(scratch);
    p.xbuf[1] = reinterpret_cast<uint2*>(static_cast<char*>(scratch) + grid);
    p.ctl = reinterpret_cast<int*>(static_cast<char*>(scratch) + 2 * grid);
    p.status = status;
    p.wait_ns = wait_ns;
    p.withhold = withhold;
    p.states = states;
    p.state_stride = state_stride;
    p.state_first = state_first;
    p.T = T;
    p.k = k;
    p.Hy = c.Hy;
    p.H = c.H;
    p.bx = c.bx;
    p.by = c.by;
    p.strips = c.strips;
    p.tiles_y = c.tiles_y;
    p.periodic = periodic;
    p.dtype = dtype;
    p.vec = vec;
    p.w = w;
    for (int i = 0; i < kMaxTaps; ++i) p.w2.w2[i] = make_float2(w.w[i], w.w[i]);
    void* args[] = {&p};
    return cudaLaunchCooperativeKernel(ref.fn, dim3((unsigned)(c.strips * c.tiles_y)), dim3((unsigned)(c.warps * 32)),
                                       args, (size_t)grid_smem_bytes(R, c.warps), st);
}

cudaError_t launch_tiles(const GridConfig& c, int R, int star, int dtype, int periodic, const void* in, void* out,
                         int ny, int nx, int vec, int T, const Weights& w, cudaStream_t st) {
    const GridKernelRef ref = grid_kernel(R, star, c.rb);
    if (!ref.fn || T > c.k || in == out) return cudaErrorInvalidValue;
    GridParams p{};
    p.in = in;
    p.out = out;
    p.ny = ny;
    p.nx = nx;
    p.ld = nx;
    p.T = T;
    p.k = c.k;
    p.Hy = c.Hy;
    p.H = c.H;
    p.bx = c.bx;
    p.by = c.by;
    p.strips = c.strips;
    p.tiles_y = c.tiles_y;
    p.periodic = periodic;
    p.dtype = dtype;
    p.vec = vec;
    p.w = w;
    for (int i = 0; i < kMaxTaps; ++i) p.w2.w2[i] = make_float2(w.w[i], w.w[i]);
    void* args[] = {&p};
    return cudaLaunchKernel(ref.fn, dim3((unsigned)(c.strips * c.tiles_y)), dim3((unsigned)(c.warps * 32)), args,
                            (size_t)grid_smem_bytes(R, c.warps), st);
}

}  // namespace gbst
