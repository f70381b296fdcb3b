// adjoint.cu -- reverse-mode gradient of T Jacobi steps (stencil_adjoint).
//
// Forward (Sec. II-C): u_{t+1} = A u_t, (A u)[i][j] = sum_{dy,dx} W[dy+R][dx+R] u~[i+dy][j+dx].
// For a loss L(u_T) with lambda_T = dL/du_T:
//     lambda_t = A^T lambda_{t+1},  (A^T l)[p][q] = sum_{dy,dx} W[dy+R][dx+R] l~[p-dy][q-dx]
//              (a correlation with the flipped weights, same boundary rule),
//     dL/dW[dy+R][dx+R] = sum_{t<T} sum_{i,j} lambda_{t+1}[i][j] u~_t[i+dy][j+dx],
//     dL/du_0 = lambda_0.
//
// Memory: the states u_t are recomputed, not stored: a checkpoint every s
// steps (adj_interval: about sqrt(T), or one segment where all states fit) is written by a temporally blocked
// forward pass; walking the segments backwards, each segment's s states are
// recomputed from its checkpoint (temporally blocked launches that store every
// time level), then the adjoint steps of the segment run from its last state
// down to its first.  Both forward paths use the same per-point arithmetic, so
// the result does not depend on s.
//
// One kernel per reverse step fuses the lambda update and the weight-gradient
// products: each warp walks down the rows of lambda_{t+1} of its strip with a
// window of them in registers, writes lambda_t, and adds its (2R+1)^2 products
// to its CTA's FP64 partial.  Tile t of a launch is always CTA t and launches
// are ordered, so each partial sums its steps in a fixed order; a last kernel
// sums the partials over tiles in a fixed order.  The gradient is deterministic.
// adjoint_stream_kernel is that step for radius 1 and widths a multiple of 4;
// for everything else adjoint_step_kernel, or, where the caller rounds the weight
// gradient to FP32 (stencil_adjoint_w32), the radius is 2 or 3 and the grid has enough
// tiles for it (adjoint_run), the faster adjoint_rows_kernel.
//
// The FP64 weight gradient of stencil_adjoint is tied to the bits of the states, so
// where those depend on how steps are grouped they come from the streaming kernel
// (plan_keep_sums) and a fixed checkpoint interval.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <new>
#include <string>
#include <vector>

#include "../../include/stencil.h"
#include "common.cuh"

namespace gbst {

// Internal accessors of a plan (plan.cu).
void plan_weights(const stencil_plan_t* p, float* w);
void** plan_aux_slot(stencil_plan_t* p, int id);
void plan_set_aux_free(stencil_plan_t* p, int id, void (*freer)(void*));
void plan_set_stream(stencil_plan_t* p, cudaStream_t st);
bool plan_keep_sums(stencil_plan_t* p, bool on);
bool plan_states_vary(const stencil_plan_t* p);
bool plan_states_one_launch(const stencil_plan_t* p, bool any_order);
int plan_states_depth(const stencil_plan_t* p);
int64_t plan_sum_launches(const stencil_plan_t* p, int64_t T);
stencil_status_t plan_run_states(stencil_plan_t* p, const void* in, float* const* outs, int64_t n, bool any_order,
                                 cudaStream_t st);

// One reverse step of radius 2 or 3, any width, for weight gradients kept in FP32.  A warp owns 120 columns (lanes 1..30, 4 each;
// lanes 0 and 31 hold halo columns) of kAdrRows output rows and walks down the
// rows of lambda_{t+1} with the last 2R+1 of them in registers, each extended by
// R columns per side (shuffles).  Per output row o of the walk:
//   lambda_t[o][x] = sum_d W[d] lambda_{t+1}[o - dy][x - dx]      (dy-major, then dx)
//   g[d]          += u_t[o][x] * lambda_{t+1}[o - dy][x - dx]
// so u_t is read at the warp's own points only (the gradient's terms grouped by
// the u_t point, as in adjoint_stream_kernel).  The row loop is rolled (7 rows of
// 300-450 instructions would leave the instruction cache); the window moves down
// by register copies.  Rows arrive two ahead, 16 bytes a lane, or element by
// element where rows are not aligned.
//
// Gradient sums: two FP32 accumulators per tap and thread (even and odd rows: 16
// products each), whose 128 sums of a CTA are added without rounding error
// (TwoSum) before they go into its FP64 partial; that keeps the FP32 part no
// longer than the staged-tile form's 8 products and 5 levels of lane sums.
//
// What bounds it: latency; two warps a scheduler have (13 or 49) + 49 FMAs per point
// for radius 3 to issue (13-point star 1000 x 1022: issue 39 %, FMA pipe 23 %).  The
// staged-tile form (one point per lane and row, both windows read
// from shared memory) ran the 13-point star at 1000 x 1022 in 26.4 us a step:
// now 14.4 (ncu).
constexpr int kAdrWarps = 4;
constexpr int kAdrRows = 8;     // output rows per warp
constexpr int kAdrCols = 120;   // output columns per warp

// Row y of g at the lane's columns c .. c + 3: zero outside the grid, or wrapped.
__device__ __forceinline__ void adr_load(float (&v)[4], const float* __restrict__ g, int y, int c, int ny, int nx,
                                         bool per, bool vec) {
    v[0] = v[1] = v[2] = v[3] = 0.f;
    if (per) {
        if ((unsigned)y >= (unsigned)ny) y = (y % ny + ny) % ny;
    } else if ((unsigned)y >= (unsigned)ny) {
        return;
    }
    const float* row = g + (size_t)y * (size_t)nx;
    if (vec) {  // nx % 4 == 0: a chunk lies wholly inside or outside, and so does its wrapped image
        if (per) c = (unsigned)c < (unsigned)nx ? c : (c % nx + nx) % nx;
        if ((unsigned)c < (unsigned)nx) {
            const float4 q = __ldg(reinterpret_cast<const float4*>(row + c));
            v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
        }
        return;
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        int x = c + e;
        if (per && (unsigned)x >= (unsigned)nx) x = (x % nx + nx) % nx;
        if ((unsigned)x < (unsigned)nx) v[e] = __ldg(row + x);
    }
}

template <int R, bool STAR>
__global__ void __launch_bounds__(kAdrWarps * 32, 2)
    adjoint_rows_kernel(const float* __restrict__ lam_in, const float* __restrict__ u, float* __restrict__ lam_out,
                        double* __restrict__ partials, int ny, int nx, int periodic, Weights w, int tiles_x, int vec) {
    constexpr int D = 2 * R + 1, E = 4 + 2 * R, NR = kAdrRows + 2 * R;
    constexpr unsigned FULL = 0xffffffffu;
    static_assert(NR % 2 == 0, "the row loop runs in pairs");
    __shared__ float sums[D * D][kAdrWarps * 32 + 1];
    __shared__ double half[D * D];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int c = ((int)blockIdx.x % tiles_x) * kAdrCols - 4 + 4 * lane;
    const int yb = ((int)blockIdx.x / tiles_x) * (kAdrWarps * kAdrRows) + warp * kAdrRows;
    const bool per = periodic != 0;
    const bool own = lane >= 1 && lane <= 30 && c < nx;
    bool live[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) live[e] = c + e < nx;
    float win[D][E];
    float g[2][D * D];
#pragma unroll
    for (int k = 0; k < D * D; ++k) g[0][k] = g[1][k] = 0.f;
#pragma unroll
    for (int k = 0; k < D; ++k)
#pragma unroll
        for (int e = 0; e < E; ++e) win[k][e] = 0.f;
    float lv[2][4], uv[2][4];  // rows in flight: slot = walked row mod 2
    auto load = [&](int i) {   // walked row i (lambda row yb - R + i, u row yb + i - 2R)
        adr_load(lv[i & 1], lam_in, yb - R + i, c, ny, nx, per, vec != 0);
        const int o = yb + i - 2 * R;
        uv[i & 1][0] = uv[i & 1][1] = uv[i & 1][2] = uv[i & 1][3] = 0.f;
        if (own && i >= 2 * R && o < ny) adr_load(uv[i & 1], u, o, c, ny, nx, false, vec != 0);
    };
    load(0);
    load(1);
#pragma unroll 1
    for (int i0 = 0; i0 < NR; i0 += 2) {
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int i = i0 + j;
#pragma unroll
            for (int k = 0; k < D - 1; ++k)
#pragma unroll
                for (int e = 0; e < E; ++e) win[k][e] = win[k + 1][e];
#pragma unroll
            for (int e = 0; e < 4; ++e) win[D - 1][R + e] = lv[j][e];
#pragma unroll
            for (int e = 0; e < R; ++e) {
                win[D - 1][e] = __shfl_up_sync(FULL, lv[j][4 - R + e], 1);
                win[D - 1][R + 4 + e] = __shfl_down_sync(FULL, lv[j][e], 1);
            }
            float uu[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) uu[e] = uv[j][e];
            if (i + 2 < NR) {  // (j is i's parity: the slot just consumed)
                adr_load(lv[j], lam_in, yb - R + i + 2, c, ny, nx, per, vec != 0);
                const int o2 = yb + i + 2 - 2 * R;
                uv[j][0] = uv[j][1] = uv[j][2] = uv[j][3] = 0.f;
                if (own && i + 2 >= 2 * R && o2 < ny) adr_load(uv[j], u, o2, c, ny, nx, false, vec != 0);
            }
            const int o = yb + i - 2 * R;
            if (i < 2 * R || o >= ny) continue;
            // window row k holds lambda row o - R + k, column e of it grid column c - R + e
            float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int dy = -R; dy <= R; ++dy)
#pragma unroll
                for (int dx = -R; dx <= R; ++dx) {
                    const int t = (dy + R) * D + dx + R;
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const float l = win[R - dy][R + e - dx];
                        if (!STAR || dy == 0 || dx == 0) acc[e] = fmaf(w.w[t], l, acc[e]);
                        // (a column beyond the grid has no term, not a zero one: lambda may be infinite)
                        if (live[e]) g[j][t] = fmaf(uu[e], l, g[j][t]);
                    }
                }
            if (own) {
                float* row = lam_out + (size_t)o * (size_t)nx + c;
                if (vec) {
                    *reinterpret_cast<float4*>(row) = make_float4(acc[0], acc[1], acc[2], acc[3]);
                } else {
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        if (c + e < nx) row[e] = acc[e];
                }
            }
        }
    }
    // Fixed order: thread (tap, half) adds the 64 sums of two warps, sum and rounding
    // error apart; where that leaves the FP32 range, once more in FP64.  (Lanes that own
    // no columns have multiplied zeros by neighbours' lambdas, which may be infinite.)
#pragma unroll
    for (int k = 0; k < D * D; ++k) sums[k][threadIdx.x] = own ? g[0][k] + g[1][k] : 0.f;
    __syncthreads();
    for (int t = threadIdx.x; t < 2 * D * D; t += kAdrWarps * 32) {
        const int k = t % (D * D), h = t / (D * D);
        float s = 0.f, err = 0.f;
        for (int i = 0; i < 64; ++i) {
            const float v = sums[k][64 * h + i], n = s + v, z = n - s;
            err += (s - (n - z)) + (v - z);
            s = n;
        }
        double d = (double)s + (double)err;
        if (!(fabs(d) <= 3.5e38)) {
            d = 0.0;
            for (int i = 0; i < 64; ++i) d += (double)sums[k][64 * h + i];
        }
        if (h) half[k] = d;
        else partials[(size_t)blockIdx.x * D * D + k] += d;
    }
    __syncthreads();
    if (threadIdx.x < D * D) partials[(size_t)blockIdx.x * D * D + threadIdx.x] += half[threadIdx.x];
}

constexpr int kAdjTX = 32;          // output tile columns (one per lane)
constexpr int kAdjTY = 64;          // output tile rows
constexpr int kAdjRowsPerThread = 8;  // 8 warps x 8 rows

// The reverse step behind the FP64 weight gradient where adjoint_stream_kernel does
// not apply, on a 32 x 64 tile.  Its FP32 sums run over 8 rows x 32 columns before
// they go to FP64; a kernel that groups the products otherwise moves the FP64
// result by ~1e-8..1e-7, which callers who keep 64 bits would see (accumulators
// that reproduce these sums would need 4 x (2R+1)^2 registers in
// adjoint_rows_kernel).  Step and state in us, FP32, GB300, this | adjoint_rows_kernel:
// 13-point star 1000 x 1022 29.8 | 17.5, 4000 x 3004 280 | 135; radius 1 at
// 1000 x 1022 10.7 | 12.6, so radius 1 keeps this kernel for FP32 gradients too.  Lane tx owns column x0 + tx and warp ty
// rows y0 + 8 ty .. + 7; it walks its rows keeping the last 2R+1 staged rows
// of lambda_{t+1} and u_t (its column +- R) in registers, so each row costs
// 2 (2R+1) shared-memory loads for (2R+1)^2 lambda FMAs and (2R+1)^2 gradient FMAs.
template <int R>
__global__ void __launch_bounds__(256)
    adjoint_step_kernel(const float* __restrict__ lam_in, const float* __restrict__ u,
                        float* __restrict__ lam_out, double* __restrict__ partials, int ny, int nx,
                        int periodic, Weights w, int tiles_x, int /*vec*/) {
    constexpr int D = 2 * R + 1;
    constexpr int SY = kAdjTY + 2 * R, SX = kAdjTX + 2 * R;
    __shared__ float sl[SY][SX + 1];
    __shared__ float su[SY][SX + 1];
    __shared__ float red[8][D * D];
    const int tx = threadIdx.x, ty = threadIdx.y;  // (32, 8)
    const int x0 = (blockIdx.x % tiles_x) * kAdjTX;
    const int y0 = (blockIdx.x / tiles_x) * kAdjTY;

    // Stage both tiles with their halo (zero outside, or wrapped).  Every
    // thread issues all of its loads before its first shared-memory store, so
    // the DRAM latencies overlap.  Item i = tid + 256 it is staged row i / SX,
    // column i % SX, advanced without division.
    {
        constexpr int ITEMS = SY * SX, ITERS = (ITEMS + 255) / 256;
        const int tid0 = ty * 32 + tx;
        int r = tid0 / SX, c = tid0 % SX;
        float va[ITERS], vb[ITERS];
        int ra[ITERS], ca[ITERS];
#pragma unroll
        for (int it = 0; it < ITERS; ++it) {
            ra[it] = r;
            ca[it] = c;
            va[it] = vb[it] = 0.f;
            if (r < SY) {
                int y = y0 - R + r, x = x0 - R + c;
                bool ok = y >= 0 && y < ny && x >= 0 && x < nx;
                if (periodic) {
                    y = (y % ny + ny) % ny;
                    x = (x % nx + nx) % nx;
                    ok = true;
                }
                if (ok) {
                    const size_t i = (size_t)y * nx + x;
                    va[it] = __ldg(lam_in + i);
                    vb[it] = __ldg(u + i);
                }
            }
            c += 256 % SX;
            r += 256 / SX;
            if (c >= SX) {
                c -= SX;
                ++r;
            }
        }
#pragma unroll
        for (int it = 0; it < ITERS; ++it) {
            if (ra[it] < SY) {
                sl[ra[it]][ca[it]] = va[it];
                su[ra[it]][ca[it]] = vb[it];
            }
        }
    }
    __syncthreads();

    float g[D * D];
#pragma unroll
    for (int k = 0; k < D * D; ++k) g[k] = 0.f;
    // Register windows: wl[i][e] = lambda staged row (row0 + i), column tx + e;
    // wu likewise for u.  The output row o = r0 + k needs lambda rows o-R..o+R
    // (flipped correlation) and u rows o-R..o+R.
    const int r0 = ty * kAdjRowsPerThread;  // first output row (tile-local)
    float wl[D][D], wu[D][D];
#pragma unroll
    for (int i = 0; i < D - 1; ++i)
#pragma unroll
        for (int e = 0; e < D; ++e) {
            wl[i + 1][e] = sl[r0 + i][tx + e];
            wu[i + 1][e] = su[r0 + i][tx + e];
        }
#pragma unroll
    for (int k = 0; k < kAdjRowsPerThread; ++k) {
        // slide: drop the oldest staged row, append staged row r0 + k + 2R
#pragma unroll
        for (int i = 0; i < D - 1; ++i)
#pragma unroll
            for (int e = 0; e < D; ++e) {
                wl[i][e] = wl[i + 1][e];
                wu[i][e] = wu[i + 1][e];
            }
#pragma unroll
        for (int e = 0; e < D; ++e) {
            wl[D - 1][e] = sl[r0 + k + 2 * R][tx + e];
            wu[D - 1][e] = su[r0 + k + 2 * R][tx + e];
        }
        // window row i holds staged row r0 + k + i, i.e. grid row o - R + i for o = y0 + r0 + k
        const int y = y0 + r0 + k, x = x0 + tx;
        if (y >= ny || x >= nx) continue;
        // lambda_t[o] = sum_d W[d] lambda_{t+1}[o - d], dy-major then dx
        float acc = 0.f;
#pragma unroll
        for (int dy = -R; dy <= R; ++dy)
#pragma unroll
            for (int dx = -R; dx <= R; ++dx)
                acc = fmaf(w.w[(dy + R) * D + (dx + R)], wl[R - dy][R - dx], acc);
        lam_out[(size_t)y * nx + x] = acc;
        // dL/dW[d] += lambda_{t+1}[o] * u_t[o + d]
        const float lp = wl[R][R];
#pragma unroll
        for (int dy = -R; dy <= R; ++dy)
#pragma unroll
            for (int dx = -R; dx <= R; ++dx)
                g[(dy + R) * D + (dx + R)] = fmaf(lp, wu[R + dy][R + dx], g[(dy + R) * D + (dx + R)]);
    }
    // Fixed-order reduction: butterfly within each warp, then warps in order.
#pragma unroll
    for (int k = 0; k < D * D; ++k) {
        float v = g[k];
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
        if (tx == 0) red[ty][k] = v;
    }
    __syncthreads();
    const int tid = ty * 32 + tx;
    if (tid < D * D) {
        double s = 0.0;
        for (int wv = 0; wv < 8; ++wv) s += (double)red[wv][tid];
        partials[(size_t)blockIdx.x * D * D + tid] += s;
    }
}

// grad_w[k] = sum over tiles of partials[tile][k] in a fixed order: thread i of
// the block sums tiles i, i + 256, ... in increasing order, then the 256
// thread sums are added pairwise in a fixed tree.  One block per tap.
__global__ void __launch_bounds__(256)
    reduce_partials_kernel(const double* __restrict__ partials, int tiles, int taps,
                           double* __restrict__ grad_w) {
    __shared__ double sh[256];
    const int k = blockIdx.x;
    double s = 0.0;
    for (int t = threadIdx.x; t < tiles; t += 256) s += partials[(size_t)t * taps + k];
    sh[threadIdx.x] = s;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if (threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) grad_w[k] = sh[0];
}

// Row-streaming variant of the reverse step (radius 1, widths a multiple of
// 4).  A warp owns a 128-column strip of kAdsRows output rows, 4 adjacent
// columns per lane, and walks down the rows of lambda_{t+1} holding the last
// 2R+1 of them in registers, each extended by R columns on either side (the
// neighbouring lanes' columns by shuffles, the strip's outer columns loaded by
// lanes 0 and 31).  Rows arrive as 16-byte chunks kAdsAhead rows before their
// use; nothing goes through shared memory on the way.
//
// The arithmetic runs as packed FP32x2 FMAs on column pairs: own pairs
// (c0, c1), (c2, c3) and the three pairs that straddle them, (c-1, c0),
// (c1, c2), (c3, c4), built once per row.  Every tap (dy, dx) reads the same
// pair of the extended lambda_{t+1} row for both products of an output pair:
//   lambda_t[o][x]   += W[dy][dx] * lambda_{t+1}[o - dy][x - dx]
//   dL/dW[dy][dx]    += u_t[o][x] * lambda_{t+1}[o - dy][x - dx]
// The second line is the weight gradient sum_o lambda_{t+1}[o] u_t[o + d]
// with its terms grouped by the u_t point (o + d -> o): every (point, tap)
// term is counted once, by the warp that owns the u_t row, and lambda_{t+1}
// outside the grid is zero (or wrapped) as in the lambda update, so u_t is
// read only at the warp's own points, without halo.  Per output the lambda
// update adds dy-major, then dx, as adjoint_rows_kernel does (same bits);
// each thread adds its gradient products row by row, the CTA reduces them in
// a fixed order into its FP64 partial.
//
// A warp whose rows and halo columns all lie inside the grid walks without any
// bounds or wrap logic (pointer increments, unconditional loads); warps at the
// grid's edge take the checked path.
//
// Measured on GB300 (Heat 4096^2, reverse steps back to back over distinct
// u_t): 38.4 us per step against 29-31 us for a plain kernel that reads two
// grids and writes one; the previous form of this step (scalar FMAs, every
// load checked, gradient per lambda point with a u_t window) took 47.3 us at
// about 235 warp instructions per output row, this one issues about 120.  More
// rows in flight
// (5 or 8 ahead in registers: fewer CTAs per SM; or a per-warp shared-memory
// ring fed by bulk copies, 5 or 8 rows ahead), 7, 22, 25, 28 or 31 rows per
// warp, and the warps of a CTA side by side instead of stacked all measured
// the same or slower; evict-first loads of the rows that die with the step
// gained ~7 %.  Two reverse steps per pass (lambda_{t-1} from lambda_{t+1} in
// registers, the middle 120 of each warp's 128 columns stored: 8 B per
// point-step instead of 12, bit-identical lambda) ran 37.2-40.3 us per step
// against 36.8-38.1 for the single step (136 registers and 3 CTAs per SM, or
// 128 with spills and 4): the step is bound by the latency of each warp's row
// walk, not by the bytes it moves.
constexpr int kAdsWarps = 4;    // warps per CTA, stacked vertically
constexpr int kAdsRows = 16;    // output rows per warp
constexpr int kAdsCols = 128;   // strip width (32 lanes x 4 columns)
constexpr int kAdsAhead = 2;    // rows loaded ahead of their use
constexpr int kAdsHint = 1;     // L2 policy of the row loads and stores (AdsPolicy)

template <int R>
struct AdsRow {
    float4 v;     // the lane's 4 columns
    float h[R];   // lane 0: columns x0 - R .. x0 - 1; lane 31: x0 + 128 .. x0 + 127 + R
};

// Grid row y of g as lane `lane` of the strip at x0 needs it; zero outside the
// grid, or wrapped.  c = x0 + 4 lane is a multiple of 4 and nx % 4 == 0, so a
// chunk lies wholly inside or wholly outside the grid, and its wrapped image
// is again an aligned chunk.
template <int R>
__device__ __forceinline__ void ads_load(AdsRow<R>& a, const float* __restrict__ g, int y, int c, int x0,
                                         int lane, int ny, int nx, bool periodic) {
    bool rok = true;
    if (periodic) {
        if (y < 0 || y >= ny) y = (y % ny + ny) % ny;
    } else {
        rok = y >= 0 && y < ny;
    }
    const float* row = g + (size_t)(rok ? y : 0) * (size_t)nx;
    int cc = c;
    bool cok = true;
    if (periodic) {
        if (cc >= nx) cc %= nx;
    } else {
        cok = cc < nx;
    }
    a.v = rok && cok ? __ldg(reinterpret_cast<const float4*>(row + cc)) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int i = 0; i < R; ++i) {
        int xc = lane == 0 ? x0 - R + i : x0 + kAdsCols + i;
        bool ok = rok && (lane == 0 || lane == 31);
        if (periodic) {
            if (xc < 0 || xc >= nx) xc = (xc % nx + nx) % nx;
        } else {
            ok = ok && xc >= 0 && xc < nx;
        }
        a.h[i] = ok ? __ldg(row + xc) : 0.f;
    }
}

// Column pairs of one extended row (radius 1).
struct AdsPairs {
    float2 p0, p1;      // (c0, c1), (c2, c3)
    float2 sm, sc, sp;  // (c-1, c0), (c1, c2), (c3, c4)
};

__device__ __forceinline__ AdsPairs ads_pairs(const AdsRow<1>& a, int lane) {
    const float l = __shfl_up_sync(0xffffffffu, a.v.w, 1);
    const float r = __shfl_down_sync(0xffffffffu, a.v.x, 1);
    AdsPairs e;
    e.p0 = make_float2(a.v.x, a.v.y);
    e.p1 = make_float2(a.v.z, a.v.w);
    e.sm = make_float2(lane == 0 ? a.h[0] : l, a.v.x);
    e.sc = make_float2(a.v.y, a.v.z);
    e.sp = make_float2(a.v.w, lane == 31 ? a.h[0] : r);
    return e;
}

// Columns (2q + s, 2q + 1 + s) of the extended row, s in {-1, 0, 1}.
__device__ __forceinline__ float2 ads_pick(const AdsPairs& e, int q, int s) {
    if (q == 0) return s < 0 ? e.sm : s == 0 ? e.p0 : e.sc;
    return s < 0 ? e.sc : s == 0 ? e.p1 : e.sp;
}

// The lambda update and gradient products of one output row o = yb + k: pair
// q of the row's 4 columns, window slot (jj - R - dy) mod D holding lambda_{t+1}
// row o - dy, uu = u_t row o.
template <int D>
__device__ __forceinline__ float4 ads_products(const AdsPairs (&win)[D], int jj, float4 uu,
                                               const float2 (&wp)[D * D], float2 (&g)[D * D]) {
    constexpr int R = 1;
    const float2 U[2] = {make_float2(uu.x, uu.y), make_float2(uu.z, uu.w)};
    float2 acc[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        acc[q] = make_float2(0.f, 0.f);
#pragma unroll
        for (int dy = -R; dy <= R; ++dy)
#pragma unroll
            for (int dx = -R; dx <= R; ++dx) {
                const int t = (dy + R) * D + (dx + R);
                const float2 L = ads_pick(win[(jj - R - dy + 2 * D) % D], q, -dx);
                acc[q] = __ffma2_rn(wp[t], L, acc[q]);
                g[t] = __ffma2_rn(U[q], L, g[t]);
            }
    }
    return make_float4(acc[0].x, acc[0].y, acc[1].x, acc[1].y);
}

// L2 eviction priorities of the reverse step's row traffic (createpolicy and
// .L2::cache_hint, PTX ISA).  lambda_{t+1} and u_t are dead once this step has
// read them; lambda_t is read again by the next reverse step at once and, for
// grids up to about half the L2, can stay there if the dead rows leave first.
// HINT 0: default policy; 1: loads evict-first; 2: loads evict-first and
// stores evict-last; 3: stores evict-last only.
template <int HINT>
struct AdsPolicy {
    unsigned long long first = 0, last = 0;
    __device__ __forceinline__ AdsPolicy() {
        if (HINT == 1 || HINT == 2) asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(first));
        if (HINT >= 2) asm("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(last));
    }
    __device__ __forceinline__ float4 load4(const float* p) const {
        if (HINT == 1 || HINT == 2) {
            float4 v;
            asm("ld.global.nc.L2::cache_hint.v4.f32 {%0, %1, %2, %3}, [%4], %5;"
                : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                : "l"(p), "l"(first));
            return v;
        }
        return __ldg(reinterpret_cast<const float4*>(p));
    }
    __device__ __forceinline__ float load1(const float* p) const {
        if (HINT == 1 || HINT == 2) {
            float v;
            asm("ld.global.nc.L2::cache_hint.f32 %0, [%1], %2;" : "=f"(v) : "l"(p), "l"(first));
            return v;
        }
        return __ldg(p);
    }
    __device__ __forceinline__ void store4(float* p, float4 v) const {
        if (HINT >= 2) {
            asm volatile("st.global.L2::cache_hint.v4.f32 [%0], {%1, %2, %3, %4}, %5;" ::"l"(p), "f"(v.x), "f"(v.y),
                         "f"(v.z), "f"(v.w), "l"(last)
                         : "memory");
        } else {
            *reinterpret_cast<float4*>(p) = v;
        }
    }
};

// One warp's walk over its ROWS output rows, rows in flight held in registers
// (AHEAD rows ahead).  EDGE: rows or halo columns may fall outside the grid
// (checked loads, wrap, skipped outputs).
template <bool EDGE, int AHEAD, int ROWS, class POL>
__device__ __forceinline__ void ads_walk(const float* __restrict__ lam_in, const float* __restrict__ u,
                                         float* __restrict__ lam_out, float2 (&g)[9], int ny, int nx,
                                         bool per, const Weights& w, int x0, int yb, int lane, const POL& pol) {
    constexpr int R = 1, D = 3;
    constexpr int NR = ROWS + 2 * R;  // lambda rows walked: yb - R .. yb + ROWS - 1 + R
    constexpr int RING = AHEAD + 1;
    constexpr int G = RING % D == 0 ? RING : D * RING;  // a group: lcm(D, RING) rows (D = 3 is prime)
    static_assert(NR % G == 0, "ring and window indices are static within a group of rows");
    const int c = x0 + 4 * lane;
    const bool col_ok = c < nx;
    const size_t snx = (size_t)nx;
    float2 wp[D * D];  // (w, w) pairs for the packed FMAs
#pragma unroll
    for (int k = 0; k < D * D; ++k) wp[k] = make_float2(w.w[k], w.w[k]);

    AdsRow<1> ra[RING];  // lambda_{t+1} rows in flight, slot = walked row % RING
    float4 ru[RING];     // u_t rows in flight, slot = (output row + 2R) % RING, i.e. the
                         // walked row whose step uses it
    AdsPairs win[D];     // extended lambda_{t+1} rows, slot = walked row % D
    // interior walk: pointers to the next row to load (never formed at EDGE)
    const float* pl = nullptr;
    const float* ph = nullptr;
    const float* pu = nullptr;
    float* po = nullptr;
    if (!EDGE) {
        pl = lam_in + (size_t)(yb - R) * snx + c;
        ph = lam_in + (size_t)(yb - R) * snx + (lane == 0 ? x0 - R : x0 + kAdsCols);
        pu = u + (size_t)yb * snx + c;
        po = lam_out + (size_t)yb * snx + c;
    }
    const bool hl = lane == 0 || lane == 31;
    auto load_lam = [&](AdsRow<1>& a, int i) {  // walked row i
        if (EDGE) {
            ads_load<1>(a, lam_in, yb - R + i, c, x0, lane, ny, nx, per);
        } else {
            a.v = pol.load4(pl);
            a.h[0] = hl ? pol.load1(ph) : 0.f;
            pl += snx;
            ph += snx;
        }
    };
    auto load_u = [&](float4& v, int k) {  // output row yb + k
        if (EDGE) {
            const int y = yb + k;
            v = y < ny && col_ok ? __ldg(reinterpret_cast<const float4*>(u + (size_t)y * snx + c))
                                 : make_float4(0.f, 0.f, 0.f, 0.f);
        } else {
            v = pol.load4(pu);
            pu += snx;
        }
    };
    // the rows the first AHEAD steps use (output row k is used at walked row k + 2R)
#pragma unroll
    for (int i = 0; i < AHEAD; ++i) {
        load_lam(ra[i % RING], i);
        if (i - 2 * R >= 0 && i - 2 * R < ROWS) load_u(ru[i % RING], i - 2 * R);
    }
    // A rolled loop over groups of rows (a fully unrolled walk overflows the
    // instruction cache); inside a group every ring and window index is static.
#pragma unroll 1
    for (int s0 = 0; s0 < NR; s0 += G) {
#pragma unroll
        for (int jj = 0; jj < G; ++jj) {
            const int i = s0 + jj;
            if (i + AHEAD < NR) load_lam(ra[(jj + AHEAD) % RING], i + AHEAD);
            const int ku = i + AHEAD - 2 * R;  // used at walked row i + AHEAD
            if (ku >= 0 && ku < ROWS) load_u(ru[(jj + AHEAD) % RING], ku);
            win[jj % D] = ads_pairs(ra[jj % RING], lane);
            // output row o = yb + k, k = i - 2R; lambda_{t+1} row o - dy is walked
            // row i - R - dy, in window slot (jj - R - dy) mod D
            const int k = i - 2 * R, o = yb + k;
            if (k < 0) continue;
            if (EDGE && (o >= ny || !col_ok)) continue;
            const float4 res = ads_products<D>(win, jj % D, ru[jj % RING], wp, g);
            if (EDGE) {
                *reinterpret_cast<float4*>(lam_out + (size_t)o * snx + c) = res;
            } else {
                pol.store4(po, res);
                po += snx;
            }
        }
    }
}

// The reverse step (radius 1; AHEAD, ROWS: see ads_walk; HINT: L2 eviction
// priorities, see AdsPolicy).
template <int R, int AHEAD = kAdsAhead, int ROWS = kAdsRows, int HINT = kAdsHint>
__global__ void __launch_bounds__(kAdsWarps * 32, 5)
    adjoint_stream_kernel(const float* __restrict__ lam_in, const float* __restrict__ u,
                          float* __restrict__ lam_out, double* __restrict__ partials, int ny, int nx,
                          int periodic, Weights w, int tiles_x) {
    static_assert(R == 1, "the row-streaming reverse step is written for radius 1");
    constexpr int D = 2 * R + 1;
    __shared__ float red[kAdsWarps][D * D];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int x0 = (blockIdx.x % tiles_x) * kAdsCols;
    const int yb = (blockIdx.x / tiles_x) * (kAdsWarps * ROWS) + warp * ROWS;
    float2 g[D * D];
#pragma unroll
    for (int k = 0; k < D * D; ++k) g[k] = make_float2(0.f, 0.f);
    const AdsPolicy<HINT> pol;
    // interior: the warp's rows yb - R .. yb + ROWS - 1 + R and columns
    // x0 - R .. x0 + 127 + R lie in the grid
    const bool interior = yb >= R && yb + ROWS + R <= ny && x0 >= R && x0 + kAdsCols + R <= nx;
    if (interior)
        ads_walk<false, AHEAD, ROWS>(lam_in, u, lam_out, g, ny, nx, periodic != 0, w, x0, yb, lane, pol);
    else
        ads_walk<true, AHEAD, ROWS>(lam_in, u, lam_out, g, ny, nx, periodic != 0, w, x0, yb, lane, pol);
    // Fixed-order reduction: the pair halves, a butterfly within each warp,
    // then the warps in order.
#pragma unroll
    for (int k = 0; k < D * D; ++k) {
        float v = g[k].x + g[k].y;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
        if (lane == 0) red[warp][k] = v;
    }
    __syncthreads();
    if (threadIdx.x < D * D) {
        double s = 0.0;
#pragma unroll
        for (int wv = 0; wv < kAdsWarps; ++wv) s += (double)red[wv][threadIdx.x];
        partials[(size_t)blockIdx.x * D * D + threadIdx.x] += s;
    }
}

static const void* adjoint_stream_kernel_fn(int R) {
    return R == 1 ? (const void*)adjoint_stream_kernel<1> : nullptr;
}

static const void* adjoint_step_kernel_fn(int R) {
    switch (R) {
        case 1: return (const void*)adjoint_step_kernel<1>;
        case 2: return (const void*)adjoint_step_kernel<2>;
        case 3: return (const void*)adjoint_step_kernel<3>;
        default: return nullptr;
    }
}

static const void* adjoint_rows_kernel_fn(int R, bool star) {
    switch (R) {
        case 2: return star ? (const void*)adjoint_rows_kernel<2, true> : (const void*)adjoint_rows_kernel<2, false>;
        case 3: return star ? (const void*)adjoint_rows_kernel<3, true> : (const void*)adjoint_rows_kernel<3, false>;
        default: return nullptr;
    }
}

}  // namespace gbst

using namespace gbst;

namespace {

thread_local std::string g_adj_error;

stencil_status_t afail(stencil_status_t st, const std::string& msg) {
    g_adj_error = msg;
    return st;
}

#define ACK(call)                                                                           \
    do {                                                                                    \
        cudaError_t e_ = (call);                                                            \
        if (e_ != cudaSuccess)                                                              \
            return afail(STENCIL_ERR_CUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
    } while (0)

// Device scratch of the adjoint, kept by the plan and grown on demand.
struct AdjScratch {
    float* base = nullptr;
    size_t grids = 0;
    double* partials = nullptr;
    size_t npartials = 0;
};

void adj_scratch_free(void* v) {
    AdjScratch* sc = static_cast<AdjScratch*>(v);
    if (sc->base) cudaFree(sc->base);
    if (sc->partials) cudaFree(sc->partials);
    delete sc;
}

int64_t adj_sqrt(int64_t T) { return (int64_t)std::ceil(std::sqrt((double)T)); }

// Steps between checkpoints.  By default the whole run is one segment while its
// states take at most 1 GiB: no checkpoint pass is needed then.  Otherwise
// ceil(sqrt(T)), for radius 1 rounded up to whole launches of 8 steps (Heat 4096^2
// x 128: 12 steps a segment 3.16 ms of forward launches, 16 steps 2.82 ms).
// vary: states whose bits depend on the checkpoints (FP64 sums resolve them): sqrt(T) always.
int64_t adj_interval(int64_t T, int64_t asked, int R, size_t bytes, bool vary) {
    if (asked > 0) return std::min<int64_t>(asked, T);
    if (vary) return adj_sqrt(T);
    if ((double)(T + 3) * (double)bytes <= (double)(1ull << 30)) return T;
    const int64_t s = adj_sqrt(T);
    return std::min<int64_t>(R == 1 ? (s + 7) / 8 * 8 : s, T);
}

bool adj_star(const Weights& w, int R) {
    const int D = 2 * R + 1;
    for (int a = 0; a < D; ++a)
        for (int c = 0; c < D; ++c)
            if (a != R && c != R && w.w[a * D + c] != 0.f) return false;
    return true;
}

stencil_status_t adj_scratch(stencil_plan_t* plan, size_t grids, size_t grid_bytes, size_t npartials,
                             AdjScratch** out) {
    void** slot = plan_aux_slot(plan, 0);
    AdjScratch* sc = static_cast<AdjScratch*>(*slot);
    if (!sc) {
        sc = new (std::nothrow) AdjScratch();
        if (!sc) return afail(STENCIL_ERR_OOM, "host allocation failed");
        *slot = sc;
        plan_set_aux_free(plan, 0, adj_scratch_free);
    }
    if (sc->grids < grids) {
        if (sc->base) cudaFree(sc->base);
        sc->base = nullptr;
        sc->grids = 0;
        if (cudaMalloc(&sc->base, grids * grid_bytes) != cudaSuccess) {
            cudaGetLastError();
            sc->base = nullptr;
            return afail(STENCIL_ERR_OOM, "cudaMalloc of " + std::to_string(grids) + " adjoint grids failed");
        }
        sc->grids = grids;
    }
    if (sc->npartials < npartials) {
        if (sc->partials) cudaFree(sc->partials);
        sc->partials = nullptr;
        sc->npartials = 0;
        if (cudaMalloc(&sc->partials, sizeof(double) * npartials) != cudaSuccess) {
            cudaGetLastError();
            sc->partials = nullptr;
            return afail(STENCIL_ERR_OOM, "cudaMalloc of the gradient partials failed");
        }
        sc->npartials = npartials;
    }
    *out = sc;
    return STENCIL_OK;
}

}  // namespace

namespace {

// The plan in the form whose states' bits the FP64 sums are tied to, for one call.
struct KeepSums {
    stencil_plan_t* p;
    const bool on;
    KeepSums(stencil_plan_t* plan, bool wanted) : p(plan), on(wanted && plan_keep_sums(plan, true)) {}
    ~KeepSums() {
        if (on) plan_keep_sums(p, false);
    }
    KeepSums(const KeepSums&) = delete;
    KeepSums& operator=(const KeepSums&) = delete;
};

// w32: the caller rounds grad_w to FP32, so its sums may be grouped freely.
stencil_status_t adjoint_run(stencil_plan_t* plan, const void* u0, const void* grad_uT, int64_t T, void* grad_u0,
                             double* grad_w, int64_t ckpt_interval, stencil_stream_t stream, bool w32) {
    if (!plan || !u0 || !grad_uT || !grad_u0) return afail(STENCIL_ERR_INVALID_ARG, "NULL argument");
    if (T < 0 || ckpt_interval < 0) return afail(STENCIL_ERR_INVALID_ARG, "T and ckpt_interval must be >= 0");
    stencil_plan_info_t info{};
    stencil_status_t s = stencil_plan_info(plan, &info);
    if (s != STENCIL_OK) return afail(s, "stencil_plan_info failed");
    if (info.dtype != STENCIL_F32 || info.compute != STENCIL_COMPUTE_FP32)
        return afail(STENCIL_ERR_UNSUPPORTED, "the adjoint supports FP32 CUDA-core plans only");
    const int R = info.radius, D = 2 * R + 1;
    const int ny = (int)info.ny, nx = (int)info.nx;
    const size_t n = (size_t)ny * (size_t)nx;
    const size_t bytes = n * sizeof(float);
    cudaStream_t st = (cudaStream_t)stream;
    plan_set_stream(plan, st);
    Weights wf{};
    plan_weights(plan, wf.w);
    Weights wadj = wf;  // the step kernels index W directly; the flip is in their loops

    // The row-streaming step where it applies (its 16-byte row chunks need
    // nx % 4 == 0, and the buffers below are then 16-byte aligned), else the
    // any-width one.
    const bool streamed = adjoint_stream_kernel_fn(R) != nullptr && nx % 4 == 0;
    // (a star's off-axis weights are zero: adjoint_rows_kernel skips them in the lambda
    // update.)  Small grids have too few of its 120 x 32 tiles to hide their latency, and
    // periodic ragged rows load element by element.  A step's time less the staged
    // kernel's, us: radius 3 256^2 +2, 256 x 259 +4 (periodic +8), 500^2 +2, 600^2 -4, 600 x
    // 603 -2 (periodic +2), 800 x 803 periodic -3, 1000^2 -14; radius 2 400^2 0, 500 x 503 +2
    // (periodic +6), 800^2 -1 to -3, 800 x 803 -1 (periodic +2), 1000^2 -4, 1000 x 1003
    // periodic 0.
    const bool star = adj_star(wf, R);
    const bool wrapped = nx % 4 != 0 && info.boundary == STENCIL_BOUNDARY_PERIODIC;
    const size_t rows_from = R == 3 ? (wrapped ? 450000 : 300000) : (wrapped ? 1000000 : 500000);
    const bool rows = w32 && R > 1 && n >= rows_from;
    const int tile_cols = streamed ? kAdsCols : rows ? kAdrCols : kAdjTX;
    const int tiles_x = (nx + tile_cols - 1) / tile_cols;
    const int tile_rows = streamed ? kAdsWarps * kAdsRows : rows ? kAdrWarps * kAdrRows : kAdjTY;
    const int tiles = tiles_x * ((ny + tile_rows - 1) / tile_rows);
    if (T == 0) {
        if (grad_u0 != grad_uT) ACK(cudaMemcpyAsync(grad_u0, grad_uT, bytes, cudaMemcpyDeviceToDevice, st));
        if (grad_w) ACK(cudaMemsetAsync(grad_w, 0, sizeof(double) * D * D, st));
        return STENCIL_OK;
    }
    const KeepSums kept(plan, !w32);
    int64_t sgm = adj_interval(T, ckpt_interval, R, bytes, !w32 && plan_states_vary(plan));
    int64_t nseg = (T + sgm - 1) / sgm;
    // Buffers: nseg checkpoints, sgm segment states, two adjoint grids.
    AdjScratch* sc = nullptr;
    s = adj_scratch(plan, (size_t)nseg + (size_t)sgm + 2, bytes, (size_t)(tiles + 1) * D * D, &sc);
    if (s == STENCIL_ERR_OOM && ckpt_interval == 0 && sgm != adj_sqrt(T)) {  // the least memory, then
        sgm = adj_sqrt(T);
        nseg = (T + sgm - 1) / sgm;
        s = adj_scratch(plan, (size_t)nseg + (size_t)sgm + 2, bytes, (size_t)(tiles + 1) * D * D, &sc);
    }
    if (s != STENCIL_OK) return s;
    float* ckpt = sc->base;
    float* seg = sc->base + (size_t)nseg * n;
    float* lam[2] = {sc->base + (size_t)(nseg + sgm) * n, sc->base + (size_t)(nseg + sgm + 1) * n};
    double* partials = sc->partials;
    ACK(cudaMemsetAsync(partials, 0, sizeof(double) * (size_t)tiles * D * D, st));

    // Checkpoints u_{j*sgm}, j = 0..nseg-1 (temporally blocked forward).
    ACK(cudaMemcpyAsync(ckpt, u0, bytes, cudaMemcpyDeviceToDevice, st));
    for (int64_t j = 1; j < nseg; ++j) {
        s = stencil_run(plan, ckpt + (size_t)(j - 1) * n, ckpt + (size_t)j * n, sgm, stream);
        if (s != STENCIL_OK) return afail(s, std::string("checkpoint pass: ") + stencil_last_error());
    }
    ACK(cudaMemcpyAsync(lam[0], grad_uT, bytes, cudaMemcpyDeviceToDevice, st));
    int cur = 0;
    const void* kfn = streamed ? adjoint_stream_kernel_fn(R)
                      : rows   ? adjoint_rows_kernel_fn(R, star)
                               : adjoint_step_kernel_fn(R);
    if (!kfn) return afail(STENCIL_ERR_UNSUPPORTED, "no adjoint kernel for this radius");
    const dim3 block = streamed ? dim3(kAdsWarps * 32) : rows ? dim3(kAdrWarps * 32) : dim3(32, 8);
    int vec = nx % 4 == 0;
    int periodic = info.boundary == STENCIL_BOUNDARY_PERIODIC;
    std::vector<float*> segp((size_t)sgm);
    for (int64_t j = nseg - 1; j >= 0; --j) {
        const int64_t t0 = j * sgm;
        const int64_t len = std::min<int64_t>(sgm, T - t0);
        // states u_{t0} .. u_{t0+len-1}: seg[0] is the checkpoint itself; the
        // others come from temporally blocked launches that store every level
        const float* state0 = ckpt + (size_t)j * n;
        if (len > 1) {
            for (int64_t t = 1; t < len; ++t) segp[t - 1] = seg + (size_t)t * n;
            s = plan_run_states(plan, state0, segp.data(), len - 1, w32, st);
            if (s != STENCIL_OK) return afail(s, std::string("segment recompute: ") + stencil_last_error());
        }
        for (int64_t t = len - 1; t >= 0; --t) {
            const float* ut = t == 0 ? state0 : seg + (size_t)t * n;
            const float* lin = lam[cur];
            float* lout = lam[cur ^ 1];
            void* args[] = {(void*)&lin, (void*)&ut, (void*)&lout, (void*)&partials, (void*)&ny,
                            (void*)&nx,  (void*)&periodic, (void*)&wadj, (void*)&tiles_x, (void*)&vec};
            ACK(cudaLaunchKernel(kfn, dim3((unsigned)tiles), block, args, 0, st));
            cur ^= 1;
        }
    }
    ACK(cudaMemcpyAsync(grad_u0, lam[cur], bytes, cudaMemcpyDeviceToDevice, st));
    if (grad_w) {
        const int taps = D * D;
        // grad_w may be host memory: then the sums go to the tail of the
        // partials scratch first and are copied back, synchronising `stream`.
        cudaPointerAttributes pa{};
        const bool host = cudaPointerGetAttributes(&pa, grad_w) != cudaSuccess ||
                          pa.type == cudaMemoryTypeHost || pa.type == cudaMemoryTypeUnregistered;
        (void)cudaGetLastError();
        double* dst = host ? partials + (size_t)tiles * D * D : grad_w;
        reduce_partials_kernel<<<taps, 256, 0, st>>>(partials, tiles, taps, dst);
        ACK(cudaGetLastError());
        if (host) {
            ACK(cudaMemcpyAsync(grad_w, dst, sizeof(double) * taps, cudaMemcpyDeviceToHost, st));
            ACK(cudaStreamSynchronize(st));
        }
    }
    return STENCIL_OK;
}

}  // namespace

extern "C" {

const char* stencil_adjoint_last_error(void) { return g_adj_error.c_str(); }

stencil_status_t stencil_adjoint(stencil_plan_t* plan, const void* u0, const void* grad_uT, int64_t T,
                                 void* grad_u0, double* grad_w, int64_t ckpt_interval,
                                 stencil_stream_t stream) {
    return adjoint_run(plan, u0, grad_uT, T, grad_u0, grad_w, ckpt_interval, stream, false);
}

stencil_status_t stencil_adjoint_w32(stencil_plan_t* plan, const void* u0, const void* grad_uT, int64_t T,
                                     void* grad_u0, double* grad_w, int64_t ckpt_interval,
                                     stencil_stream_t stream) {
    return adjoint_run(plan, u0, grad_uT, T, grad_u0, grad_w, ckpt_interval, stream, true);
}

int64_t stencil_adjoint_launches(const stencil_plan_t* plan, int64_t T, int64_t ckpt_interval) {
    if (!plan || T < 0 || ckpt_interval < 0) return -1;
    if (T == 0) return 0;
    stencil_plan_info_t info{};
    const bool fused = stencil_plan_info(plan, &info) == STENCIL_OK && info.dtype == STENCIL_F32 &&
                       info.nx % 4 == 0;
    const int64_t sgm = adj_interval(T, ckpt_interval, info.radius,
                                     (size_t)info.ny * (size_t)info.nx * sizeof(float), plan_states_vary(plan));
    const int64_t nseg = (T + sgm - 1) / sgm;
    int64_t L = (nseg - 1) * plan_sum_launches(plan, sgm);  // checkpoints
    const bool one = plan_states_one_launch(plan, false);
    const int64_t step = fused ? 0 : plan_sum_launches(plan, 1);
    for (int64_t j = 0; j < nseg; ++j) {  // segment recompute: all-states launches of 8/4/2/1 steps
        int64_t m = std::min<int64_t>(sgm, T - j * sgm) - 1;
        if (one) {  // (register tiles)
            L += m > 0;
            continue;
        }
        if (!fused) {
            L += m * step;
            continue;
        }
        const int top = plan_states_depth(plan);
        for (int d = top; d >= 1 && m > 0; d /= 2)
            while (m >= d) {
                m -= d;
                ++L;
            }
    }
    L += T;      // adjoint steps
    return L + 1;  // reduction
}

}  // extern "C"
