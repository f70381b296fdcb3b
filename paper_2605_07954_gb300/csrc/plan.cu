// plan.cu -- host side of the C ABI: plans, launch sequencing, workspace.
//
// A plan fixes (shape, radius, weights, dtype, boundary) and picks a kernel
// configuration: the temporal-blocking depth k, the CTA size and the tile
// shape of the streaming kernel (sweep_stream.cuh), or the naive kernel.
// stencil_run() then issues ceil(T/k) launches that ping-pong between the
// caller's output and one plan-owned workspace grid, so that the last launch
// writes `out` and `in` is never written.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <string>
#include <tuple>
#include <vector>

#include "../../include/stencil.h"
#include "common.cuh"
#include "stream_depths.h"
#include "sweep_grid.h"
#include "sweep_stream.cuh"

namespace gbst {
#define GBST_DECL_STREAM(R, DT) StreamKernelRef get_stream_kernel_r##R##_##DT(int star, int k, int vec);
GBST_DECL_STREAM(1, f32) GBST_DECL_STREAM(1, bf16) GBST_DECL_STREAM(1, f16)
GBST_DECL_STREAM(2, f32) GBST_DECL_STREAM(2, bf16) GBST_DECL_STREAM(2, f16)
GBST_DECL_STREAM(3, f32) GBST_DECL_STREAM(3, bf16) GBST_DECL_STREAM(3, f16)
#undef GBST_DECL_STREAM
StreamKernelRef get_stream_states_kernel(int R, int star, int k);
StreamKernelRef get_stream_pad_kernel_f32(int R, int star, int k);
StreamKernelRef get_stream_pad_kernel_bf16(int R, int star, int k);
StreamKernelRef get_stream_pad_kernel_f16(int R, int star, int k);
const void* get_warp_kernel(int star, int dtype, int nc);
const void* get_warp_states_kernel();
StreamKernelRef get_stream_tma_kernel_r1(int star, int k);
StreamKernelRef get_stream_tma_kernel_r2(int star, int k);
StreamKernelRef get_stream_tma_kernel_r3(int star, int k);
const void* get_naive_kernel(int radius, int dtype);
int lowrank_factor(const float* w, int R, int rank, float col[7][7], float row[7][7], double* sv);
const void* get_lowrank_kernel(int R, int rho);
cudaError_t launch_lowrank(const void* fn, const float* src, float* dst, long long ny, long long nx, int periodic,
                           const float col[7][7], const float row[7][7], int sms, cudaStream_t st);
const void* get_box49_tc_kernel(int dtype, int engine);       // engine: 0 TF32, 1 BF16, 2 3xTF32
const void* get_box49_tc_pipe_kernel(int dtype, int engine);
int box49_tc_smem_bytes(int engine);
const void* get_box49_umma_kernel(int tf32, int nt);
int box49_umma_smem_bytes(int tf32, int nt);
int box49_umma_threads(int nt);
int box49_umma_tile_rows(int nt);
cudaError_t launch_box49_umma(int tf32, int nt, const void* src, void* dst, int ny, int nx, int ld,
                              int round_out, unsigned* status, const float* w, int ctas, cudaStream_t st,
                              int timeout_ms, int withhold);
const void* get_box49_phase_kernel(int tf32);
int box49_phase_smem_bytes(int tf32);
int box49_phase_rows();
int box49_phase_cols(int tf32);
cudaError_t launch_box49_phase(int tf32, const void* src, void* dst, int ny, int nx, int round_out, unsigned* status,
                               const float* w, int ctas, cudaStream_t st, int timeout_ms, int withhold);
const void* get_resident_kernel(int radius, int star, int dtype);
int resident_threads();
int resident_max_cluster();
int resident_config(int ny, int nx, int radius, int periodic, int C, int kb, int max_smem, int* rp_out);
cudaError_t launch_resident(const void* fn, int C, int smem, const ResidentParams& prm, cudaStream_t st);
bool resident_cluster_fits(const void* fn, int C, int smem, int max_smem);
struct TcParams {  // must match box49_tc.cu
    const void* in;
    void* out;
    int ny, nx, ld;
    int periodic;
    int tiles_x, tiles;
    int vec;
    int convert_in;
    int round_out;
    float w[49];
};
}  // namespace gbst

using namespace gbst;

static thread_local std::string g_last_error;

static stencil_status_t fail(stencil_status_t st, const std::string& msg) {
    g_last_error = msg;
    return st;
}

#define CK(call)                                                                     \
    do {                                                                             \
        cudaError_t e_ = (call);                                                     \
        if (e_ != cudaSuccess) {                                                     \
            return fail(STENCIL_ERR_CUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
        }                                                                            \
    } while (0)

struct stencil_plan {
    int64_t ny = 0, nx = 0;
    int R = 0;
    int star = 0;
    int dtype = 0, boundary = 0, compute = 0;
    Weights w{};
    stencil_options_t opt{};
    int device = 0, sms = 0;
    // chosen configuration
    int kernel = STENCIL_KERNEL_STREAM;
    int k = 1, threads = 0, H = 0, bx = 0, by = 0, strips = 0, tiles_y = 0, smem = 0;
    int per_sm = 0;
    int tma = 0;  // streaming kernel fed by the tensor-memory-access engine
    // separable (low-rank) form of the weights: rank and FP32 factors
    int lr_rank = 0;
    float lr_col[7][7] = {}, lr_row[7][7] = {};
    const void* lr_fn = nullptr;
    const void* tc_pipe = nullptr;  // persistent double-buffered tensor-core kernel
    int tc_pipe_smem = 0, tc_pipe_ctas = 0;
    int umma_n = 0;     // tcgen05 engine in use: N of one MMA (0: warp-MMA engine)
    int umma_ok = 0;    // usable tcgen05 MMA widths, bit n / 16
    int umma_ctas = 0;
    int phase_ok = 0, phase = 0;  // tcgen05 kernel with four output rows per MMA row: usable, in use
    int phase_ctas = 0;
    // one-warp streaming kernel (sweep_warp.cuh) for launches of kWarpDepth steps: columns per
    // lane (0: not in use) and its tiles
    int warp_nc = 0, warp_bx = 0, warp_by = 0, warp_strips = 0, warp_tiles = 0;
    // cluster-resident kernel (sweep_resident.cu): usable cluster sizes (bit log2 C), the one in use
    const void* res_fn = nullptr;
    int res_ok = 0, res_c = 0, res_rp = 0, res_kb = 1, res_smem = 0, res_max_smem = 0;
    // chip-resident register tiles (sweep_grid.cuh): usable, in use (kernel == RESIDENT then), scratch
    int grid_ok = 0, grid_on = 0;
    GridConfig grid;
    // streaming plans: launches of up to tiles.k steps as register tiles: usable, in use
    int tiles_ok = 0, tiles_on = 0;
    int kept_kernel = 0, kept_grid = 0, kept_tiles = 0;  // what plan_keep_sums puts back
    GridConfig tiles;
    void* grid_mem = nullptr;
    void* status_mem = nullptr;  // the status word's own allocation, where it has one
    // streaming runs of a width that is not a multiple of 4 (zero rule): two grids of padded rows
    int64_t pad_ld = 0;
    unsigned pad_set = 0;  // bit k: that kernel's shared-memory attribute is set
    void* pad[2] = {nullptr, nullptr};
    unsigned smem_set = 0;  // bit 2k+vec: that kernel's shared-memory attribute is set
    int tuned = 0;
    const void* naive = nullptr;
    // memory
    size_t elem = 4;
    void* ws = nullptr;
    void* host_in = nullptr;
    void* host_out = nullptr;
    unsigned int* status = nullptr;
    cudaStream_t last_stream = nullptr;
    // Scratch of other subsystems (0: adjoint, 1: residual runs), released with the plan.
    void* aux[4] = {nullptr, nullptr, nullptr, nullptr};
    void (*aux_free[4])(void*) = {nullptr, nullptr, nullptr, nullptr};
};

namespace gbst {
void plan_weights(const stencil_plan_t* p, float* w) {
    for (int i = 0; i < kMaxTaps; ++i) w[i] = p->w.w[i];
}
void** plan_aux_slot(stencil_plan_t* p, int id) { return &p->aux[id]; }
// The stream whose work stencil_plan_status waits for.
void plan_set_stream(stencil_plan_t* p, cudaStream_t st) { p->last_stream = st; }
void plan_set_aux_free(stencil_plan_t* p, int id, void (*freer)(void*)) { p->aux_free[id] = freer; }
// Whether the bits of a run's states depend on how its steps are grouped into calls.
bool plan_states_vary(const stencil_plan_t* p) {
    return (p->kernel == STENCIL_KERNEL_RESIDENT && (!p->grid_on || p->grid.plain)) ||
           (p->boundary == STENCIL_BOUNDARY_PERIODIC && p->nx % 4 != 0);
}
}  // namespace gbst

static size_t elem_size(int dtype) { return dtype == STENCIL_F32 ? 4 : 2; }

static int64_t ceil_div(int64_t a, int64_t b) { return (a + b - 1) / b; }

static StreamKernelRef stream_kernel(int R, int star, int k, int dtype, int vec) {
    typedef StreamKernelRef (*Getter)(int, int, int);
    static const Getter table[3][3] = {
        {get_stream_kernel_r1_f32, get_stream_kernel_r1_bf16, get_stream_kernel_r1_f16},
        {get_stream_kernel_r2_f32, get_stream_kernel_r2_bf16, get_stream_kernel_r2_f16},
        {get_stream_kernel_r3_f32, get_stream_kernel_r3_bf16, get_stream_kernel_r3_f16}};
    if (R < 1 || R > 3 || dtype < 0 || dtype > 2) return {nullptr, 0};
    return table[R - 1][dtype](star, k, vec);
}

// Largest instantiated depth for (R, star), and the largest one <= k.
static int stream_kmax(int R, int star) {
    int m = 0;
    for (int i = 0; i < 8 && kStreamDepths[R - 1][star][i]; ++i) m = kStreamDepths[R - 1][star][i];
    return m;
}

static int stream_depth_at_most(int R, int star, int k) {
    int m = 0;
    for (int i = 0; i < 8 && kStreamDepths[R - 1][star][i]; ++i)
        if (kStreamDepths[R - 1][star][i] <= k) m = kStreamDepths[R - 1][star][i];
    return m;
}

// Default depth before any tuning: deep enough that HBM stops binding for the
// light stencils, 2 for the 49-point box (arithmetic-bound already at k = 1;
// at 16384^2 FP32, k = 2 with 256-thread CTAs 509 GStencil/s against 478 for
// k = 1 with 128 threads).
// These are the best measured choices for 8192^2 FP32 grids on GB300 (the
// 13-point star: k = 3 with its 128-register bound, 4 CTAs per SM, ties k = 2
// at 1173 GStencil/s and moves a third less DRAM traffic; k = 4 needs more
// registers than fit 4 CTAs).
static int default_depth(int R, int star) {
    if (R == 1) return 8;
    if (R == 2) return 4;
    return star ? 3 : 2;
}

// CTA size and row feed before tuning: the configurations the autotuner keeps
// for 8192^2 FP32 grids on GB300 (9-point box at k = 8: 64-thread CTAs, 2354
// GStencil/s against 2256 with 128 threads and TMA rows, 2142 with 128 threads
// and cp.async rows; 13-point star at k = 3: 128 threads, cp.async 1271).  The
// TMA-fed ring is behind the cp.async ring elsewhere (5-point star at k = 6, 8:
// 2772 / 2924 against 2811 / 3050; 9-point box at k = 6 with 128 threads 2012
// against 2107; 13-point star at k = 2, 3, 4: 1060 / 1128 / 780 against 1223 /
// 1244 / 963), so it is never the default and the autotuner times both.
static int default_threads(int R, int star) {
    if (R == 1 && !star) return 64;
    return (R == 3 && !star) ? 256 : 128;
}
static const int kDefaultTma = 0;

// Plans whose rows the TMA-fed streaming kernel can load: FP32 storage, the
// zero rule (the copy engine's zero fill is the zero halo) and rows of a
// multiple of 16 bytes (the tensor map's row pitch).
static bool tma_eligible(const stencil_plan* p) {
    return p->dtype == STENCIL_F32 && p->boundary == STENCIL_BOUNDARY_ZERO && p->nx % 4 == 0;
}

static StreamKernelRef stream_tma_kernel(int R, int star, int k) {
    switch (R) {
        case 1: return get_stream_tma_kernel_r1(star, k);
        case 2: return get_stream_tma_kernel_r2(star, k);
        case 3: return get_stream_tma_kernel_r3(star, k);
        default: return {nullptr, 0};
    }
}

// The depth-`depth` streaming kernel (TMA-fed, VEC or element-wise variant),
// with its shared-memory attribute set on first use.
// `smem` receives the dynamic shared memory of a launch with CTAs of `nt`
// threads; the kernel's attribute allows the largest CTA.
static stencil_status_t stream_fn(stencil_plan* p, int depth, int vec, const void** fn, int* smem,
                                  int tma, int nt) {
    tma = tma && vec;
    StreamKernelRef r = tma ? stream_tma_kernel(p->R, p->star, depth)
                            : stream_kernel(p->R, p->star, depth, p->dtype, vec);
    if (!r.fn) return fail(STENCIL_ERR_UNSUPPORTED, "no streaming kernel for depth " + std::to_string(depth));
    *smem = stream_smem_bytes(p->R, depth, (int)p->elem, vec != 0, tma != 0, nt);
    const unsigned bit = 1u << (2 * depth + (vec ? 1 : 0) + (tma ? 16 : 0));
    if (!(p->smem_set & bit)) {
        CK(cudaFuncSetAttribute(r.fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                stream_smem_bytes(p->R, depth, (int)p->elem, vec != 0, tma != 0, kStreamMaxThreads)));
        p->smem_set |= bit;
    }
    *fn = r.fn;
    return STENCIL_OK;
}

// Tensor map of an FP32 grid for the TMA-fed streaming kernel: nx x ny
// elements, row pitch ld, boxes of kStreamTmaBox columns x 1 row, zero fill.
typedef CUresult (*TmaEncodeFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static TmaEncodeFn tma_encoder() {
    static TmaEncodeFn fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* ptr = nullptr;
        cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &ptr, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess && ptr)
            fn = reinterpret_cast<TmaEncodeFn>(ptr);
        else
            cudaGetLastError();
    });
    return fn;
}

static bool stream_tensor_map(CUtensorMap* map, const void* src, int64_t ny, int64_t nx) {
    TmaEncodeFn enc = tma_encoder();
    if (!enc || (uintptr_t)src % 16 != 0) return false;
    const cuuint64_t dims[2] = {(cuuint64_t)nx, (cuuint64_t)ny};
    const cuuint64_t strides[1] = {(cuuint64_t)nx * 4};
    const cuuint32_t box[2] = {(cuuint32_t)kStreamTmaBox, 1};
    const cuuint32_t estr[2] = {1, 1};
    return enc(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<void*>(src), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

static StreamKernelRef pad_kernel(const stencil_plan* p, int k) {
    return p->dtype == STENCIL_F32    ? get_stream_pad_kernel_f32(p->R, p->star, k)
           : p->dtype == STENCIL_BF16 ? get_stream_pad_kernel_bf16(p->R, p->star, k)
                                      : get_stream_pad_kernel_f16(p->R, p->star, k);
}

// One-warp tiles for the depth-8 launches of radius-1 plans that leave the
// streaming kernel's options alone.  Each SM holds 16 warps (8 at NC = 8) and the
// tiles are cut to one wave of them; a tile needs enough rows to pay for its 16
// halo rows.  Measured on GB300, 64 steps FP32 in us, one-warp tiles | CTA-wide:
// 5-point star 16384^2 (NC = 8) 3776 | 4764, 8192^2 1019 | 1252 (NC = 4: 1187),
// 4096^2 (64-row tiles, NC = 4; NC = 8: 389) 397 | 473, 3500^2 (47 rows) 317 |
// 338, 3000^2 (34 rows) 312 | 281; 9-point box 16384^2 6712 | 6901, 8192^2 1796 |
// 1827, 4096^2 561 | 576, 3500^2 439 | 445, 3000^2 476 | 363.
// NC = 8 needs widths that are a multiple of 8: where the right edge cuts a lane's
// chunk, the checks of those tiles set the time of the whole wave.  5-point star,
// NC = 8 | NC = 4 | CTA-wide: 8191 x 8188 1459 | 1260 | 1272, 6600 x 7012 1062 | 901 |
// 933, 16383^2 5668 | 5122 | 5468; BF16 8191^2 1428 | 1263 | 1375, 12000 x 9001 2154 |
// 1909 | 2108; periodic 8192 x 8188 1444 | 1307 | 1372.  16-bit storage gains as FP32
// does: BF16 4096^2 359 | 439 (star), 544 | 569 (box), 8192^2 955 | 1208, 1746 | 1799,
// periodic 1012 | 1225, 1768 | 1801, 4001 x 5003 459 | 528, 671 | 692.
static bool pad_eligible(const stencil_plan* p);
constexpr int kWarpDepth = 8;
constexpr int kWarpMinRows = 44;      // NC = 4, 5-point star
constexpr int kWarpMinRowsBox = 52;   // 9-point box (7000 x 1901, 49 rows, 544 | 526; 5200 x 2600, 52 rows, 486 | 491)
constexpr int kWarpMinRowsWide = 128;  // NC = 8: fewer warps, so taller tiles before it pays

struct WarpTiles {
    int bx, by, strips, tiles;
};

// One wave of one-warp tiles with nc columns per lane.
static WarpTiles warp_tiles(const stencil_plan* p, int nc) {
    const int64_t bx_max = 32 * nc - 2 * kWarpDepth;
    int64_t bx = ceil_div(ceil_div(p->nx, ceil_div(p->nx, bx_max)), nc) * nc;
    // (a last strip narrower than the halo columns does the same to the strip beside it as
    // a low last tile row, below: 9-point box, 64 steps, 8192 x 8180, 4 columns left over,
    // 2246 us, 8192 x 8184 1805; 5-point star 1457, 8192 x 8188 1255)
    while (bx > nc && bx < p->nx && p->nx % bx != 0 && p->nx % bx < kWarpDepth) bx -= nc;
    const int64_t strips = ceil_div(p->nx, bx);
    const int64_t warps = (int64_t)p->sms * (nc == 8 ? 8 : 16);
    int64_t by = ceil_div(p->ny, std::max<int64_t>(1, warps / strips));
    // A last tile row of fewer rows than a tile loads beyond its own puts the whole row of
    // tiles above it on the path that checks for the grid's edge, and those set the time
    // of the wave: 9-point box, 64 steps, 7192 x 2000 613 us with 10 rows left over, 7193 x
    // 2000 509 with 11.
    while (by < p->ny && p->ny % by != 0 && p->ny % by < kWarpDepth + 3) ++by;
    return {(int)bx, (int)by, (int)strips, (int)ceil_div(p->ny, by)};
}

static void configure_warp(stencil_plan* p, int threads_asked) {
    p->warp_nc = 0;
    const stencil_options_t& o = p->opt;
    const bool vec = p->nx % 4 == 0 || pad_eligible(p);
    if (p->R != 1 || p->k != kWarpDepth || p->tma || !vec || o.tb_depth > 0 || o.threads > 0 || o.tile_rows > 0 ||
        o.load != STENCIL_LOAD_AUTO || threads_asked != default_threads(p->R, p->star))
        return;
    for (int nc = p->star ? 8 : 4; nc >= 4; nc -= 4) {
        if (nc == 8 && p->nx % 8 != 0) continue;
        const WarpTiles t = warp_tiles(p, nc);
        if (t.by < (nc == 8 ? kWarpMinRowsWide : p->star ? kWarpMinRows : kWarpMinRowsBox)) continue;
        p->warp_nc = nc;
        p->warp_bx = t.bx;
        p->warp_by = t.by;
        p->warp_strips = t.strips;
        p->warp_tiles = t.tiles;
        return;
    }
}

// Plans whose ragged rows go through padded grids (see run_padded).
static bool pad_eligible(const stencil_plan* p) {
    return p->nx % 4 != 0 && p->boundary == STENCIL_BOUNDARY_ZERO && pad_kernel(p, 1).fn;
}

// Fill the streaming kernel's tile configuration for depth k and CTA size threads.
static stencil_status_t configure_stream(stencil_plan* p, int k, int threads, int tile_rows) {
    const int kmax = stream_kmax(p->R, p->star);
    if (k < 1 || k > kmax)
        return fail(STENCIL_ERR_UNSUPPORTED,
                    "tb_depth " + std::to_string(k) + " outside 1.." + std::to_string(kmax) +
                        " for radius " + std::to_string(p->R));
    k = stream_depth_at_most(p->R, p->star, k);
    if (threads < 32 || threads > kStreamMaxThreads || threads % 32)
        return fail(STENCIL_ERR_INVALID_ARG, "threads must be a multiple of 32 in 32..256");
    const int vec = p->nx % 4 == 0 || pad_eligible(p);
    const int H = (p->R * k + 3) / 4 * 4;
    const int bx_max = 4 * threads - 2 * H;
    if (bx_max < 4) return fail(STENCIL_ERR_UNSUPPORTED, "CTA too narrow for this depth");
    const int64_t strips = ceil_div(p->nx, bx_max);
    const int bx = (int)(ceil_div(ceil_div(p->nx, strips), 4) * 4);
    const int nt = (int)(ceil_div(ceil_div(bx + 2 * H, 4), 32) * 32);
    const void* fn = nullptr;
    int smem = 0;
    stencil_status_t st = stream_fn(p, k, vec, &fn, &smem, p->tma, nt);
    if (st != STENCIL_OK) return st;
    int per_sm = 0;
    CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, nt, smem));
    if (per_sm < 1) return fail(STENCIL_ERR_UNSUPPORTED, "streaming kernel does not fit on an SM");
    int64_t tiles_y;
    int by;
    if (tile_rows > 0) {
        by = tile_rows;
        tiles_y = ceil_div(p->ny, by);
    } else {
        const int64_t resident = (int64_t)per_sm * p->sms;
        const int64_t by_min = std::max<int64_t>(8, 4LL * p->R * k);
        const int64_t want = std::max<int64_t>(1, resident / strips);
        tiles_y = std::max<int64_t>(1, std::min<int64_t>(want, ceil_div(p->ny, by_min)));
        by = (int)ceil_div(p->ny, tiles_y);
        tiles_y = ceil_div(p->ny, by);
    }
    if (strips * tiles_y > 0x7fffffffLL) return fail(STENCIL_ERR_UNSUPPORTED, "grid too large");
    p->kernel = STENCIL_KERNEL_STREAM;
    p->grid_on = 0;
    p->tiles_on = 0;
    p->k = k;
    p->threads = nt;
    p->H = H;
    p->bx = bx;
    p->by = by;
    p->strips = (int)strips;
    p->tiles_y = (int)tiles_y;
    p->smem = smem;
    p->per_sm = per_sm;
    configure_warp(p, threads);
    return STENCIL_OK;
}

// Default N of one tcgen05 MMA per operand type (BF16, TF32), and whether
// that engine is the default for the tensor-core kernel family (kernel = TC or
// AUTO without autotuning).  Measured on GB300, 16384^2 Box-49, 200 steps:
// BF16 tcgen05 N = 64 916 GStencil/s (N = 32: 856, N = 16: 614; three or four
// weight rows per MMA, N = 96: 784, N = 128: 596) against 708 for the warp-MMA
// engine; TF32 tcgen05 N = 96 547 (N = 32: 492, N = 16: 417, N = 128: 457)
// against 421.  Autotuning times both engines and every width.
static const int kUmmaDefaultN[2] = {64, 96};
// MMA widths of the tcgen05 kernels: N = 16, 32, 64 with one weight row per
// MMA; N = 96 and 128 stack three or four weight rows over 32-column N-tiles.
static const int kUmmaWidths[5] = {16, 32, 64, 96, 128};
static const int kUmmaPreferred[2] = {1, 1};

// The tcgen05 engine (box49_umma.cu) takes zero-boundary grids whose storage is
// the MMA operand type (BF16 storage for TC_BF16, FP32 for TC_TF32), with
// 16-byte aligned rows and at least one full staged tile.  With TF32 the first
// launch of a run stays on the warp-MMA engine, which rounds the caller's
// input (and every output but the last) to TF32.  kernel = TC_UMMA makes the
// engine mandatory, TC_WARP switches it off.  p->umma_ok collects the usable
// MMA widths (bit n / 16), p->umma_n the one in use (0: warp-MMA engine).
static stencil_status_t configure_umma(stencil_plan* p) {
    p->umma_n = 0;
    p->umma_ok = 0;
    const int want = p->opt.kernel;
    if (want == STENCIL_KERNEL_TC_WARP) return STENCIL_OK;
    const int tf32 = p->compute == STENCIL_COMPUTE_TC_TF32;
    const char* why = nullptr;
    if (p->compute == STENCIL_COMPUTE_TC_3XTF32) why = "the tcgen05 engine runs TF32 and BF16 operands only";
    else if (p->boundary != STENCIL_BOUNDARY_ZERO) why = "the tcgen05 engine takes zero-boundary grids";
    else if (tf32 ? p->dtype != STENCIL_F32 : p->dtype != STENCIL_BF16)
        why = "the tcgen05 engine needs FP32 storage for TF32 and BF16 storage for BF16";
    else if ((p->nx * (int64_t)p->elem) % 16 != 0) why = "the tcgen05 engine needs rows of a multiple of 16 bytes";
    else if (p->ny < 134 || p->nx < 128) why = "the tcgen05 engine needs ny >= 134 and nx >= 128";
    else if (p->opt.mma_n > 0 && !get_box49_umma_kernel(tf32, p->opt.mma_n))
        why = "no tcgen05 kernel for this mma_n (BF16: 16, 32, 64, 96, 128; TF32: 16, 32, 96, 128)";
    if (!why) {
        for (int nt : kUmmaWidths) {
            if (p->opt.mma_n > 0 && nt != p->opt.mma_n) continue;
            const void* fn = get_box49_umma_kernel(tf32, nt);
            if (!fn) continue;
            const int smem = box49_umma_smem_bytes(tf32, nt);
            CK(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
            int per_sm = 0;
            CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, box49_umma_threads(nt), smem));
            if (per_sm >= 1) p->umma_ok |= 1 << (nt / 16);
        }
        if (!p->umma_ok) why = "the tcgen05 kernel does not fit an SM";
    }
    if (why) {
        if (want == STENCIL_KERNEL_TC_UMMA) return fail(STENCIL_ERR_UNSUPPORTED, why);
        return STENCIL_OK;
    }
    // One CTA per SM: each holds 256 (one weight row per MMA) or 512 (row
    // groups) tensor-memory columns for its whole life.
    p->umma_ctas = (int)std::min<int64_t>((int64_t)p->sms, (int64_t)p->strips * p->tiles_y);
    const int nt = p->opt.mma_n > 0 ? p->opt.mma_n : kUmmaDefaultN[tf32];
    if (want == STENCIL_KERNEL_TC_UMMA || kUmmaPreferred[tf32]) p->umma_n = (p->umma_ok >> (nt / 16)) & 1 ? nt : 0;
    if (want == STENCIL_KERNEL_TC_UMMA && !p->umma_n) return fail(STENCIL_ERR_UNSUPPORTED, "tcgen05 kernel unusable");
    // The phase kernel (box49_phase.cu) takes rows in groups of four.  It is the
    // default wherever it applies: us per step, phase | kUmmaDefaultN above, BF16
    // 512^2 12.5 | 16.5, 2048^2 12.4 | 18.6, 4096^2 21.5 | 31.8, 16384^2 209.5 |
    // 293.2; TF32 12.3 | 16.0, 14.8 | 18.4, 32.4 | 43.7, 390 | 509.
    p->phase_ok = p->phase = 0;
    if (p->opt.mma_n == 0 && p->umma_n && p->ny % 4 == 0) {
        const void* fn = get_box49_phase_kernel(tf32);
        const int smem = box49_phase_smem_bytes(tf32);
        int per_sm = 0;
        CK(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
        CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, box49_umma_threads(0), smem));
        const int64_t tiles = ceil_div(p->ny, box49_phase_rows()) * ceil_div(p->nx, box49_phase_cols(tf32));
        p->phase_ok = per_sm >= 1;
        p->phase_ctas = (int)std::min<int64_t>(p->sms, tiles);
        p->phase = p->phase_ok;
    }
    p->kernel = p->umma_n ? STENCIL_KERNEL_TC_UMMA : STENCIL_KERNEL_TC;
    return STENCIL_OK;
}

static stencil_status_t configure_tc(stencil_plan* p) {
    if (p->R != 3) return fail(STENCIL_ERR_UNSUPPORTED, "tensor-core engines need radius 3 (7x7 weights)");
    if (p->dtype == STENCIL_F16) return fail(STENCIL_ERR_UNSUPPORTED, "tensor-core engines take FP32 or BF16 storage");
    const int engine = p->compute == STENCIL_COMPUTE_TC_BF16 ? 1 : p->compute == STENCIL_COMPUTE_TC_3XTF32 ? 2 : 0;
    if (engine == 2 && p->dtype != STENCIL_F32)
        return fail(STENCIL_ERR_UNSUPPORTED, "3xTF32 splits FP32 values: it takes FP32 storage");
    p->naive = get_box49_tc_kernel(p->dtype, engine);
    if (!p->naive) return fail(STENCIL_ERR_UNSUPPORTED, "no tensor-core kernel for this dtype");
    p->kernel = STENCIL_KERNEL_TC;
    p->k = 1;
    p->threads = 256;
    p->H = 3;
    p->bx = 128;
    p->by = 128;
    p->strips = (int)ceil_div(p->nx, 128);
    p->tiles_y = (int)ceil_div(p->ny, 128);
    p->smem = box49_tc_smem_bytes(engine);
    CK(cudaFuncSetAttribute(p->naive, cudaFuncAttributeMaxDynamicSharedMemorySize, p->smem));
    p->tc_pipe = p->nx % 4 == 0 ? get_box49_tc_pipe_kernel(p->dtype, engine) : nullptr;
    if (p->tc_pipe) {
        p->tc_pipe_smem = 2 * p->smem;
        CK(cudaFuncSetAttribute(p->tc_pipe, cudaFuncAttributeMaxDynamicSharedMemorySize, p->tc_pipe_smem));
        int per_sm = 0;
        CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, p->tc_pipe, 256, p->tc_pipe_smem));
        if (per_sm < 1) {
            p->tc_pipe = nullptr;
        } else {
            p->tc_pipe_ctas = (int)std::min<int64_t>((int64_t)per_sm * p->sms, (int64_t)p->strips * p->tiles_y);
        }
    }
    return configure_umma(p);
}

// The cluster-resident kernel holds the grid in the shared memory of one
// cluster of C <= 16 CTAs and runs a whole run in one launch.  It applies when
// some C in {1, 2, 4, 8, 16} gives slabs that fit a CTA's shared memory and
// are at least R rows high (periodic grids also need nx >= R), and the
// cluster can be scheduled.  Sets p->res_ok (bit log2 C per usable C) and
// returns the largest usable C, or 0.
static int resident_candidates(stencil_plan* p, int kb = 1) {
    p->res_ok = 0;
    if (p->compute != STENCIL_COMPUTE_FP32) return 0;
    const int periodic = p->boundary == STENCIL_BOUNDARY_PERIODIC;
    if (periodic && p->nx < p->R) return 0;
    if (p->ny > (1 << 20) || p->nx > (1 << 20)) return 0;
    const void* fn = get_resident_kernel(p->R, p->star, p->dtype);
    if (!fn) return 0;
    int max_smem = 0;
    if (cudaDeviceGetAttribute(&max_smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, p->device) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    p->res_max_smem = max_smem;
    int best = 0;
    for (int C = 1; C <= resident_max_cluster(); C *= 2) {
        int rp = 0;
        const int smem = resident_config((int)p->ny, (int)p->nx, p->R, periodic, C, kb, max_smem, &rp);
        if (smem < 0) continue;
        if (!resident_cluster_fits(fn, C, smem, max_smem)) continue;
        int lg = 0;
        while ((1 << lg) < C) ++lg;
        p->res_ok |= 1 << lg;
        best = C;
    }
    p->res_fn = fn;
    return best;
}

// Switch the plan to the resident kernel with cluster size C and kb steps per
// halo exchange (kb = 1 by default: deeper blocking only pays where a step's
// work is small next to the cluster barrier, which autotuning measures).
static stencil_status_t use_resident(stencil_plan* p, int C, int kb = 1) {
    const int periodic = p->boundary == STENCIL_BOUNDARY_PERIODIC;
    int rp = 0;
    const int smem = resident_config((int)p->ny, (int)p->nx, p->R, periodic, C, kb, p->res_max_smem, &rp);
    if (smem < 0) return fail(STENCIL_ERR_UNSUPPORTED, "grid does not fit the cluster-resident kernel");
    // (the kernel's limit, which all plans share: the largest any of them may need)
    CK(cudaFuncSetAttribute(p->res_fn, cudaFuncAttributeMaxDynamicSharedMemorySize, p->res_max_smem));
    if (C > 8) CK(cudaFuncSetAttribute(p->res_fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    p->kernel = STENCIL_KERNEL_RESIDENT;
    p->grid_on = 0;
    p->res_c = C;
    p->res_rp = rp;
    p->res_kb = kb;
    p->res_smem = smem;
    return STENCIL_OK;
}

// The chip-resident register-tile kernel: one tile per SM over the whole chip.
// AUTO takes it wherever a configuration fits, in place of the cluster-resident
// kernel (at most 16 SMs) and of the streaming kernel (launches).  It was the
// faster one at every size it takes, from a 4-step run on: 96 steps in us,
// register tiles | streaming kernel, FP32 on GB300: 5-point star 300^2 47 | 235,
// 1000^2 83 | 248, 1500^2 (about the largest) 151 | 273; 9-point box 57 | 298,
// 111 | 322, 212 | 371; 13-point star 97 | 658, 211 | 658, 1400^2 423 | 725; 7x7
// box 183 | 1478, 433 | 1379, 1400^2 743 | 1575; 4 steps 11-38 | 16-67.  Against
// the cluster-resident kernel: 512^2 5-point star, 100 steps, 52 | 219 (FP32);
// 130 x 517 13-point star, 20 steps, 24 | 74.  (Shorter runs and periodic ragged widths:
// cluster_run below.)  That is one run at a time: tiles use every SM, so eight or more
// small plans on streams of their own ran up to twice as fast in one cluster each (9-point
// box 256^2, 100 steps, us per run with 1, 4, 8 plans: 55 | 116, 36 | 30, 36 | 19).  A plan the caller steers (kernel,
// tb_depth, threads, tile_rows or load set) keeps what it asked for.
static bool grid_candidate(stencil_plan* p) {
    if (p->compute != STENCIL_COMPUTE_FP32 || p->ny > (1 << 20) || p->nx > (1 << 20)) return false;
    int coop = 0;
    if (cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, p->device) != cudaSuccess || !coop) {
        cudaGetLastError();
        return false;
    }
    const int periodic = p->boundary == STENCIL_BOUNDARY_PERIODIC;
    if (!grid_config((int)p->ny, (int)p->nx, p->R, p->star, periodic, p->sms, 0, 0, &p->grid)) return false;
    // the cluster-resident kernel's bits where AUTO would otherwise take that kernel
    const int C = resident_candidates(p);
    p->grid.plain = C > 0;
    // (boxes of radius 2 and 3 of up to about 140^2 points, where each tile is mostly
    // halo, stay with it: 96 x 100, 7x7 100 steps 129 us against 164, 5x5 16 steps 21
    // against 22; at 160^2 it is 1.2 and 1.3 times as slow, at 400^2 2.4 and 2.6)
    // 16-bit storage: the streaming kernel rounds once per launch, which adds up over a
    // long run; grids that it takes keep its roundings
    if (p->dtype != STENCIL_F32 && !p->grid.plain) return false;
    if (p->grid.plain && p->R >= 2 && !p->star && p->ny * p->nx <= 20000) return false;
    p->grid_ok = grid_fits(p->grid, p->R, p->star, p->sms);
    if (p->grid_ok && C > 0 && use_resident(p, C) != STENCIL_OK) p->res_c = 0;  // (for cluster_run)
    return p->grid_ok != 0;
}

// Grids too large for one register tile per SM: the same tiles as launches of up
// to tiles.k steps, two or three waves of them, in place of the streaming
// kernel's launches.  Between the register tiles' limit and about 2048^2 the
// streaming kernel has too few rows per tile: a launch is 15-20 us of pipeline
// fill and halo rows.  48 steps in us, register tiles | streaming kernel, FP32,
// zero rule, GB300:
//   1600^2       5-point star 108 | 138  9-point box 152 | 188  9-point star 176 | 274
//                5x5 box 324 | 519  13-point star 244 | 401  7x7 box 594 | 790
//   2048^2       141 | 176  208 | 187  249 | 348  597 | 741  362 | 528  828 | 1140
//   2304^2       176 | 175  275 | 224  323 | 348  619 | 741  463 | 561  1036 | 1235
//   1024 x 4096  166 | 140  224 | 187  258 | 289  540 | 716  373 | 495  862 | 1137
//   4096 x 1024  141 | 163  193 | 224  259 | 322  541 | 742  373 | 560  840 | 1441
//   2001 x 2003  176 | 187  225 | 220  311 | 383  545 | 778  449 | 636  1037 | 1232
// (above 2400^2 the streaming kernel is the faster one: 3000^2 321 |
// 212 ... 1629 | 1479).  So: up to 4.3 M points (radius 1: 3.3 M for stars, whose
// runs of a few launches gain nothing above: 1900 x 2000, 16 steps 54 | 46; 2.8 M
// for boxes), and for radius 1 no grids much wider than high, which the streaming
// kernel covers with fewer halo rows.  Periodic rows that are not a multiple of 4 wide, which
// the streaming kernel must load element by element through the wrap in every
// launch, take the tiles at every size: 2001 x 2003 186 | 643 ... 1673 | 2742,
// 4001 x 5003 719 | 1415 ... 4198 | 6094, 9001 x 8003 2611 | 4408 ... 14997 |
// 18195.
static void choose_tiles(stencil_plan* p) {
    // (16-bit storage rounds once per launch, so its results depend on the depth)
    if (p->dtype != STENCIL_F32 || p->ny > (1 << 20) || p->nx > (1 << 20)) return;
    const int periodic = p->boundary == STENCIL_BOUNDARY_PERIODIC;
    const double points = (double)p->ny * (double)p->nx;
    if (!(periodic && p->nx % 4 != 0)) {
        if (points > (p->R > 1 ? 4.3e6 : p->star ? 3.3e6 : 2.8e6)) return;
        if (p->R == 1 && p->nx > 1.5 * p->ny) return;
    }
    if (!tiles_config((int)p->ny, (int)p->nx, p->R, p->star, periodic, p->sms, 2, &p->tiles)) return;
    p->tiles_ok = p->tiles_on = grid_fits(p->tiles, p->R, p->star, 0);
    if (p->tiles_on) p->warp_nc = 0;
}

// Whether a launch of nlev steps runs as register tiles.  Launches of a step or two
// (a short run, or a run's remainder), and for the 5-point star every depth below 8
// that the streaming kernel has as one launch, are cheaper without the tiles' deep
// halo.  Zero rule, among others, us as tiles | streaming: 5-point star 1600^2 3 steps
// 16.5 | 14.4, 4 17.5 | 16.6, 5 (4 + 1) 18.6 | 28.5, 6 20.7 | 18.6, 8 22.7 | 22.7; 1833 x
// 1459 1 step 18.4 | 14.6, 2 19.2 | 14.5, 3 20.7 | 16.5, 6 26.0 | 22.7, 8 28.9 | 34.7;
// 9-point box 1833 x 1459 1 14.5 | 13.6, 2 16.6 | 14.5, 3 18.6 | 18.6, 4 20.7 | 22.7;
// 9-point star 1 18.6 | 16.5, 2 21.3 | 22.6; 5x5 box 1800 x 2047 1 24.6 | 17.3, 2 29.7 |
// 23.7, 3 35.5 | 42.3 (1833 x 1459 2 22.7 | 22.9); 13-point star 1833 x 1459 1 20.0 |
// 16.5, 2 22.7 | 20.6, 3 26.4 | 33.5; 7x7 box 1 27.5 | 26.7, 2 37.2 | 44.5.  Aligned
// 2048^2: 1 step, 13-point star 19 | 15, 7x7 box 27 | 25; 2 steps 23 | 17, 42 | 48.
// (Element-wise launches of the 9-point box and of radius 2 gain as whole runs only:
// behind launches of tiles, 1833 x 1459, 8 + 1 steps, 9-point box 43.1 | 45.2, 5x5 box
// 4 + 1 51.3 | 53.4.)  Periodic ragged launches stay tiles (see choose_tiles).
static bool tiles_launch(const stencil_plan* p, int nlev, bool vec, bool whole_run) {
    if (!p->tiles_on) return false;
    // (a full launch of a long run, or no streaming launch of that depth in the plan)
    if ((nlev > 2 && nlev == p->tiles.k) || nlev > p->k || stream_depth_at_most(p->R, p->star, nlev) != nlev) return true;
    if (vec) return nlev > (p->R == 1 && p->star ? 6 : p->star ? 2 : 1);
    if (p->boundary == STENCIL_BOUNDARY_PERIODIC) return true;
    if ((p->R == 2 || (p->R == 1 && !p->star)) && !whole_run) return true;
    return nlev > (p->R == 1 ? (p->star ? 6 : 2) : p->R == 2 ? (p->star ? 1 : 2) : p->star ? 2 : 1);
}

static void use_grid(stencil_plan* p) {
    p->kernel = STENCIL_KERNEL_RESIDENT;
    p->grid_on = 1;
}

// Register-tile plans in the cluster-resident kernel's order keep that kernel
// configured: the bits are the same, so each run takes the faster of the two.
//
// One step: the cooperative launch and its end cost ~2 us more than the cluster's, and
// in place, where a tile may not write before its neighbours have read, the tiles copy
// the input first (two steps: they exchange after the first).  In us, alone and among
// others, register tiles | cluster: 5-point star 64^2 16.4 / 6.3 | 14.8 / 5.2, 9-point
// box 140 x 141 17.7 / 8.2 | 14.4 / 6.3, 13-point star 300 x 110 17.7 / 8.3 | 16.6 / 6.5,
// 200^2 even; in place, among others, 5-point star 200 x 201 12.1 | 6.9, 256^2 10.4 |
// 8.3, 300^2 11.4 | 9.4, 7x7 box 300^2 12.4 | 12.4; two steps in place 260 x 161 10.4 |
// 8.4, 300 x 201 10.4 | 9.2, 200^2 8.8 | 8.3.
//
// 7x7 boxes on narrow grids, of which a strip holds little but halo, 100 steps: 256 x 96
// 159 | 154, 400 x 64 160 | 154, 700 x 40 191 | 163, 200 x 128 155 | 158, 800 x 64 188 | 214.
//
// Periodic ragged widths: the tiles read their halos element by element through the
// wrap, twice the cost of an exchange, and the more of a tile is halo the worse.
// 100 steps, register tiles | cluster: 13-point star 60 x 61 192 | 131, 300 x 110
// 238 | 183, 250 x 251 245 | 216, 300 x 301 290 | 342; 7x7 box 300 x 110 390 | 211,
// 300 x 201 387 | 271, 300 x 301 395 | 462; 5x5 box 300 x 110 267 | 164, 250 x 251
// 215 | 193; 9-point star 141^2 152 | 138, 200 x 201 183 | 190; 9-point box 100 x 99
// 132 | 118, 200 x 201 143 | 197; 5-point star always fewer as tiles, but for short
// runs: 2 steps 300 x 110 19.7 / 10.3 | 17.9 / 8.4, 3 steps 141^2 18.8 / 10.4 | 19.4 /
// 8.4, 1 step 250 x 251 20.5 / 10.4 | 18.6 / 9.0.  Flat grids give the cluster's CTAs
// few rows each: 50 x 403, 13-point star, 100 steps 171 | 221.
static bool cluster_run(const stencil_plan* p, int64_t T, bool in_place) {
    if (!p->grid.plain || p->res_c == 0) return false;
    const int64_t points = p->ny * p->nx;
    const bool ragged = p->nx % 4 != 0;
    if (in_place && (T == 1 || (T == 2 && ragged)) && points <= (T == 1 ? 90000 : 60000)) return true;
    if (ragged && p->boundary == STENCIL_BOUNDARY_PERIODIC) {
        if (p->nx > 4 * p->ny) return false;
        const int64_t any = p->R == 1 ? (p->star ? 0 : 15000) : p->R == 2 && p->star ? 36000 : 65000;
        return points <= std::max<int64_t>(any, T == 1 ? 65000 : T == 2 ? 36000 : T == 3 ? 20000 : 0);
    }
    if (p->R == 3 && !p->star && points <= 28000 && p->nx <= 112) return true;
    return T == 1 && points <= (ragged ? 60000 : p->R == 1 ? 36000 : 20000);
}

static stencil_status_t configure_naive(stencil_plan* p) {
    p->naive = get_naive_kernel(p->R, p->dtype);
    if (!p->naive) return fail(STENCIL_ERR_UNSUPPORTED, "no naive kernel for this radius");
    p->kernel = STENCIL_KERNEL_NAIVE;
    p->k = 1;
    p->threads = 256;
    p->H = 0;
    p->bx = 32;
    p->by = 8;
    p->strips = (int)ceil_div(p->nx, 32);
    p->tiles_y = (int)std::min<int64_t>(ceil_div(p->ny, 8), 65535);
    p->smem = 0;
    return STENCIL_OK;
}

// Separable form (compute = LOWRANK): factor the weights, one step per launch.
static stencil_status_t configure_lowrank(stencil_plan* p) {
    if (p->dtype != STENCIL_F32) return fail(STENCIL_ERR_UNSUPPORTED, "the low-rank form takes FP32 storage");
    if (p->opt.kernel != STENCIL_KERNEL_AUTO)
        return fail(STENCIL_ERR_UNSUPPORTED, "the low-rank form has its own kernel (kernel must be AUTO)");
    p->lr_rank = lowrank_factor(p->w.w, p->R, p->opt.rank, p->lr_col, p->lr_row, nullptr);
    if (p->lr_rank < 1) p->lr_rank = 1;  // all-zero weights: one zero term
    p->lr_fn = get_lowrank_kernel(p->R, p->lr_rank);
    if (!p->lr_fn) return fail(STENCIL_ERR_UNSUPPORTED, "no low-rank kernel for this rank");
    p->kernel = STENCIL_KERNEL_LOWRANK;
    p->k = 1;
    p->threads = 128;
    p->H = p->R;
    p->bx = 128;
    p->strips = (int)ceil_div(p->nx, 128);
    p->tiles_y = 1;
    p->by = (int)p->ny;
    p->smem = 0;
    return STENCIL_OK;
}

// A streaming launch's parameters except its grids, pitches and alignment.
static StreamParams stream_params(const stencil_plan* p, int nlev) {
    StreamParams sp{};
    sp.ny = p->ny;
    sp.nx = p->nx;
    sp.ld = sp.ld_out = p->nx;
    sp.nlev = nlev;
    sp.H = p->H;
    sp.bx = p->bx;
    sp.by = p->by;
    sp.strips = p->strips;
    sp.periodic = p->boundary == STENCIL_BOUNDARY_PERIODIC;
    sp.w = p->w;
    for (int i = 0; i < kMaxTaps; ++i) sp.w2.w2[i] = make_float2(p->w.w[i], p->w.w[i]);
    sp.status = p->status;
    sp.wait_ns = (long long)(p->opt.timeout_ms > 0 ? p->opt.timeout_ms : 2000) * 1000000LL;
    sp.debug_withhold = p->opt.debug_withhold;
    return sp;
}

// The launch as one-warp tiles (sp: grids and pitches set).
static stencil_status_t launch_warp(stencil_plan* p, StreamParams& sp, cudaStream_t st) {
    sp.H = kWarpDepth;
    sp.bx = p->warp_bx;
    sp.by = p->warp_by;
    sp.strips = p->warp_strips;
    void* args[] = {&sp};
    CK(cudaLaunchKernel(get_warp_kernel(p->star, p->dtype, p->warp_nc), dim3((unsigned)(p->warp_strips * p->warp_tiles)),
                        dim3(32), args, 0, st));
    return STENCIL_OK;
}

// One launch advancing `nlev` steps from src to dst.  `first` / `last`: this
// launch starts / ends a run (the pipelined TF32 engine rounds its input on
// the first launch and keeps intermediate states TF32-rounded until the last).
static stencil_status_t launch_once(stencil_plan* p, const void* src, void* dst, int nlev,
                                    cudaStream_t st, int first = 1, int last = 1) {
    if (p->kernel == STENCIL_KERNEL_TC || p->kernel == STENCIL_KERNEL_TC_UMMA) {
        TcParams tp{};
        tp.in = src;
        tp.out = dst;
        tp.ny = (int)p->ny;
        tp.nx = (int)p->nx;
        tp.ld = (int)p->nx;
        tp.periodic = p->boundary == STENCIL_BOUNDARY_PERIODIC;
        tp.tiles_x = p->strips;
        tp.tiles = p->strips * p->tiles_y;
        tp.vec = (p->nx % 4 == 0) && ((uintptr_t)src % (4 * p->elem) == 0) &&
                 ((uintptr_t)dst % (4 * p->elem) == 0);
        tp.convert_in = first;
        tp.round_out = !last;
        for (int i = 0; i < 49; ++i) tp.w[i] = p->w.w[i];
        const int tf32 = p->compute == STENCIL_COMPUTE_TC_TF32;
        if (p->umma_n && !(tf32 && first) && (uintptr_t)src % 16 == 0 && (uintptr_t)dst % 16 == 0) {
            const cudaError_t e =
                p->phase ? launch_box49_phase(tf32, src, dst, tp.ny, tp.nx, tf32 && !last, p->status, p->w.w,
                                              p->phase_ctas, st, p->opt.timeout_ms, p->opt.debug_withhold)
                         : launch_box49_umma(tf32, p->umma_n, src, dst, tp.ny, tp.nx, tp.ld,
                                                    tf32 && !last, p->status, p->w.w, p->umma_ctas, st,
                                                    p->opt.timeout_ms, p->opt.debug_withhold);
            if (e == cudaSuccess) return STENCIL_OK;
            if (e != cudaErrorNotSupported) CK(e);
            // no tensor map for this layout: the warp-MMA engine takes the step
        }
        void* args[] = {&tp};
        if (p->tc_pipe && tp.vec) {
            CK(cudaLaunchKernel(p->tc_pipe, dim3((unsigned)p->tc_pipe_ctas), dim3(256), args,
                                (size_t)p->tc_pipe_smem, st));
        } else {
            CK(cudaLaunchKernel(p->naive, dim3((unsigned)tp.tiles), dim3(256), args, (size_t)p->smem, st));
        }
        return STENCIL_OK;
    }
    if (p->kernel == STENCIL_KERNEL_RESIDENT && p->grid_on && !cluster_run(p, nlev, src == dst)) {
        const size_t vec_bytes = 4 * p->elem;
        const int vec = p->nx % 4 == 0 && (uintptr_t)src % vec_bytes == 0 && (uintptr_t)dst % vec_bytes == 0;
        // In place, a tile may only write once its neighbours have read: at least
        // one exchange (a single step in place is staged by the caller).
        int k = p->grid.k;
        if (src == dst) k = std::min(k, (nlev + 1) / 2);
        const cudaError_t e =
            launch_grid(p->grid, p->R, p->star, p->dtype, p->boundary == STENCIL_BOUNDARY_PERIODIC, src, dst,
                        (int)p->ny, (int)p->nx, vec, nlev, k, p->grid_mem, p->status,
                        (long long)(p->opt.timeout_ms > 0 ? p->opt.timeout_ms : 2000) * 1000000LL,
                        p->opt.debug_withhold, p->w, st);
        if (e == cudaErrorCooperativeLaunchTooLarge) {  // fewer SMs than the device reports (a partition)
            cudaGetLastError();
            p->grid_on = p->grid_ok = 0;
            p->kernel = STENCIL_KERNEL_STREAM;
            const int C = p->grid.plain ? resident_candidates(p) : 0;  // (the kernel the tiles stood in for)
            if (C > 0) use_resident(p, C);
            return fail(STENCIL_ERR_UNSUPPORTED, "the chip-resident tiles do not fit at once");
        }
        CK(e);
        return STENCIL_OK;
    }
    if (p->kernel == STENCIL_KERNEL_RESIDENT) {
        ResidentParams rp{};
        rp.in = src;
        rp.out = dst;
        rp.ny = (int)p->ny;
        rp.nx = (int)p->nx;
        rp.ld = (int)p->nx;
        rp.T = nlev;
        rp.periodic = p->boundary == STENCIL_BOUNDARY_PERIODIC;
        rp.rp = p->res_rp;
        rp.pitch = (int)p->nx + 2 * p->R;
        rp.kb = p->res_kb;
        rp.H = p->res_kb * p->R;
        rp.w = p->w;
        CK(launch_resident(p->res_fn, p->res_c, p->res_smem, rp, st));
        return STENCIL_OK;
    }
    if (p->kernel == STENCIL_KERNEL_LOWRANK) {
        CK(launch_lowrank(p->lr_fn, static_cast<const float*>(src), static_cast<float*>(dst), p->ny, p->nx,
                          p->boundary == STENCIL_BOUNDARY_PERIODIC, p->lr_col, p->lr_row, p->sms, st));
        return STENCIL_OK;
    }
    if (p->kernel == STENCIL_KERNEL_NAIVE) {
        dim3 block(32, 8), grid((unsigned)p->strips, (unsigned)p->tiles_y);
        long long ny = p->ny, nx = p->nx;
        int periodic = p->boundary;
        void* args[] = {(void*)&src, (void*)&dst, &ny, &nx, &periodic, &p->w};
        CK(cudaLaunchKernel(p->naive, grid, block, args, 0, st));
        return STENCIL_OK;
    }
    StreamParams sp = stream_params(p, nlev);
    sp.in = src;
    sp.out = dst;
    const size_t vec_bytes = 4 * p->elem;
    sp.vec = (p->nx % 4 == 0) && ((uintptr_t)src % vec_bytes == 0) &&
             ((uintptr_t)dst % vec_bytes == 0);
    if (tiles_launch(p, nlev, sp.vec, first && last)) {
        CK(launch_tiles(p->tiles, p->R, p->star, p->dtype, sp.periodic, src, dst, (int)p->ny, (int)p->nx, sp.vec, nlev,
                        p->w, st));
        return STENCIL_OK;
    }
    if (p->warp_nc && nlev == kWarpDepth && sp.vec) return launch_warp(p, sp, st);
    dim3 grid((unsigned)(p->strips * p->tiles_y)), block((unsigned)p->threads);
    const void* fn = nullptr;
    int smem = 0;
    alignas(64) CUtensorMap map;
    // The TMA-fed kernel when the plan uses it and this source has a tensor
    // map (16-byte aligned); otherwise the cp.async kernel, same arithmetic.
    const int tma = p->tma && sp.vec && stream_tensor_map(&map, src, p->ny, p->nx);
    stencil_status_t s = stream_fn(p, nlev, sp.vec, &fn, &smem, tma, p->threads);
    if (s != STENCIL_OK) return s;
    if (tma) {
        void* args[] = {&map, &sp};
        CK(cudaLaunchKernel(fn, grid, block, args, (size_t)smem, st));
    } else {
        void* args[] = {&sp};
        CK(cudaLaunchKernel(fn, grid, block, args, (size_t)smem, st));
    }
    return STENCIL_OK;
}

// ---- padded rows for ragged widths ---------------------------------------------------
//
// A width that is not a multiple of 4 leaves the rows of a dense grid unaligned,
// and the streaming kernel then loads and stores them element by element.
// Runs of the zero rule go through two plan-owned grids of padded rows instead:
// one pass copies the input, every launch streams 16-byte chunks, and only
// the last one stores element by element into the caller's grid.  (Periodic
// rows cannot be padded: a wrapped chunk would read the padding.)  Measured on
// GB300, 64 steps, us padded | element-wise: 4001 x 5003 5-point star FP32 540 |
// 809, BF16 519 | 849; 9-point box 706 | 871, 683 | 1030; 13-point star 1622 |
// 2242, 1567 | 2241; 5x5 box BF16 2353 | 2512.  The FP32 boxes of radius 2 and the
// 7x7 boxes are bound by arithmetic either way and keep the dense grids (5x5 FP32
// 1600 x 1701 830 | 777; 7x7 FP32 4001 x 5003 3512 | 3233; 7x7 BF16 4001 x 5003 3568 |
// 3724, but 3001 x 2053, 400 steps, 13145 | 11525).

constexpr int kPadElems = 16;  // pitch granularity

template <typename TW>
__global__ void __launch_bounds__(256)
    pad_rows_kernel(const TW* __restrict__ in, TW* __restrict__ out, int64_t ny, int64_t nx, int64_t ld) {
    // one thread per 4 columns; the padding is written as zeros
    const int64_t chunks = ld / 4, n = ny * chunks;
    for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < n; i += (int64_t)gridDim.x * 256) {
        const int64_t y = i / chunks, x = (i - y * chunks) * 4;
        const TW* row = in + y * nx;
        alignas(4 * sizeof(TW)) TW v[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) v[e] = x + e < nx ? row[x + e] : TW(0);
        if constexpr (sizeof(TW) == 4)
            *reinterpret_cast<uint4*>(out + y * ld + x) = *reinterpret_cast<uint4*>(v);
        else
            *reinterpret_cast<uint2*>(out + y * ld + x) = *reinterpret_cast<uint2*>(v);
    }
}

// One launch from a padded grid to the other, or (dense) to the caller's grid.
static stencil_status_t launch_padded(stencil_plan* p, const void* src, void* dst, int nlev, bool dense,
                                      cudaStream_t st) {
    StreamParams sp = stream_params(p, nlev);
    sp.in = src;
    sp.out = dst;
    sp.ld = p->pad_ld;
    sp.ld_out = dense ? p->nx : p->pad_ld;
    sp.dense_out = dense;
    sp.vec = 1;
    if (p->warp_nc && nlev == kWarpDepth && !dense) return launch_warp(p, sp, st);
    const StreamKernelRef r = pad_kernel(p, nlev);
    const int smem = stream_smem_bytes(p->R, nlev, (int)p->elem, true, false, p->threads);
    if (!((p->pad_set >> nlev) & 1)) {
        CK(cudaFuncSetAttribute(r.fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                stream_smem_bytes(p->R, nlev, (int)p->elem, true, false, kStreamMaxThreads)));
        p->pad_set |= 1u << nlev;
    }
    void* args[] = {&sp};
    CK(cudaLaunchKernel(r.fn, dim3((unsigned)(p->strips * p->tiles_y)), dim3((unsigned)p->threads), args,
                        (size_t)smem, st));
    return STENCIL_OK;
}

static stencil_status_t run_padded(stencil_plan* p, const void* in, void* out, const std::vector<int>& depths,
                                   cudaStream_t st) {
    const int64_t chunks = p->ny * (p->pad_ld / 4);
    const unsigned blocks = (unsigned)std::min<int64_t>(ceil_div(chunks, 256), 16LL * p->sms);
    if (p->elem == 4)
        pad_rows_kernel<uint32_t><<<blocks, 256, 0, st>>>(static_cast<const uint32_t*>(in),
                                                          static_cast<uint32_t*>(p->pad[0]), p->ny, p->nx, p->pad_ld);
    else
        pad_rows_kernel<uint16_t><<<blocks, 256, 0, st>>>(static_cast<const uint16_t*>(in),
                                                          static_cast<uint16_t*>(p->pad[0]), p->ny, p->nx, p->pad_ld);
    CK(cudaGetLastError());
    int cur = 0;
    for (size_t i = 0; i < depths.size(); ++i) {
        const bool last = i + 1 == depths.size();
        stencil_status_t s = launch_padded(p, p->pad[cur], last ? out : p->pad[cur ^ 1], depths[i], last, st);
        if (s != STENCIL_OK) return s;
        cur ^= 1;
    }
    return STENCIL_OK;
}

// Whether a run of these launches goes through the padded grids (a single
// launch would pay the copy for one pass: 9-point box BF16 4001 x 5003, 4 steps
// 64 us padded, 63 element-wise; 16 steps 150 against 223).
static bool use_padded(const stencil_plan* p, size_t launches) {
    return p->kernel == STENCIL_KERNEL_STREAM && p->pad[0] && launches >= 2;
}

// Depths of the launches for T steps: full blocks of k, then the remainder
// split greedily into instantiated depths.
static std::vector<int> launch_depths(const stencil_plan* p, int64_t T) {
    std::vector<int> d;
    if (p->kernel == STENCIL_KERNEL_RESIDENT) {  // the whole run in one launch (chunks of 2^30 steps)
        for (int64_t t = 0; t < T; t += (1 << 30)) d.push_back((int)std::min<int64_t>(T - t, 1 << 30));
        return d;
    }
    const int k = p->kernel != STENCIL_KERNEL_STREAM ? 1 : p->tiles_on ? p->tiles.k : p->k;
    for (int64_t t = 0; t < T / k; ++t) d.push_back(k);
    int rem = (int)(T % k);
    while (rem > 0) {
        const int step = p->kernel != STENCIL_KERNEL_STREAM ? 1
                         : p->tiles_on                      ? std::min(rem, p->tiles.k)
                                                            : stream_depth_at_most(p->R, p->star, rem);
        d.push_back(step);
        rem -= step;
    }
    return d;
}

// ---- all states of a run (the adjoint's segment recomputation) ------------------------
//
// outs[i] = u_{i+1} for i < n, from u_0 = in: launches of the all-states
// kernels (depths 8 / 4 / 2 / 1 as available), each reading the last state the
// previous launch wrote and storing every level.  FP32 plans whose rows are
// 16-byte aligned; anything else runs one single-step stencil_run per state.
// Each state is the same bits as stencil_run produces (same arithmetic per
// point, independent of the launch depths).

// One all-states launch of d steps: level l+1 to outs[l] (null: not stored, but the last must be).
static stencil_status_t launch_states(stencil_plan_t* p, const void* src, float* const* outs, int d, cudaStream_t st) {
    if (d == kWarpDepth && p->R == 1 && p->star) {
        // one-warp tiles for the 5-point star where they have enough rows (4096^2: 123 us
        // per launch, 153 CTA-wide).  Not the 9-point box, whose levels' stores spill
        // there: gradients of 18 steps with 8 states a segment, one-warp | CTA-wide, us:
        // 4096^2 1188 | 1141, 7567 x 3036 1722 | 1614, 8192^2 4267 | 4178.
        const WarpTiles t = warp_tiles(p, 4);
        if (t.by >= kWarpMinRows) {
            StreamParams sp = stream_params(p, d);
            sp.in = src;
            sp.out = outs[d - 1];
            sp.H = kWarpDepth;
            sp.bx = t.bx;
            sp.by = t.by;
            sp.strips = t.strips;
            sp.vec = 1;
            for (int l = 0; l < d - 1; ++l) sp.lvl_out[l] = outs[l];
            void* args[] = {&sp};
            CK(cudaLaunchKernel(get_warp_states_kernel(), dim3((unsigned)(t.strips * t.tiles)), dim3(32), args, 0,
                                st));
            return STENCIL_OK;
        }
    }
    const int threads = 128;
    const StreamKernelRef r = get_stream_states_kernel(p->R, p->star, d);
    if (!r.fn) return fail(STENCIL_ERR_UNSUPPORTED, "no all-states kernel");
    const int H = (p->R * d + 3) / 4 * 4;
    const int64_t strips = ceil_div(p->nx, 4 * threads - 2 * H);
    const int bx = (int)(ceil_div(ceil_div(p->nx, strips), 4) * 4);
    const int nt = (int)(ceil_div(ceil_div(bx + 2 * H, 4), 32) * 32);
    const int smem = stream_smem_bytes(p->R, d, 4, true, false, nt);
    const unsigned bit = 1u << d;
    static std::mutex mu;
    {
        std::lock_guard<std::mutex> g(mu);
        static unsigned set_bits[3][2] = {};
        if (!(set_bits[p->R - 1][p->star] & bit)) {
            CK(cudaFuncSetAttribute(r.fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    stream_smem_bytes(p->R, d, 4, true, false, kStreamMaxThreads)));
            set_bits[p->R - 1][p->star] |= bit;
        }
    }
    int per_sm = 0;
    CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, r.fn, nt, smem));
    if (per_sm < 1) return fail(STENCIL_ERR_UNSUPPORTED, "all-states kernel does not fit on an SM");
    const int64_t want = std::max<int64_t>(1, (int64_t)per_sm * p->sms / strips);
    const int64_t by_min = std::max<int64_t>(8, 4LL * p->R * d);
    int64_t tiles_y = std::max<int64_t>(1, std::min<int64_t>(want, ceil_div(p->ny, by_min)));
    const int by = (int)ceil_div(p->ny, tiles_y);
    tiles_y = ceil_div(p->ny, by);
    StreamParams sp = stream_params(p, d);
    sp.in = src;
    sp.out = outs[d - 1];
    sp.H = H;
    sp.bx = bx;
    sp.by = by;
    sp.strips = (int)strips;
    sp.vec = 1;
    for (int l = 0; l < d - 1; ++l) sp.lvl_out[l] = outs[l];
    void* args[] = {&sp};
    CK(cudaLaunchKernel(r.fn, dim3((unsigned)(strips * tiles_y)), dim3((unsigned)nt), args, (size_t)smem, st));
    return STENCIL_OK;
}

namespace gbst {
// The entry points that return sums over the grid in FP64 (weight gradients,
// residuals) resolve the last bits of the states.  Register tiles give the bits of
// the kernel they stand in for (cluster-resident: GridConfig::plain; else
// streaming), except where the streaming kernel's depend on how steps are grouped:
// periodic widths that are not a multiple of 4.  For one such call, on = true puts
// such a plan back on the streaming kernel (true: it did, and on = false undoes it).
bool plan_keep_sums(stencil_plan_t* p, bool on) {
    if (!on) {
        p->kernel = p->kept_kernel;
        p->grid_on = p->kept_grid;
        p->tiles_on = p->kept_tiles;
        return false;
    }
    if (!(p->grid_on || p->tiles_on) || p->opt.autotune || (p->grid_on && p->grid.plain)) return false;
    if (!(p->boundary == STENCIL_BOUNDARY_PERIODIC && p->nx % 4 != 0)) return false;
    p->kept_kernel = p->kernel;
    p->kept_grid = p->grid_on;
    p->kept_tiles = p->tiles_on;
    p->kernel = STENCIL_KERNEL_STREAM;
    p->grid_on = p->tiles_on = 0;
    return true;
}

// stencil_run_launches(p, T) in the form that plan_keep_sums gives the plan for such a call.
int64_t plan_sum_launches(const stencil_plan_t* p, int64_t T) {
    stencil_plan q = *p;  // (the caller's plan stays as it is: another thread may be running it)
    plan_keep_sums(&q, true);
    return stencil_run_launches(&q, T);
}

// Chip-resident plans: every state in one launch (13-point star 1000 x 1022: a
// single-step launch per state took 13 us each).  Not for periodic ragged widths,
// whose bits depend on how the steps are grouped, and in the streaming kernel's
// summation order only (any_order: any will do).
bool plan_states_one_launch(const stencil_plan_t* p, bool any_order) {
    return p->kernel == STENCIL_KERNEL_RESIDENT && p->grid_on && (any_order || !p->grid.plain) &&
           p->dtype == STENCIL_F32 && !(p->boundary == STENCIL_BOUNDARY_PERIODIC && p->nx % 4 != 0);
}

// Most states of one all-states launch.  The 5-point star's CTA-wide kernel stores eight
// levels at a higher cost than twice four (gradients of 33 steps, 8 | 4 levels, us: 1032 x
// 2712 725 | 628, 2048^2 799 | 674, 1500 x 4000 1008 | 883), its one-warp tiles do not.
int plan_states_depth(const stencil_plan_t* p) {
    if (p->R == 1) return p->star && warp_tiles(p, 4).by < kWarpMinRows ? 4 : 8;
    return p->R == 3 && !p->star ? 2 : 4;
}

stencil_status_t plan_run_states(stencil_plan_t* p, const void* in, float* const* outs, int64_t n, bool any_order,
                                 cudaStream_t st) {
    bool fused = p->dtype == STENCIL_F32 && p->nx % 4 == 0 && (uintptr_t)in % 16 == 0;
    for (int64_t i = 0; i < n && fused; ++i) fused = (uintptr_t)outs[i] % 16 == 0;
    // (one state alone: 945 x 1700 8 us streaming, 12 as tiles)
    bool strided = plan_states_one_launch(p, any_order) && n >= (fused ? 2 : 1) && n < (1 << 30);
    const int64_t stride = n > 1 ? outs[1] - outs[0] : 0;
    for (int64_t i = 1; i < n && strided; ++i) strided = outs[i] - outs[i - 1] == stride;
    if (strided) {
        const int vec = p->nx % 4 == 0 && stride % 4 == 0 && (uintptr_t)in % 16 == 0 && (uintptr_t)outs[0] % 16 == 0;
        const cudaError_t e =
            launch_grid(p->grid, p->R, p->star, p->dtype, p->boundary == STENCIL_BOUNDARY_PERIODIC, in, outs[n - 1],
                        (int)p->ny, (int)p->nx, vec, (int)n, p->grid.k, p->grid_mem, p->status,
                        (long long)(p->opt.timeout_ms > 0 ? p->opt.timeout_ms : 2000) * 1000000LL,
                        p->opt.debug_withhold, p->w, st, outs[0], stride);
        if (e == cudaSuccess) return STENCIL_OK;
        if (e != cudaErrorCooperativeLaunchTooLarge) CK(e);
        cudaGetLastError();  // (fewer SMs than the device reports: the paths below)
    }
    if (!fused) {
        const void* src = in;
        for (int64_t i = 0; i < n; ++i) {
            stencil_status_t s = stencil_run(p, src, outs[i], 1, st);
            if (s != STENCIL_OK) return s;
            src = outs[i];
        }
        return STENCIL_OK;
    }
    const void* src = in;
    for (int64_t i = 0; i < n;) {
        int d = plan_states_depth(p);
        for (; d > 1; d /= 2)
            if (d <= n - i && get_stream_states_kernel(p->R, p->star, d).fn) break;
        stencil_status_t s = launch_states(p, src, outs + i, d, st);
        if (s != STENCIL_OK) return s;
        src = outs[i + d - 1];
        i += d;
    }
    return STENCIL_OK;
}

// u_{m-1} and u_m (m >= 2, FP32), the last launch storing both, in two of the
// grids g1, g2 and g0 (*prev, *next).  `in` may be g0, and is then overwritten
// when launches come before that last one.  STENCIL_ERR_UNSUPPORTED, with nothing
// enqueued, where the plan has no kernel that stores two steps.
stencil_status_t plan_run_last_two(stencil_plan_t* p, const void* in, void* g1, void* g2, void* g0, int64_t m,
                                   cudaStream_t st, const void** prev, const void** next) {
    if (p->dtype != STENCIL_F32 || m < 2 || (p->opt.autotune && !p->tuned)) return STENCIL_ERR_UNSUPPORTED;
    if (p->kernel == STENCIL_KERNEL_RESIDENT && p->grid_on && !p->grid.plain && m < (1 << 30) &&
        !(p->boundary == STENCIL_BOUNDARY_PERIODIC && p->nx % 4 != 0)) {
        const int vec = p->nx % 4 == 0 && (uintptr_t)in % 16 == 0 && (uintptr_t)g1 % 16 == 0 && (uintptr_t)g2 % 16 == 0;
        const cudaError_t e = launch_grid(p->grid, p->R, p->star, p->dtype, p->boundary == STENCIL_BOUNDARY_PERIODIC, in,
                                          g2, (int)p->ny, (int)p->nx, vec, (int)m, p->grid.k, p->grid_mem, p->status,
                                          (long long)(p->opt.timeout_ms > 0 ? p->opt.timeout_ms : 2000) * 1000000LL,
                                          p->opt.debug_withhold, p->w, st, static_cast<float*>(g1), 0, (int)m - 1);
        p->last_stream = st;
        *prev = g1;
        *next = g2;
        if (e == cudaSuccess) return STENCIL_OK;
        if (e != cudaErrorCooperativeLaunchTooLarge) CK(e);
        cudaGetLastError();
        return STENCIL_ERR_UNSUPPORTED;
    }
    if (p->kernel != STENCIL_KERNEL_STREAM || p->nx % 4 != 0 || ((uintptr_t)in | (uintptr_t)g1 | (uintptr_t)g2 | (uintptr_t)g0) % 16 != 0)
        return STENCIL_ERR_UNSUPPORTED;
    // the depth of the last launch that leaves the fewest launches before it
    int best = 0;
    size_t fewest = 0;
    for (int d = 2; d <= 8; d *= 2) {  // (of equals the shallowest: it stores its levels at less cost)
        if (d > m || !get_stream_states_kernel(p->R, p->star, d).fn) continue;
        const size_t before = launch_depths(p, m - d).size();
        if (!best || before < fewest) {
            best = d;
            fewest = before;
        }
    }
    // (m = 8 j + 1 and the like: as many launches with the step apart, which stores one grid less)
    if (!best || launch_depths(p, m - 1).size() <= fewest) return STENCIL_ERR_UNSUPPORTED;
    void *a = g1, *b = g2;
    if (m > best) {
        stencil_status_t s = stencil_run(p, in, g2, m - best, st);
        if (s != STENCIL_OK) return s;
        in = g2;
        b = g0;
    }
    p->last_stream = st;
    float* outs[8] = {};
    outs[best - 2] = static_cast<float*>(a);
    outs[best - 1] = static_cast<float*>(b);
    *prev = a;
    *next = b;
    return launch_states(p, in, outs, best, st);
}
}  // namespace gbst

// ---- autotuning ---------------------------------------------------------------------
//
// With opt.autotune, the first stencil_run times every instantiated depth k
// with CTAs of 64, 128 and 256 threads (the depth and CTA size the caller
// fixed, if any, stay fixed) and keeps the fastest per step.  Each candidate
// runs one launch from `in` into the plan's workspace, so neither `in` nor
// `out` is touched.  Results are cached per (shape, radius, footprint, dtype,
// boundary, device) for the life of the process.

typedef std::tuple<int64_t, int64_t, int, int, int, int, int> TuneKey;
static std::map<TuneKey, std::pair<int, int>> g_tune_cache;
static std::mutex g_tune_mu;

static stencil_status_t time_launch(stencil_plan* p, const void* in, int reps, cudaStream_t st,
                                    float* ms) {
    cudaEvent_t e0, e1;
    CK(cudaEventCreate(&e0));
    CK(cudaEventCreate(&e1));
    auto once = [&] {
        return p->pad[0] ? launch_padded(p, p->pad[0], p->pad[1], p->k, false, st)
                         : launch_once(p, in, p->ws, p->tiles_on ? p->tiles.k : p->k, st);
    };
    stencil_status_t s = once();  // warm-up
    if (s == STENCIL_OK) {
        cudaEventRecord(e0, st);
        for (int i = 0; i < reps && s == STENCIL_OK; ++i) s = once();
        cudaEventRecord(e1, st);
    }
    cudaError_t e = cudaEventSynchronize(e1);
    if (s == STENCIL_OK && e == cudaSuccess) e = cudaEventElapsedTime(ms, e0, e1);
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (s != STENCIL_OK) return s;
    if (e != cudaSuccess) return fail(STENCIL_ERR_CUDA, std::string("autotune timing: ") + cudaGetErrorString(e));
    return STENCIL_OK;
}

// Tensor-core plans: time the warp-MMA engine and every usable tcgen05 MMA
// width (one step per launch, `in` into the workspace) and keep the fastest.
// A plan created with kernel = TC_UMMA, or with mma_n set, keeps that choice.
typedef std::tuple<int64_t, int64_t, int, int, int> TcTuneKey;
static std::map<TcTuneKey, int> g_tc_tune_cache;  // MMA width (0: warp MMAs), + kTunePhase for the phase kernel
static const int kTunePhase = 1024;

static stencil_status_t autotune_tc(stencil_plan* p, const void* in, cudaStream_t st) {
    if (!p->umma_ok || p->opt.kernel == STENCIL_KERNEL_TC_UMMA || p->opt.mma_n > 0) return STENCIL_OK;
    const TcTuneKey key(p->ny, p->nx, p->dtype, p->compute, p->device);
    int best_n = -1;
    {
        std::lock_guard<std::mutex> g(g_tune_mu);
        auto it = g_tc_tune_cache.find(key);
        if (it != g_tc_tune_cache.end()) best_n = it->second;
    }
    if (best_n < 0) {
        const int reps = (int)std::max(2.0, std::min(32.0, 4e9 / ((double)p->ny * (double)p->nx)));
        float best = 1e30f;
        for (int c = 0; c <= 6; ++c) {
            const int nt = c == 6 ? kUmmaDefaultN[p->compute == STENCIL_COMPUTE_TC_TF32] : c ? kUmmaWidths[c - 1] : 0;
            if (nt && !((p->umma_ok >> (nt / 16)) & 1)) continue;
            if (c == 6 && !p->phase_ok) continue;
            p->umma_n = nt;
            p->phase = c == 6;
            cudaEvent_t e0, e1;
            CK(cudaEventCreate(&e0));
            CK(cudaEventCreate(&e1));
            stencil_status_t s = launch_once(p, in, p->ws, 1, st, 0, 1);  // warm-up
            if (s == STENCIL_OK) {
                cudaEventRecord(e0, st);
                for (int i = 0; i < reps && s == STENCIL_OK; ++i) s = launch_once(p, in, p->ws, 1, st, 0, 1);
                cudaEventRecord(e1, st);
            }
            cudaError_t e = cudaEventSynchronize(e1);
            float ms = 0.f;
            if (s == STENCIL_OK && e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
            cudaEventDestroy(e0);
            cudaEventDestroy(e1);
            if (s != STENCIL_OK) return s;
            if (e != cudaSuccess) return fail(STENCIL_ERR_CUDA, std::string("autotune timing: ") + cudaGetErrorString(e));
            if (ms < best) {
                best = ms;
                best_n = nt + (c == 6 ? kTunePhase : 0);
            }
        }
        std::lock_guard<std::mutex> g(g_tune_mu);
        g_tc_tune_cache[key] = best_n;
    }
    p->phase = best_n >= kTunePhase;
    best_n %= kTunePhase;
    p->umma_n = best_n;
    p->kernel = best_n ? STENCIL_KERNEL_TC_UMMA : STENCIL_KERNEL_TC;
    return STENCIL_OK;
}

static stencil_status_t autotune(stencil_plan* p, const void* in, cudaStream_t st) {
    const TuneKey key(p->ny, p->nx, p->R + 32 * p->tiles_ok, p->star, p->dtype, p->boundary, p->device);
    {
        std::lock_guard<std::mutex> g(g_tune_mu);
        auto it = g_tune_cache.find(key);
        if (it != g_tune_cache.end()) {
            p->tma = (it->second.second >> 16) & 1;
            stencil_status_t s = configure_stream(p, it->second.first, it->second.second & 0xffff, p->opt.tile_rows);
            if (s == STENCIL_OK) p->tiles_on = it->second.second >> 17;
            return s;
        }
    }
    const int ths[3] = {64, 128, 256};
    float best = 1e30f, def_time = -1.f;
    int bk = p->k, bt = p->threads, btma = p->tma;
    const int k0 = p->k, t0 = p->opt.threads > 0 ? p->opt.threads : default_threads(p->R, p->star), tma0 = p->tma;
    const double points = (double)p->ny * (double)p->nx;
    // Row loads: both the cp.async ring and the TMA-fed ring where the plan
    // allows either (load = AUTO), else the one it fixed.
    const int tma_lo = p->opt.load == STENCIL_LOAD_TMA ? 1 : 0;
    const int tma_hi = (p->opt.load != STENCIL_LOAD_CP_ASYNC && tma_eligible(p)) ? 1 : 0;
    for (int tma = tma_lo; tma <= tma_hi; ++tma) {
        p->tma = tma;
        for (int i = 0; i < 8 && kStreamDepths[p->R - 1][p->star][i]; ++i) {
            const int k = kStreamDepths[p->R - 1][p->star][i];
            if (p->opt.tb_depth > 0 && k != p->opt.tb_depth) continue;
            for (int th : ths) {
                if (p->opt.threads > 0 && th != p->opt.threads) continue;
                if (configure_stream(p, k, th, p->opt.tile_rows) != STENCIL_OK) continue;
                // About 2e9 point-steps of work per candidate, at least one launch.
                const int reps = (int)std::max(1.0, std::min(64.0, 2e9 / (points * k)));
                float ms = 0.f;
                stencil_status_t s = time_launch(p, in, reps, st, &ms);
                if (s != STENCIL_OK) return s;
                const float per_step = ms / (float)(reps * k);
                if (k == k0 && th == t0 && tma == tma0) def_time = per_step;
                if (per_step < best) {
                    best = per_step;
                    bk = k;
                    bt = th;
                    btma = tma;
                }
            }
        }
    }
    // Keep the default configuration unless a candidate beats it by more than
    // 2 %: closer timings are within run-to-run noise, and a stable choice
    // keeps launch counts and profiles reproducible.
    if (def_time > 0.f && def_time <= 1.02f * best) {
        bk = k0;
        bt = t0;
        btma = tma0;
    }
    p->tma = btma;
    stencil_status_t s = configure_stream(p, bk, bt, p->opt.tile_rows);
    if (s != STENCIL_OK) return s;
    if (p->tiles_ok) {
        // the register tiles are this plan's default: they stay unless the best above is clearly faster
        const int tk = p->tiles.k, reps = (int)std::max(1.0, std::min(64.0, 2e9 / (points * tk)));
        float ms = 0.f;
        p->tiles_on = 1;
        s = time_launch(p, in, reps, st, &ms);
        if (s != STENCIL_OK) return s;
        p->tiles_on = ms / (float)(reps * tk) <= 1.02f * best;
    }
    std::lock_guard<std::mutex> g(g_tune_mu);
    g_tune_cache[key] = std::make_pair(bk, bt | (btma << 16) | (p->tiles_on << 17));
    return STENCIL_OK;
}

// Small grids (plans that chose a resident kernel): time the chip-resident
// kernel, the cluster-resident one at every usable cluster size (runs of 64
// steps from `in` into the workspace) and the autotuned streaming kernel, per step, and keep the faster.  The
// decision is cached like the streaming kernel's.
static std::map<TuneKey, int> g_res_tune_cache;  // 16 * kb + log2(C) + 1, kTuneGrid, or 0 for the streaming kernel
static const int kTuneGrid = 1 << 20;

static stencil_status_t autotune_resident(stencil_plan* p, const void* in, cudaStream_t st) {
    // (plans that asked for the cluster-resident kernel have no chip-resident candidate)
    auto tune_key = [&] {
        return TuneKey(p->ny, p->nx, p->R + 16 * p->grid_ok, p->star, p->dtype, p->boundary, p->device);
    };
    int decision = -1;
    {
        std::lock_guard<std::mutex> g(g_tune_mu);
        auto it = g_res_tune_cache.find(tune_key());
        if (it != g_res_tune_cache.end()) decision = it->second;
    }
    if (decision < 0) {
        constexpr int S = 64;
        const int reps = (int)std::max(2.0, std::min(16.0, 1e8 / ((double)p->ny * (double)p->nx * S)));
        float best = 1e30f;
        decision = 0;
        // S steps from `in` into the workspace with the resident kernel in use.
        auto try_resident = [&](int code) -> stencil_status_t {
            cudaEvent_t e0, e1;
            CK(cudaEventCreate(&e0));
            CK(cudaEventCreate(&e1));
            stencil_status_t s = launch_once(p, in, p->ws, S, st);  // warm-up
            if (s == STENCIL_OK) {
                cudaEventRecord(e0, st);
                for (int i = 0; i < reps && s == STENCIL_OK; ++i) s = launch_once(p, in, p->ws, S, st);
                cudaEventRecord(e1, st);
            }
            cudaError_t e = cudaEventSynchronize(e1);
            float ms = 0.f;
            if (s == STENCIL_OK && e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
            cudaEventDestroy(e0);
            cudaEventDestroy(e1);
            if (s != STENCIL_OK) return s;
            if (e != cudaSuccess) return fail(STENCIL_ERR_CUDA, std::string("autotune timing: ") + cudaGetErrorString(e));
            const float per_step = ms / (float)(reps * S);
            if (per_step < best) {
                best = per_step;
                decision = code;
            }
            return STENCIL_OK;
        };
        if (p->grid_ok) {
            use_grid(p);
            stencil_status_t s = try_resident(kTuneGrid);
            // (a partition too small for the tiles, which launch_once then rules out: the others are left)
            if (s != STENCIL_OK && !(s == STENCIL_ERR_UNSUPPORTED && !p->grid_ok)) return s;
        }
        for (int lg = 0; (1 << lg) <= resident_max_cluster(); ++lg) {
            if (!((p->res_ok >> lg) & 1)) continue;
            for (int kb = 1; kb <= 8; kb *= 2) {
                int rp = 0;
                const int periodic = p->boundary == STENCIL_BOUNDARY_PERIODIC;
                if (resident_config((int)p->ny, (int)p->nx, p->R, periodic, 1 << lg, kb, p->res_max_smem, &rp) < 0)
                    continue;
                stencil_status_t s = use_resident(p, 1 << lg, kb);
                if (s != STENCIL_OK) return s;
                s = try_resident(16 * kb + lg + 1);
                if (s != STENCIL_OK) return s;
            }
        }
        stencil_status_t s = autotune(p, in, st);  // configures the best streaming kernel
        if (s != STENCIL_OK) return s;
        const int sreps = (int)std::max(2.0, std::min(64.0, 1e8 / ((double)p->ny * (double)p->nx * p->k)));
        float ms = 0.f;
        s = time_launch(p, in, sreps, st, &ms);
        if (s != STENCIL_OK) return s;
        if (ms / (float)(sreps * p->k) < best) decision = 0;
        std::lock_guard<std::mutex> g(g_tune_mu);
        g_res_tune_cache[tune_key()] = decision;  // (for the candidates that there were)
    }
    if (decision == kTuneGrid) {
        if (p->grid.plain) {  // (for cluster_run: the default configuration, not the last one timed)
            const int C = resident_candidates(p);
            if (C > 0) {
                stencil_status_t s = use_resident(p, C);
                if (s != STENCIL_OK) return s;
            }
        }
        use_grid(p);
        return STENCIL_OK;
    }
    if (decision > 0) return use_resident(p, 1 << ((decision & 15) - 1), decision >> 4);
    return autotune(p, in, st);
}

// Clear device memory before returning, without touching the caller's streams:
// a first run on any stream must see it cleared.
// (One stream per device, kept for the life of the process: creating one per
// plan cost more than the rest of the call.)
static cudaError_t zero_now(int device, void* ptr, size_t bytes) {
    static std::mutex mu;
    static std::map<int, cudaStream_t> streams;
    std::lock_guard<std::mutex> g(mu);
    cudaStream_t& st = streams[device];
    cudaError_t e = cudaSuccess;
    if (!st) e = cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaMemsetAsync(ptr, 0, bytes, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    return e;
}

namespace gbst {
cudaError_t plan_zero_now(const stencil_plan_t* p, void* ptr, size_t bytes) { return zero_now(p->device, ptr, bytes); }
}  // namespace gbst

extern "C" {

const char* stencil_status_string(stencil_status_t s) {
    switch (s) {
        case STENCIL_OK: return "STENCIL_OK";
        case STENCIL_ERR_INVALID_ARG: return "STENCIL_ERR_INVALID_ARG";
        case STENCIL_ERR_UNSUPPORTED: return "STENCIL_ERR_UNSUPPORTED";
        case STENCIL_ERR_CUDA: return "STENCIL_ERR_CUDA";
        case STENCIL_ERR_OOM: return "STENCIL_ERR_OOM";
        case STENCIL_ERR_TIMEOUT: return "STENCIL_ERR_TIMEOUT";
        case STENCIL_ERR_DEVICE_CHECK: return "STENCIL_ERR_DEVICE_CHECK";
        default: return "STENCIL_ERR_UNKNOWN";
    }
}

const char* stencil_last_error(void) { return g_last_error.c_str(); }

int stencil_version(void) { return 100; }

stencil_status_t stencil_plan_create(stencil_plan_t** out, int64_t ny, int64_t nx, int radius,
                                     const float* weights, int dtype, int boundary,
                                     const stencil_options_t* opt) {
    if (!out) return fail(STENCIL_ERR_INVALID_ARG, "plan pointer is NULL");
    *out = nullptr;
    if (ny < 1 || nx < 1) return fail(STENCIL_ERR_INVALID_ARG, "ny and nx must be >= 1");
    if (radius < 1) return fail(STENCIL_ERR_INVALID_ARG, "radius must be >= 1");
    if (radius > kMaxRadius) return fail(STENCIL_ERR_UNSUPPORTED, "radius > 3 is not supported");
    if (ny > (1LL << 30) || nx > (1LL << 30))
        return fail(STENCIL_ERR_UNSUPPORTED, "ny and nx must be <= 2^30");
    if (!weights) return fail(STENCIL_ERR_INVALID_ARG, "weights pointer is NULL");
    if (dtype < STENCIL_F32 || dtype > STENCIL_F16) return fail(STENCIL_ERR_INVALID_ARG, "bad dtype");
    if (boundary != STENCIL_BOUNDARY_ZERO && boundary != STENCIL_BOUNDARY_PERIODIC)
        return fail(STENCIL_ERR_INVALID_ARG, "bad boundary");
    stencil_options_t o{};
    if (opt) o = *opt;
    if (o.compute < 0 || o.compute > STENCIL_COMPUTE_LOWRANK || o.kernel < 0 ||
        o.kernel > STENCIL_KERNEL_RESIDENT || o.tb_depth < 0 || o.threads < 0 || o.tile_rows < 0 ||
        o.mma_n < 0 || o.timeout_ms < 0 || o.debug_withhold < 0 || o.debug_withhold > 1 ||
        o.load < STENCIL_LOAD_AUTO || o.load > STENCIL_LOAD_TMA || o.rank < 0 || o.rank > 2 * radius + 1)
        return fail(STENCIL_ERR_INVALID_ARG, "bad option value");

    stencil_plan* p = new (std::nothrow) stencil_plan();
    if (!p) return fail(STENCIL_ERR_OOM, "host allocation failed");
    p->ny = ny;
    p->nx = nx;
    p->R = radius;
    p->dtype = dtype;
    p->boundary = boundary;
    p->compute = (o.compute == STENCIL_COMPUTE_TC_TF32 || o.compute == STENCIL_COMPUTE_TC_BF16 ||
                  o.compute == STENCIL_COMPUTE_TC_3XTF32 || o.compute == STENCIL_COMPUTE_LOWRANK)
                     ? o.compute : STENCIL_COMPUTE_FP32;
    p->opt = o;
    p->elem = elem_size(dtype);
    const int D = 2 * radius + 1;
    int star = 1;
    for (int a = 0; a < D; ++a)
        for (int b = 0; b < D; ++b) {
            const float v = weights[a * D + b];
            if (!std::isfinite(v)) {
                delete p;
                return fail(STENCIL_ERR_INVALID_ARG, "weights must be finite");
            }
            p->w.w[a * D + b] = v;
            if (a != radius && b != radius && v != 0.f) star = 0;
        }
    p->star = star;

    auto bail = [&](stencil_status_t st) {
        stencil_plan_destroy(p);
        return st;
    };
    cudaError_t e = cudaGetDevice(&p->device);
    if (e != cudaSuccess) {
        delete p;
        return fail(STENCIL_ERR_CUDA, std::string("cudaGetDevice: ") + cudaGetErrorString(e));
    }
    e = cudaDeviceGetAttribute(&p->sms, cudaDevAttrMultiProcessorCount, p->device);
    if (e != cudaSuccess) {
        delete p;
        return fail(STENCIL_ERR_CUDA, std::string("cudaDeviceGetAttribute: ") + cudaGetErrorString(e));
    }

    // Small grids the chip-resident kernel does not take: the cluster-resident
    // kernel, unless the caller asked for the streaming kernel or set one of its
    // options.  With kernel = RESIDENT, tb_depth is its number of steps per halo exchange.
    auto cluster_choice = [&](stencil_status_t st) -> stencil_status_t {
        const bool stream_opts = o.tb_depth > 0 || o.threads > 0 || o.tile_rows > 0;
        if (st == STENCIL_OK && (o.kernel == STENCIL_KERNEL_RESIDENT ||
                                 (o.kernel == STENCIL_KERNEL_AUTO && !stream_opts))) {
            const int kb = (o.kernel == STENCIL_KERNEL_RESIDENT && o.tb_depth > 0) ? o.tb_depth : 1;
            const int C = resident_candidates(p, kb);
            if (C > 0)
                st = use_resident(p, C, kb);
            else if (o.kernel == STENCIL_KERNEL_RESIDENT)
                st = fail(STENCIL_ERR_UNSUPPORTED, "grid too large for the cluster-resident kernel at this depth");
        }
        return st;
    };
    stencil_status_t st;
    const bool tc_kernel = o.kernel == STENCIL_KERNEL_TC || o.kernel == STENCIL_KERNEL_TC_WARP ||
                           o.kernel == STENCIL_KERNEL_TC_UMMA;
    if (p->compute == STENCIL_COMPUTE_LOWRANK) {
        st = configure_lowrank(p);
    } else if (p->compute != STENCIL_COMPUTE_FP32 || tc_kernel) {
        if (p->compute == STENCIL_COMPUTE_FP32) p->compute = STENCIL_COMPUTE_TC_TF32;
        st = configure_tc(p);
    } else if (o.kernel == STENCIL_KERNEL_NAIVE) {
        st = configure_naive(p);
    } else {
        const int k = o.tb_depth > 0 ? o.tb_depth : default_depth(radius, star);
        const int threads = o.threads > 0 ? o.threads : default_threads(radius, star);
        if (o.load == STENCIL_LOAD_TMA && !tma_eligible(p))
            return bail(fail(STENCIL_ERR_UNSUPPORTED,
                             "TMA-fed rows need FP32 storage, the zero rule and nx a multiple of 4"));
        const int k0 = std::min(k, stream_kmax(radius, star));
        p->tma = o.load == STENCIL_LOAD_TMA || (o.load == STENCIL_LOAD_AUTO && tma_eligible(p) && kDefaultTma);
        st = configure_stream(p, k0, threads, o.tile_rows);
        const bool stream_opts = o.tb_depth > 0 || o.threads > 0 || o.tile_rows > 0;
        const bool may_grid = o.kernel == STENCIL_KERNEL_AUTO && !stream_opts && o.load == STENCIL_LOAD_AUTO;
        if (st == STENCIL_OK && may_grid && grid_candidate(p)) use_grid(p);
        if (st == STENCIL_OK && p->grid_on && o.autotune) resident_candidates(p);  // to be timed as well
        if (!p->grid_on) st = cluster_choice(st);
        if (st == STENCIL_OK && may_grid && p->kernel == STENCIL_KERNEL_STREAM) choose_tiles(p);
    }
    if (st != STENCIL_OK) return bail(st);

    // The ping-pong workspace, what the plan's kernel needs besides, and the status word: one
    // allocation (each costs ~30 us, and ~27 to free) unless the word would need a 2 MiB page
    // of its own there (8192^2: 187 us to create the plan, 155 with the word apart).
    const size_t bytes = (size_t)ny * (size_t)nx * p->elem;
    auto allocate = [&](size_t size) {
        const size_t page = 2 << 20, off = (size + 255) / 256 * 256;
        const bool fits = (off + sizeof(unsigned) + page - 1) / page == (size + page - 1) / page;
        if (cudaMalloc(&p->ws, fits ? off + sizeof(unsigned) : size) != cudaSuccess) {
            cudaGetLastError();
            p->ws = nullptr;
            return false;
        }
        if (fits) {
            p->status = reinterpret_cast<unsigned*>(static_cast<char*>(p->ws) + off);
        } else if (cudaMalloc(&p->status_mem, sizeof(unsigned)) == cudaSuccess) {
            p->status = static_cast<unsigned*>(p->status_mem);
        } else {
            cudaGetLastError();
            p->status_mem = nullptr;
            cudaFree(p->ws);
            p->ws = nullptr;
            return false;
        }
        return true;
    };
    if (p->grid_ok) {  // the chip-resident kernel's scratch
        const size_t off = (bytes + 255) / 256 * 256;
        const size_t scratch = grid_scratch_bytes((int)ny, (int)nx);
        if (allocate(off + scratch)) {
            p->grid_mem = static_cast<char*>(p->ws) + off;
            const char* end = p->status_mem ? static_cast<char*>(p->grid_mem) + scratch
                                            : reinterpret_cast<char*>(p->status + 1);
            e = zero_now(p->device, p->grid_mem, (size_t)(end - static_cast<char*>(p->grid_mem)));
            if (e != cudaSuccess) {
                bail(STENCIL_ERR_CUDA);
                return fail(STENCIL_ERR_CUDA, std::string("clearing the exchange grids: ") + cudaGetErrorString(e));
            }
        } else {  // no room for the exchange grids: the kernels that need none
            p->grid_ok = 0;
            if (p->grid_on) {
                p->grid_on = 0;
                p->kernel = STENCIL_KERNEL_STREAM;
                st = cluster_choice(STENCIL_OK);
                if (st != STENCIL_OK) return bail(st);
            }
        }
    }
    // Ragged widths under the zero rule: two grids of padded rows, the first of
    // which doubles as the workspace.
    if (!p->ws && p->kernel == STENCIL_KERNEL_STREAM && !p->tiles_on && pad_eligible(p)) {
        const int64_t ld = ceil_div(nx, kPadElems) * kPadElems;
        const size_t grid = ((size_t)ny * (size_t)ld * p->elem + 255) / 256 * 256;
        if (allocate(2 * grid)) {  // (no room: element-wise loads and stores on the dense grids)
            p->pad_ld = ld;
            p->pad[0] = p->ws;
            p->pad[1] = static_cast<char*>(p->ws) + grid;
        }
    }
    if (!p->ws && !allocate(bytes)) {
        bail(STENCIL_ERR_OOM);
        return fail(STENCIL_ERR_OOM, "cudaMalloc of the workspace failed");
    }
    if ((!p->grid_mem || p->status_mem) && (e = cudaMemset(p->status, 0, sizeof(unsigned))) != cudaSuccess) {
        cudaGetLastError();
        bail(STENCIL_ERR_CUDA);
        return fail(STENCIL_ERR_CUDA, std::string("clearing the status word: ") + cudaGetErrorString(e));
    }
    *out = p;
    return STENCIL_OK;
}

void stencil_plan_destroy(stencil_plan_t* p) {
    if (!p) return;
    for (int i = 0; i < 4; ++i)
        if (p->aux[i] && p->aux_free[i]) p->aux_free[i](p->aux[i]);
    if (p->ws) cudaFree(p->ws);
    if (p->status_mem) cudaFree(p->status_mem);
    if (p->host_in) cudaFree(p->host_in);
    if (p->host_out) cudaFree(p->host_out);
    delete p;
}

stencil_status_t stencil_plan_set_weights(stencil_plan_t* p, const float* weights) {
    if (!p || !weights) return fail(STENCIL_ERR_INVALID_ARG, "NULL argument");
    const int R = p->R, D = 2 * R + 1;
    int star = 1;
    for (int a = 0; a < D; ++a)
        for (int b = 0; b < D; ++b) {
            const float v = weights[a * D + b];
            if (!std::isfinite(v)) return fail(STENCIL_ERR_INVALID_ARG, "weights must be finite");
            if (a != R && b != R && v != 0.f) star = 0;
        }
    const bool footprint_bound = p->kernel == STENCIL_KERNEL_STREAM || p->kernel == STENCIL_KERNEL_RESIDENT;
    if (footprint_bound && star != p->star)
        return fail(STENCIL_ERR_UNSUPPORTED,
                    "the new weights change the footprint (star / box) the plan's kernel was chosen for");
    if (p->kernel == STENCIL_KERNEL_LOWRANK) {
        float col[7][7], row[7][7];
        int rho = lowrank_factor(weights, R, p->opt.rank, col, row, nullptr);
        if (rho < 1) rho = 1;
        const void* fn = get_lowrank_kernel(R, rho);
        if (!fn) return fail(STENCIL_ERR_UNSUPPORTED, "no low-rank kernel for this rank");
        p->lr_rank = rho;
        p->lr_fn = fn;
        std::memcpy(p->lr_col, col, sizeof(col));
        std::memcpy(p->lr_row, row, sizeof(row));
    }
    for (int i = 0; i < D * D; ++i) p->w.w[i] = weights[i];
    if (!footprint_bound) p->star = star;
    return STENCIL_OK;
}

stencil_status_t stencil_plan_info(const stencil_plan_t* p, stencil_plan_info_t* info) {
    if (!p || !info) return fail(STENCIL_ERR_INVALID_ARG, "NULL argument");
    stencil_plan_info_t i{};
    i.ny = p->ny;
    i.nx = p->nx;
    i.radius = p->R;
    i.shape = p->star;
    i.dtype = p->dtype;
    i.boundary = p->boundary;
    i.compute = p->compute;
    i.kernel = p->kernel;
    i.tb_depth = p->k;
    i.threads = p->threads;
    i.halo_cols = p->H;
    i.tile_cols = p->bx;
    i.tile_rows = p->by;
    i.ctas = p->strips * p->tiles_y;
    i.smem_bytes = p->smem;
    i.workspace_bytes = (int64_t)((size_t)p->ny * p->nx * p->elem) +
                        (p->grid_mem ? (int64_t)grid_scratch_bytes((int)p->ny, (int)p->nx) : 0);
    if (p->pad[0]) i.workspace_bytes = 2 * (int64_t)((size_t)p->ny * p->pad_ld * p->elem);
    i.mma_n = p->umma_n;
    i.load = p->kernel == STENCIL_KERNEL_STREAM ? (p->tma ? STENCIL_LOAD_TMA : STENCIL_LOAD_CP_ASYNC) : 0;
    i.rank = p->kernel == STENCIL_KERNEL_LOWRANK ? p->lr_rank : 0;
    if (p->kernel == STENCIL_KERNEL_STREAM && p->tiles_on) {
        i.tb_depth = p->tiles.k;
        i.threads = 32 * p->tiles.warps;
        i.halo_cols = p->tiles.H;
        i.tile_cols = p->tiles.bx;
        i.tile_rows = p->tiles.by;
        i.ctas = p->tiles.strips * p->tiles.tiles_y;
        i.smem_bytes = 0;
    }
    if (p->kernel == STENCIL_KERNEL_STREAM && p->warp_nc && !p->tiles_on) {
        i.threads = 32;
        i.halo_cols = kWarpDepth;
        i.tile_cols = p->warp_bx;
        i.tile_rows = p->warp_by;
        i.ctas = p->warp_strips * p->warp_tiles;
        i.smem_bytes = 0;
    }
    if (p->kernel == STENCIL_KERNEL_RESIDENT && p->grid_on) {
        i.tb_depth = 0;  // every step of a run in one launch
        i.threads = 32 * p->grid.warps;
        i.halo_cols = p->grid.H;
        i.tile_cols = p->grid.bx;
        i.tile_rows = p->grid.by;
        i.ctas = 1;  // the cluster size: its CTAs, one per tile, are not clustered
        i.smem_bytes = 0;
    } else if (p->kernel == STENCIL_KERNEL_RESIDENT) {
        i.tb_depth = 0;  // every step of a run in one launch
        i.threads = resident_threads();
        i.halo_cols = p->R;
        i.tile_cols = (int)p->nx;
        i.tile_rows = p->res_rp;
        i.ctas = p->res_c;
        i.smem_bytes = p->res_smem;
    }
    if (p->umma_n) {
        i.threads = box49_umma_threads(p->umma_n);
        i.ctas = p->umma_ctas;
        i.smem_bytes = box49_umma_smem_bytes(p->compute == STENCIL_COMPUTE_TC_TF32, p->umma_n);
        i.tile_rows = box49_umma_tile_rows(p->umma_n);
    }
    if (p->umma_n && p->phase) {
        const int tf32 = p->compute == STENCIL_COMPUTE_TC_TF32;
        i.mma_n = 128;  // the widest MMA: four column blocks of 32
        i.ctas = p->phase_ctas;
        i.smem_bytes = box49_phase_smem_bytes(tf32);
        i.tile_rows = box49_phase_rows();
        i.tile_cols = box49_phase_cols(tf32);
    }
    *info = i;
    return STENCIL_OK;
}

int64_t stencil_run_launches(const stencil_plan_t* p, int64_t T) {
    if (!p || T < 0) return -1;
    const int64_t n = (int64_t)launch_depths(p, T).size();
    return n + (n > 0 && use_padded(p, (size_t)n) ? 1 : 0);  // (the pass that pads the rows)
}

stencil_status_t stencil_run(stencil_plan_t* p, const void* in, void* out, int64_t T,
                             stencil_stream_t stream) {
    if (!p) return fail(STENCIL_ERR_INVALID_ARG, "plan is NULL");
    if (!in || !out) return fail(STENCIL_ERR_INVALID_ARG, "in/out is NULL");
    if (T < 0) return fail(STENCIL_ERR_INVALID_ARG, "T must be >= 0");
    cudaStream_t st = (cudaStream_t)stream;
    p->last_stream = st;
    const size_t bytes = (size_t)p->ny * p->nx * p->elem;
    if (p->opt.autotune && !p->tuned && T > 0 &&
        (p->kernel == STENCIL_KERNEL_TC || p->kernel == STENCIL_KERNEL_TC_UMMA)) {
        stencil_status_t s = autotune_tc(p, in, st);
        if (s != STENCIL_OK) return s;
        p->tuned = 1;
    }
    if (p->opt.autotune && !p->tuned && p->kernel == STENCIL_KERNEL_RESIDENT && T > 0) {
        stencil_status_t s = autotune_resident(p, in, st);
        if (s != STENCIL_OK) return s;
        p->tuned = 1;
    }
    if (p->opt.autotune && !p->tuned && p->kernel == STENCIL_KERNEL_STREAM && T > 0) {
        stencil_status_t s = autotune(p, in, st);
        if (s != STENCIL_OK) return s;
        p->tuned = 1;
    }
    if (T == 0) {
        if (in != out) CK(cudaMemcpyAsync(out, in, bytes, cudaMemcpyDeviceToDevice, st));
        return STENCIL_OK;
    }
    std::vector<int> depths = launch_depths(p, T);
    const void* src = in;
    if (p->kernel == STENCIL_KERNEL_RESIDENT && p->grid_on && in == out && T == 1 && !cluster_run(p, T, true)) {
        // a single step in place has no exchange that orders the reads before the writes
        CK(cudaMemcpyAsync(p->ws, in, bytes, cudaMemcpyDeviceToDevice, st));
        src = p->ws;
    }
    if (p->kernel == STENCIL_KERNEL_RESIDENT) {
        // one launch reads all of its input before it writes any output
        for (size_t i = 0; i < depths.size(); ++i) {
            const bool tiles = p->grid_on;
            stencil_status_t s = launch_once(p, src, out, depths[i], st);
            if (s == STENCIL_ERR_UNSUPPORTED && tiles && !p->grid_on) {
                // (nothing was launched: the kernel that launch_once put in its place takes the run)
                return stencil_run(p, src == p->ws ? in : src, out, T - (int64_t)i * (1 << 30), stream);
            }
            if (s != STENCIL_OK) return s;
            src = out;
        }
        return STENCIL_OK;
    }
    if (use_padded(p, depths.size())) return run_padded(p, in, out, depths, st);
    if (in == out && depths.size() % 2 == 1) {
        // An odd launch count would make launch 1 write the grid it reads.
        // Split one launch in two when possible, else stage the input.
        auto it = std::find_if(depths.begin(), depths.end(), [](int d) { return d >= 2; });
        if (it != depths.end()) {
            const int d = *it;
            *it = d / 2;
            depths.insert(it, d - d / 2);
        } else {
            CK(cudaMemcpyAsync(p->ws, in, bytes, cudaMemcpyDeviceToDevice, st));
            src = p->ws;
        }
    }
    const size_t L = depths.size();
    for (size_t i = 0; i < L; ++i) {
        // Launch i (0-based) writes `out` when L-1-i is even, else the workspace.
        void* dst = ((L - 1 - i) % 2 == 0) ? out : p->ws;
        stencil_status_t s = launch_once(p, src, dst, depths[i], st, i == 0, i + 1 == L);
        if (s != STENCIL_OK) return s;
        src = dst;
    }
    return STENCIL_OK;
}

stencil_status_t stencil_run_host_async(stencil_plan_t* p, const void* in_host, void* out_host,
                                        int64_t T, stencil_stream_t stream) {
    if (!p) return fail(STENCIL_ERR_INVALID_ARG, "plan is NULL");
    if (!in_host || !out_host) return fail(STENCIL_ERR_INVALID_ARG, "in/out is NULL");
    if (T < 0) return fail(STENCIL_ERR_INVALID_ARG, "T must be >= 0");
    const size_t bytes = (size_t)p->ny * p->nx * p->elem;
    if (!p->host_in) {
        if (cudaMalloc(&p->host_in, bytes) != cudaSuccess) {
            cudaGetLastError();
            p->host_in = nullptr;
            return fail(STENCIL_ERR_OOM, "cudaMalloc of the staging input failed");
        }
    }
    if (!p->host_out) {
        if (cudaMalloc(&p->host_out, bytes) != cudaSuccess) {
            cudaGetLastError();
            p->host_out = nullptr;
            return fail(STENCIL_ERR_OOM, "cudaMalloc of the staging output failed");
        }
    }
    cudaStream_t st = (cudaStream_t)stream;
    CK(cudaMemcpyAsync(p->host_in, in_host, bytes, cudaMemcpyHostToDevice, st));
    stencil_status_t s = stencil_run(p, p->host_in, p->host_out, T, stream);
    if (s != STENCIL_OK) return s;
    CK(cudaMemcpyAsync(out_host, p->host_out, bytes, cudaMemcpyDeviceToHost, st));
    return STENCIL_OK;
}

stencil_status_t stencil_run_host(stencil_plan_t* p, const void* in_host, void* out_host,
                                  int64_t T, stencil_stream_t stream) {
    stencil_status_t s = stencil_run_host_async(p, in_host, out_host, T, stream);
    if (s != STENCIL_OK) return s;
    CK(cudaStreamSynchronize((cudaStream_t)stream));
    return STENCIL_OK;
}

stencil_status_t stencil_plan_status(stencil_plan_t* p) {
    if (!p) return fail(STENCIL_ERR_INVALID_ARG, "plan is NULL");
    CK(cudaStreamSynchronize(p->last_stream));
    unsigned int word = 0;
    CK(cudaMemcpy(&word, p->status, sizeof(word), cudaMemcpyDeviceToHost));
    CK(cudaMemset(p->status, 0, sizeof(word)));
    if (word == 0) return STENCIL_OK;
    return word == STENCIL_ERR_TIMEOUT ? STENCIL_ERR_TIMEOUT : STENCIL_ERR_DEVICE_CHECK;
}

}  // extern "C"
