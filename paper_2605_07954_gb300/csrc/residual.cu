// residual.cu -- T steps with a convergence check every m steps.
//
// The paper's host drives the wafer through long uninterrupted runs "save for
// periodic convergence checks" (Sec. IV).  stencil_run_residual runs T Jacobi
// steps (Sec. II-C) and, after every m-th step t, records
//     residual[j] = || u_t - u_{t-1} ||_2   (j = t/m - 1),
// the change made by that step, accumulated in FP64 over the whole grid.
//
// To have u_{t-1} and u_t both in memory, the last launch of a checked interval
// stores its last two time levels where the plan has a kernel that can
// (plan_run_last_two); else the interval runs m-1 steps and then one apart.
// residual_kernel then reads both grids.  The per-point arithmetic of every step
// is the one stencil_run uses, so the final state is bit-identical to
// stencil_run's.  The reduction is deterministic: a fixed grid of CTAs each sums
// a fixed index range, then the last one adds the CTA sums in a fixed tree.
#include <cuda_runtime.h>

#include <algorithm>
#include <new>
#include <string>

#include "../../include/stencil.h"
#include "common.cuh"

namespace gbst {

void** plan_aux_slot(stencil_plan_t* p, int id);
void plan_set_aux_free(stencil_plan_t* p, int id, void (*freer)(void*));

bool plan_keep_sums(stencil_plan_t* p, bool on);
stencil_status_t plan_run_last_two(stencil_plan_t* p, const void* in, void* g1, void* g2, void* g0, int64_t m,
                                   cudaStream_t st, const void** prev, const void** next);

constexpr int kResBlocks = 1024;

// A running sum of squared differences.  FP64 FMAs run at 1/64 of the FP32 rate
// here, so the sum is kept in two FP32 numbers: the difference, its square and
// the addition each with their rounding error (TwoDiff, FMA, TwoSum), about 45
// bits in all.  Differences whose square or its error would leave the FP32 range
// take the FP64 sum.
struct SquareSum {
    float s = 0.f, err = 0.f;
    double wide = 0.0;
    __device__ __forceinline__ void add(float a, float b) {
        const float d = a - b, z = d - a;
        const float e = (a - (d - z)) - (b + z);  // a - b = d + e
        const float m = fabsf(d);
        if (m >= 0x1p-40f && m <= 0x1p+60f) {
            const float p = d * d, pe = fmaf(d, d, -p);
            const float n = s + p, y = n - s;
            err += ((s - (n - y)) + (p - y)) + (pe + 2.f * d * e);
            s = n;
        } else if (!(m == 0.f)) {  // (infinities and NaN too)
            const double w = (double)a - (double)b;
            wide += w * w;
        }
    }
    __device__ __forceinline__ double total() const { return ((double)s + (double)err) + wide; }
};

// partials[block] = the block's share of sum (a - b)^2, in a fixed order; the last
// block to finish adds them in a fixed tree and writes *out = sqrt(sum).
// 2048^2 FP32: 6 us, against 39 + 4 for FP64 sums of scalar loads and a second launch.
template <typename TS>
__global__ void __launch_bounds__(256)
    residual_kernel(const TS* __restrict__ a, const TS* __restrict__ b, long long n, int vec,
                    double* __restrict__ partials, unsigned* __restrict__ finished, double* __restrict__ out) {
    __shared__ double sh[256];
    __shared__ bool s_last;
    // whole multiples of 4 per block, so that its chunks stay aligned
    const long long chunk = ((n + gridDim.x - 1) / gridDim.x + 3) / 4 * 4;
    const long long lo = (long long)blockIdx.x * chunk;
    const long long hi = lo + chunk < n ? lo + chunk : n;
    SquareSum q;
    if (vec) {
        long long i = lo + 4 * threadIdx.x;
        for (; i + 3 < hi; i += 4 * 256) {
            const float4 x = Storage<TS>::load4(a + i), y = Storage<TS>::load4(b + i);
            q.add(x.x, y.x);
            q.add(x.y, y.y);
            q.add(x.z, y.z);
            q.add(x.w, y.w);
        }
        for (; i < hi; ++i) q.add(Storage<TS>::load1(a + i), Storage<TS>::load1(b + i));  // (one thread's tail)
    } else {
        for (long long i = lo + threadIdx.x; i < hi; i += 256) q.add(Storage<TS>::load1(a + i), Storage<TS>::load1(b + i));
    }
    sh[threadIdx.x] = q.total();
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if (threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        partials[blockIdx.x] = sh[0];
        __threadfence();
        s_last = atomicAdd(finished, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    double s = 0.0;
    for (int i = threadIdx.x; i < (int)gridDim.x; i += 256) s += __ldcg(partials + i);
    sh[threadIdx.x] = s;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if (threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        *out = sqrt(sh[0]);
        *finished = 0u;  // for the next launch
    }
}

}  // namespace gbst

using namespace gbst;

namespace {

thread_local std::string g_res_error;

stencil_status_t rfail(stencil_status_t st, const std::string& msg) {
    g_res_error = msg;
    return st;
}

#define RCK(call)                                                                           \
    do {                                                                                    \
        cudaError_t e_ = (call);                                                            \
        if (e_ != cudaSuccess)                                                              \
            return rfail(STENCIL_ERR_CUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
    } while (0)

struct ResScratch {
    char* grids = nullptr;  // three grids (two where there is no room for more)
    int count = 0;
    size_t bytes = 0;       // from one grid to the next
    double* partials = nullptr;  // kResBlocks sums, then the count of finished blocks
};

void res_scratch_free(void* v) {
    ResScratch* sc = static_cast<ResScratch*>(v);
    if (sc->grids) cudaFree(sc->grids);
    if (sc->partials) cudaFree(sc->partials);
    delete sc;
}

}  // namespace

extern "C" {

const char* stencil_residual_last_error(void) { return g_res_error.c_str(); }

stencil_status_t stencil_run_residual(stencil_plan_t* plan, const void* in, void* out, int64_t T,
                                      int64_t m, double* residuals, stencil_stream_t stream) {
    if (!plan || !in || !out || !residuals) return rfail(STENCIL_ERR_INVALID_ARG, "NULL argument");
    if (T < 0 || m < 1) return rfail(STENCIL_ERR_INVALID_ARG, "need T >= 0 and m >= 1");
    stencil_plan_info_t info{};
    stencil_status_t s = stencil_plan_info(plan, &info);
    if (s != STENCIL_OK) return rfail(s, "stencil_plan_info failed");
    const size_t elem = info.dtype == STENCIL_F32 ? 4 : 2;
    const long long n = info.ny * info.nx;
    const size_t bytes = (size_t)n * elem;
    cudaStream_t st = (cudaStream_t)stream;

    void** slot = plan_aux_slot(plan, 1);
    ResScratch* sc = static_cast<ResScratch*>(*slot);
    if (!sc) {
        sc = new (std::nothrow) ResScratch();
        if (!sc) return rfail(STENCIL_ERR_OOM, "host allocation failed");
        *slot = sc;
        plan_set_aux_free(plan, 1, res_scratch_free);
    }
    if (!sc->grids) {
        sc->bytes = (bytes + 255) / 256 * 256;
        sc->count = 3;
        if (cudaMalloc((void**)&sc->grids, 3 * sc->bytes) != cudaSuccess) {
            cudaGetLastError();
            sc->count = 2;
            if (cudaMalloc((void**)&sc->grids, 2 * sc->bytes) != cudaSuccess) {
                cudaGetLastError();
                sc->grids = nullptr;
                return rfail(STENCIL_ERR_OOM, "cudaMalloc of the residual scratch failed");
            }
        }
    }
    if (!sc->partials) {
        const size_t pb = sizeof(double) * kResBlocks + sizeof(unsigned);
        if (cudaMalloc((void**)&sc->partials, pb) != cudaSuccess) {
            cudaGetLastError();
            sc->partials = nullptr;
            return rfail(STENCIL_ERR_OOM, "cudaMalloc of the residual scratch failed");
        }
    }
    unsigned* finished = reinterpret_cast<unsigned*>(sc->partials + kResBlocks);
    RCK(cudaMemsetAsync(finished, 0, sizeof(unsigned), st));
    char* const G[3] = {sc->grids, sc->grids + sc->bytes, sc->count == 3 ? sc->grids + 2 * sc->bytes : nullptr};
    // (residuals resolve the last bits of the states)
    struct KeepSums {
        stencil_plan_t* p;
        const bool on;
        ~KeepSums() {
            if (on) plan_keep_sums(p, false);
        }
    } const kept{plan, T >= m && plan_keep_sums(plan, true)};
    const void* cur = in;
    int64_t t = 0, j = 0;
    while (t + m <= T) {
        // m steps to u_{t+m}, keeping u_{t+m-1}: in one go where the last launch can
        // store both, else m-1 steps (temporally blocked) and then one.
        // g0: `cur`'s own grid (or any, while cur is the caller's input), g1 and g2 the others
        const int c = cur == G[1] ? 1 : cur == G[2] && G[2] ? 2 : 0;
        void* const g0 = G[c];
        void* const g1 = G[sc->count == 3 ? (c + 1) % 3 : 1 - c];
        void* const g2 = sc->count == 3 ? G[(c + 2) % 3] : nullptr;
        const void* prev = cur;
        const void* next = nullptr;
        s = STENCIL_ERR_UNSUPPORTED;
        if (m > 1 && g2) s = plan_run_last_two(plan, cur, g1, g2, g0, m, st, &prev, &next);
        if (s == STENCIL_ERR_UNSUPPORTED) {
            void* to = g1;
            if (m > 1) {
                s = stencil_run(plan, cur, g1, m - 1, stream);
                if (s != STENCIL_OK) return rfail(s, std::string("run: ") + stencil_last_error());
                prev = g1;
                to = g0;  // (`cur` is no longer needed)
            }
            s = stencil_run(plan, prev, to, 1, stream);
            next = to;
        }
        if (s != STENCIL_OK) return rfail(s, std::string("run: ") + stencil_last_error());
        const int vec = ((uintptr_t)prev | (uintptr_t)next) % (4 * elem) == 0;
        if (info.dtype == STENCIL_F32)
            residual_kernel<float><<<kResBlocks, 256, 0, st>>>(static_cast<const float*>(prev),
                                                               static_cast<const float*>(next), n, vec, sc->partials,
                                                               finished, residuals + j);
        else if (info.dtype == STENCIL_BF16)
            residual_kernel<__nv_bfloat16><<<kResBlocks, 256, 0, st>>>(static_cast<const __nv_bfloat16*>(prev),
                                                                       static_cast<const __nv_bfloat16*>(next), n, vec,
                                                                       sc->partials, finished, residuals + j);
        else
            residual_kernel<__half><<<kResBlocks, 256, 0, st>>>(static_cast<const __half*>(prev),
                                                                static_cast<const __half*>(next), n, vec, sc->partials,
                                                                finished, residuals + j);
        RCK(cudaGetLastError());
        cur = next;
        t += m;
        ++j;
    }
    // the remaining T mod m steps, straight into `out`
    s = stencil_run(plan, cur, out, T - t, stream);
    if (s != STENCIL_OK) return rfail(s, std::string("run: ") + stencil_last_error());
    return STENCIL_OK;
}

}  // extern "C"
