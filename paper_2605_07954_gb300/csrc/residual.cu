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

cudaError_t plan_zero_now(const stencil_plan_t* p, void* ptr, size_t bytes);
bool plan_keep_sums(stencil_plan_t* p, bool on);
stencil_status_t plan_run_last_two(stencil_plan_t* p, const void* in, void* g1, void* g2, void* g0, int64_t m,
                                   cudaStream_t st, const void** prev, const void** next);

constexpr int kResBlocks = 1024;  // CTAs of a norm at most

// CTAs of a norm over n points: the last one to finish counts ~3 ns for each, a pass
// over 1024 points of a CTA takes ~0.7 us unless other CTAs hide it.  Steps with a
// check each, 9-point box, 608 | 1024 CTAs, us: 1000^2 20.7 | 23.9, 2048^2 28.9 | 30.9,
// 4096^2 66.2 | 62.2, 8192^2 230 | 210.
static unsigned residual_blocks(long long n) {
    const long long many = (n + 8191) / 8192, few = std::min(608LL, (n + 1023) / 1024);
    return (unsigned)std::min<long long>(kResBlocks, std::max(many, few));
}

// A running sum of squared differences, at no less than FP64's accuracy.  FP64 FMAs
// run at 1/64 of the FP32 rate here, so half of the terms (WIDE) take one of them
// each and the other half FP32 arithmetic that keeps every rounding error: the
// difference d + e = a - b and the square p + pe = d^2 are exact (TwoDiff, FMA), p
// goes into `s` and the errors into `c` with their own errors (TwoSum), and those
// plainly into `low`; 2^-70 of the sum is dropped.  Per thread, against exact sums
// of 16 to 1024 random terms, the FP32 half is within 1e-16 and a plain FP64 sum
// within 3e-15.  Terms whose square or its error would leave the FP32 range are
// summed in FP64 from the start: below 2^-40, and above 2^40, so that no number of
// terms that a thread can meet overflows `s`.
struct SquareSum {
    float s = 0.f, c = 0.f, low = 0.f;
    double wide = 0.0;
    // acc + v, and the rounding error of that addition
    static __device__ __forceinline__ float two_sum(float& acc, float v) {
        const float n = acc + v, y = n - acc, err = (acc - (n - y)) + (v - y);
        acc = n;
        return err;
    }
    template <bool WIDE>
    __device__ __forceinline__ void add(float a, float b) {
        const float d = a - b, z = d - a;
        const float e = (a - (d - z)) - (b + z);  // a - b = d + e
        const float m = fabsf(d);
        if (m >= 0x1p-40f && m <= 0x1p+40f) {
            if (WIDE) {
                // |d| as a double by its bits (a normal number: 896 is the difference of the exponents' biases)
                const unsigned u = __float_as_uint(m);
                const double w = __hiloint2double((int)((u >> 3) + (896u << 20)), (int)(u << 29));
                wide = fma(w, w, wide);
            } else {
                const float p = __fmul_rn(d, d), pe = fmaf(d, d, -p);  // (never fused into the sum)
                const float l = two_sum(c, two_sum(s, p));
                low += l + two_sum(c, pe);
            }
            if (e != 0.f) {  // (a and b within a factor of two differ by a float)
                const float d2 = 2.f * d, x = __fmul_rn(d2, e), xe = fmaf(d2, e, -x);
                low += two_sum(c, x) + fmaf(e, e, xe);
            }
        } else if (!(m == 0.f)) {  // (infinities and NaN too)
            const double w = (double)a - (double)b;
            wide = fma(w, w, wide);
        }
    }
    __device__ __forceinline__ double total() const { return ((double)s + ((double)c + (double)low)) + wide; }
};

// partials[block] = the block's share of sum (a - b)^2, in a fixed order; the last
// block to finish adds them in a fixed tree and writes *out = sqrt(sum).
// A check of 2048^2 FP32 takes 6-8 us, with plain FP64 sums, scalar loads and a second
// launch 39 + 4.  Two FP32 numbers a thread (2^-45 of the sum, and overflow beyond
// differences of 2^57) took 6.  A step and its check, 16384^2: 751 us; 918 with FP32
// alone (47 instructions a term), 830 with one term in four in FP64, 743 with two
// FP32 numbers.
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
    // four terms a pass: one 4-wide piece (vec; only the grid's last piece is cut), else 256 apart
    const int step = vec ? 1 : 256;
    for (long long i = lo + (vec ? 4 : 1) * (int)threadIdx.x; i < hi; i += 4 * 256) {
        float4 x = make_float4(0.f, 0.f, 0.f, 0.f), y = x;
        if (vec && i + 3 < hi) {
            x = Storage<TS>::load4(a + i);
            y = Storage<TS>::load4(b + i);
        } else {
            x.x = Storage<TS>::load1(a + i);
            y.x = Storage<TS>::load1(b + i);
            if (i + step < hi) x.y = Storage<TS>::load1(a + i + step), y.y = Storage<TS>::load1(b + i + step);
            if (i + 2 * step < hi) x.z = Storage<TS>::load1(a + i + 2 * step), y.z = Storage<TS>::load1(b + i + 2 * step);
            if (i + 3 * step < hi) x.w = Storage<TS>::load1(a + i + 3 * step), y.w = Storage<TS>::load1(b + i + 3 * step);
        }
        // (one copy of the two bodies: unrolled, a launch took 2 us longer to fetch them)
#pragma unroll 1
        for (int h = 0; h < 2; ++h) {
            q.add<true>(x.x, y.x);
            q.add<false>(x.y, y.y);
            x.x = x.z, x.y = x.w, y.x = y.z, y.y = y.w;
        }
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
        // the count of finished blocks starts at 0; every norm leaves it there
        const cudaError_t e = plan_zero_now(plan, sc->partials + kResBlocks, sizeof(unsigned));
        if (e != cudaSuccess) {
            cudaFree(sc->partials);
            sc->partials = nullptr;
            return rfail(STENCIL_ERR_CUDA, std::string("clearing the residual scratch: ") + cudaGetErrorString(e));
        }
    }
    unsigned* finished = reinterpret_cast<unsigned*>(sc->partials + kResBlocks);
    const unsigned blocks = residual_blocks(n);
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
            residual_kernel<float><<<blocks, 256, 0, st>>>(static_cast<const float*>(prev),
                                                               static_cast<const float*>(next), n, vec, sc->partials,
                                                               finished, residuals + j);
        else if (info.dtype == STENCIL_BF16)
            residual_kernel<__nv_bfloat16><<<blocks, 256, 0, st>>>(static_cast<const __nv_bfloat16*>(prev),
                                                                       static_cast<const __nv_bfloat16*>(next), n, vec,
                                                                       sc->partials, finished, residuals + j);
        else
            residual_kernel<__half><<<blocks, 256, 0, st>>>(static_cast<const __half*>(prev),
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
