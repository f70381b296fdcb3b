// sweep_grid.cuh -- medium and small grids held in the registers of the whole
// chip, all T steps of a run in one cooperative launch (sm_103a).
//
// The Jacobi update of Sec. II-C as the streaming kernel computes it (same
// products in the same order, so the same bits for FP32 storage; the PLAIN kernels
// have the cluster-resident kernel's order and bits, for the grids that it would
// take: FP64 residuals and gradients resolve the difference), for grids
// that fit on the chip as one register tile per SM.  A CTA stages its tile with
// a halo of Hy = R*k rows and H >= R*k columns per side (none at the grid's own
// edges): warp w keeps staged rows [w*RB, w*RB+RB), each lane 4 adjacent columns
// of them (128 columns per warp).  The steps run in groups of k (temporal
// blocking: the paper's per-tile halo of Sec. IV-A made k times deeper):
//   1. every step: a warp publishes its first and last R rows to the warps
//      above and below through shared memory (double-buffered, one barrier),
//      takes the neighbouring columns by shuffles and updates its rows in
//      place, row by row, with 2R+1 partial sums per column in registers.
//      The outermost R rows and columns of what is still valid are lost; after
//      k steps the tile's own points remain.
//   2. after a group, the points within the halo depth of the tile's border go
//      to an exchange grid in global memory as (value, epoch) pairs of 8 bytes,
//      and every thread reads its own halo points back, repeating until the
//      epochs are this group's.  A pair is one 64-bit access, so it needs no
//      fence and no flag: an exchange costs one store and one load through L2
//      instead of store, fence, flag, poll, load.  Two exchange grids alternate;
//      a tile writes epoch e + 2 over epoch e only after it has read epoch
//      e + 1 of every tile that reads from it, which those wrote after they had
//      read epoch e.
// The state stays FP32 in registers between the first read and the last write.
// Points outside the grid read as zero at every step (zero rule, Sec. IV-A) or
// are wrapped images (periodic): a lane at the grid's left or right edge takes
// zeros instead of a neighbour's columns, a warp at the top or bottom edge reads
// zero rows, and only tiles whose edge cuts a lane's chunk or a warp's rows mask
// what they compute.
//
// What bounds it.  Latency: one CTA barrier per step for two to five warps a scheduler
// and one exchange of ~1.5 us per group (5-point star 1024^2: about 120 warp
// instructions per warp and step, 154 with the exchanges, issue 44 %, FMA pipe 31 %;
// 13-point star 512^2 41 %, 28 %); the cost model in sweep_grid.cu weighs the two.
// The cluster-resident kernel runs such grids on at most 16 SMs at ~0.7 us of
// cluster barrier per step, the streaming kernel at 15-20 us of launch, pipeline
// fill and drain per k steps.  Measured (FP32, GB300): 5-point star 1024^2, 1000
// steps, 802 us (streaming kernel 2559: 410 -> 1308 GStencil/s); 512^2, 100
// steps, 52 us (cluster-resident 219); 13-point star 130 x 517, 20 steps, 24 us
// (cluster-resident 74).  Tried and not kept: flags with a fence instead of
// marked pairs (an exchange cost twice as much), 16 rows per warp (fewer warps
// to hide latency: up to twice as slow at 1024^2), two or three CTAs per SM with
// smaller tiles (3-25 % slower: more halo rows than they hide).
//
// One group of steps exchanges nothing, so a launch of at most k steps is also an
// ordinary kernel over any number of tiles (launch_tiles): grids a little too
// large for one tile per SM, and periodic ragged rows (the lines and both sides'
// times stand at choose_tiles in plan.cu).
//
// Waits.  Tiles wait for one another, so the launch is cooperative (all CTAs
// resident).  Each wait is bounded (globaltimer limit and an iteration cap): an
// expired one records STENCIL_ERR_TIMEOUT, raises an abort flag that every
// waiting thread reads, and the launch ends.  Epochs only grow: a launch counts
// its groups from the generation word, which the last CTA to leave moves past
// them, so nothing has to be cleared between launches and a replayed graph
// works like a first run.
#pragma once

#include <type_traits>
#include <utility>

#include "../../include/stencil.h"
#include "common.cuh"
#include "sweep_stream.cuh"

namespace gbst {

constexpr int kGridCols = 128;  // staged columns of a tile (32 lanes x 4)
// control words, 64 bytes apart: generation, exit counter, abort flag
constexpr int kGridCtlStride = 16;
constexpr int kGridCtlInts = 3 * kGridCtlStride;

struct GridParams {
    const void* in;
    void* out;
    uint2* xbuf[2];   // exchange grids: ny rows of xld (value, epoch) pairs
    int* ctl;         // control words (null: a launch of at most k steps, which exchanges nothing)
    unsigned* status;
    long long wait_ns;
    int ny, nx, ld, xld;
    int T, k;         // steps of this launch; steps per exchange
    int H, Hy;        // halo columns (multiple of 4, >= R*k) and rows (>= R*k)
    int bx, by, strips, tiles_y;
    int periodic;
    int dtype;        // storage type of in and out
    int vec;          // rows of in and out aligned for 4-element access
    float* states;    // STATES kernels: step i, state_first <= i < T, also stores its result (FP32, dense)
    long long state_stride;  // ... at states + (i - state_first) * state_stride
    int state_first;
    int withhold;     // test hook: tile 0 marks its border points with no epoch, so waits run out
    Weights w;
    WeightPairs w2;
};

// Weights of one launch.  The (w, w) pairs that packed FMAs use are pinned in
// registers (left to itself the compiler may reload them from the constant
// bank at every use).  Footprints whose products run as scalar FMAs
// (stream_scalar_weights, and the centre row of the 13-point star) take theirs
// from the constant bank.
template <int R, bool STAR>
struct GridWeights {
    static constexpr int D = 2 * R + 1;
    static constexpr bool kScalar = stream_scalar_weights(R, STAR);
    const GridParams& p;
    float2 reg[kScalar ? 1 : D * D];
    __device__ __forceinline__ GridWeights(const GridParams& prm) : p(prm) {
        if constexpr (!kScalar) {
#pragma unroll
            for (int i = 0; i < D * D; ++i)
                if (pinned(i)) {
                    float w = p.w.w[i];
                    asm volatile("" : "+f"(w));
                    reg[i] = make_float2(w, w);
                }
        }
    }
    static __host__ __device__ constexpr bool pinned(int i) {
        if (kScalar) return false;
        if (!STAR) return true;
        if (R == 3) return i % D == R && i / D != R;  // the centre row runs as scalar FMAs
        return i % D == R || i / D == R;
    }
    __device__ __forceinline__ float2 w2(int i) const { return pinned(i) ? reg[i] : p.w2.w2[i]; }
};

// Largest CTA per instantiation: what the register file holds at the
// registers a thread needs (RB * 4 for the tile, (2R+1) * 4 partial sums, the
// weight pairs and about 40 more).
__host__ __device__ constexpr int grid_max_threads(int R, int RB) {
    return RB == 4 ? 768 : R == 1 ? 640 : 512;
}

// Shared memory: the edge rows (2 parities x warps x first and last R rows)
// and R zero rows, 32 chunks of 16 bytes each.
__host__ __device__ constexpr int grid_smem_bytes(int R, int warps) { return (4 * warps + 1) * R * 32 * 16; }

// Which lanes read zeros instead of a neighbour's columns, and which columns of
// the lane's chunk and rows of the warp lie in the grid (masked tiles).
struct GridEdges {
    bool zl, zr;        // left / right neighbour columns read as zero
    unsigned m[4];      // ~0: column in the grid
    int yrow0, ny;      // grid row of the warp's first row
};

template <int... I, class F>
__device__ __forceinline__ void grid_for_rows(std::integer_sequence<int, I...>, F&& f) {
    (f(std::integral_constant<int, I>{}), ...);
}

__device__ __forceinline__ float grid_keep(float v, unsigned m) {
    return __uint_as_float(__float_as_uint(v) & m);
}

// One step of a warp's RB rows in place.  `top` / `bot`: the R staged rows
// above and below (32 chunks per row, as column pairs); MASK: points outside
// the grid are forced to zero.
//
// PLAIN: every output adds its products row by row with dx ascending, the
// cluster-resident kernel's order, in place of the streaming kernel's (own chunk
// first).
template <int R, bool STAR, int RB, bool MASK, bool PLAIN, class WS>
__device__ __forceinline__ void grid_step(const WS& ws, float2 (&u)[RB][2], const float4* top, const float4* bot,
                                          int lane, const GridEdges& ed) {
    constexpr int D = 2 * R + 1;
    constexpr unsigned FULL = 0xffffffffu;
    float2 acc[D][2];
#pragma unroll
    for (int m = 0; m < D; ++m) acc[m][0] = acc[m][1] = make_float2(0.f, 0.f);
    auto left = [&](float v) {
        const float s = __shfl_up_sync(FULL, v, 1);
        return ed.zl ? 0.f : s;
    };
    auto right = [&](float v) {
        const float s = __shfl_down_sync(FULL, v, 1);
        return ed.zr ? 0.f : s;
    };
    // (a fold over the rows: the loop form left the 13-point star's arrays in local memory)
    grid_for_rows(std::make_integer_sequence<int, RB + 2 * R>{}, [&](auto ic) {
        constexpr int i = decltype(ic)::value;
        // input row i - R of the warp's tile
        float2 Pa, Pb;
        constexpr bool halo_row = i < R || i >= RB + R;
        if constexpr (halo_row) {
            const float4 q = i < R ? top[i * 32 + lane] : bot[(i - RB - R) * 32 + lane];
            Pa = make_float2(q.x, q.y);
            Pb = make_float2(q.z, q.w);
        } else {
            Pa = u[i - R][0];
            Pb = u[i - R][1];
        }
        if constexpr (PLAIN) {
            // q[d]: the output pairs' operands at column offset d - R
            float2 q0[D], q1[D];
            constexpr bool centre = STAR && halo_row;
            if constexpr (R == 1) {
                q0[1] = Pa;
                q1[1] = Pb;
                if constexpr (!centre) {
                    q0[0] = make_float2(left(Pb.y), Pb.x);
                    q0[2] = Pb;
                    q1[0] = Pa;
                    q1[2] = make_float2(Pa.y, right(Pa.x));
                }
            } else if constexpr (centre) {
                q0[R] = Pa;
                q1[R] = Pb;
            } else {
                float ext[4 + 2 * R];
                ext[R + 0] = Pa.x;
                ext[R + 1] = Pa.y;
                ext[R + 2] = Pb.x;
                ext[R + 3] = Pb.y;
                ext[R - 1] = left(Pb.y);
                ext[R - 2] = left(Pb.x);
                if (R == 3) ext[0] = left(Pa.y);
                ext[R + 4] = right(Pa.x);
                ext[R + 5] = right(Pa.y);
                if (R == 3) ext[R + 6] = right(Pb.x);
#pragma unroll
                for (int d = 0; d < D; ++d) {
                    q0[d] = make_float2(ext[d], ext[d + 1]);
                    q1[d] = make_float2(ext[d + 2], ext[d + 3]);
                }
            }
#pragma unroll
            for (int a = 0; a < D; ++a) {  // weight row: output row i - a
                if (i - a < 0 || i - a >= RB) continue;
                const int slot = (i - a + R) % D;
                if (a == 0) acc[slot][0] = acc[slot][1] = make_float2(0.f, 0.f);
#pragma unroll
                for (int d = 0; d < D; ++d) {
                    if (STAR && a != R && d != R) continue;
                    if (WS::pinned(a * D + d)) {
                        acc[slot][0] = __ffma2_rn(ws.w2(a * D + d), q0[d], acc[slot][0]);
                        acc[slot][1] = __ffma2_rn(ws.w2(a * D + d), q1[d], acc[slot][1]);
                    } else {  // weights from the constant bank
                        const float w = ws.p.w.w[a * D + d];
                        acc[slot][0] = make_float2(fmaf(w, q0[d].x, acc[slot][0].x), fmaf(w, q0[d].y, acc[slot][0].y));
                        acc[slot][1] = make_float2(fmaf(w, q1[d].x, acc[slot][1].x), fmaf(w, q1[d].y, acc[slot][1].y));
                    }
                }
            }
        } else if constexpr (R == 1) {
            own_products<R, STAR, 0, 2 * R>(ws, acc, Pa, Pb, i);
            if constexpr (!(STAR && halo_row)) {
                ExtRow<R> ext;
                ext.Pa = Pa;
                ext.Pb = Pb;
                ext.hl = left(Pb.y);
                ext.hr = right(Pa.x);
                halo_products<R, STAR, 0, 2 * R>(ws, acc, ext, i);
            }
        } else {
            own_products_adj<R, STAR, 0, 2 * R>(ws, acc, Pa, Pb, make_float2(Pa.y, Pb.x), i);
            if constexpr (!(STAR && halo_row)) {
                float4 lft = make_float4(0.f, 0.f, 0.f, 0.f), rgt = lft;
                if (R == 3) lft.y = left(Pa.y);
                lft.z = left(Pb.x);
                lft.w = left(Pb.y);
                rgt.x = right(Pa.x);
                rgt.y = right(Pa.y);
                if (R == 3) rgt.z = right(Pb.x);
                if constexpr (STAR && R == 3) {
                    halo_products_star3(ws, acc, lft, rgt, Pa, Pb, i);
                } else {
                    float ext[4 + 2 * R];
                    ext[R + 0] = Pa.x;
                    ext[R + 1] = Pa.y;
                    ext[R + 2] = Pb.x;
                    ext[R + 3] = Pb.y;
                    const float l4[4] = {lft.x, lft.y, lft.z, lft.w}, r4[4] = {rgt.x, rgt.y, rgt.z, rgt.w};
#pragma unroll
                    for (int e = 0; e < R; ++e) {
                        ext[e] = l4[4 - R + e];
                        ext[R + 4 + e] = r4[e];
                    }
                    halo_products_adj<R, STAR, 0, 2 * R>(ws, acc, ext, i);
                }
            }
        }
        if constexpr (i >= 2 * R) {  // output row i - 2R is complete (its input row was consumed R rows ago)
            constexpr int o = i - 2 * R, slot = (i - R + D) % D;
            float2 A0 = acc[slot][0], A1 = acc[slot][1];
            if constexpr (MASK) {
                constexpr int e0y = R == 1 ? 2 : 1, e1x = R == 1 ? 1 : 2;  // column of A0.y, of A1.x
                const unsigned rm = (unsigned)(ed.yrow0 + o) < (unsigned)ed.ny ? ~0u : 0u;
                A0.x = grid_keep(A0.x, ed.m[0] & rm);
                A0.y = grid_keep(A0.y, ed.m[e0y] & rm);
                A1.x = grid_keep(A1.x, ed.m[e1x] & rm);
                A1.y = grid_keep(A1.y, ed.m[3] & rm);
            }
            u[o][0] = A0;
            u[o][1] = A1;
        }
    });
}

// Column pairs of a 4-column chunk: (c0, c2), (c1, c3) for radius 1, else
// (c0, c1), (c2, c3).
template <int R>
__device__ __forceinline__ void grid_to_pairs(float4 v, float2 (&u)[2]) {
    if (R == 1) {
        u[0] = make_float2(v.x, v.z);
        u[1] = make_float2(v.y, v.w);
    } else {
        u[0] = make_float2(v.x, v.y);
        u[1] = make_float2(v.z, v.w);
    }
}
template <int R>
__device__ __forceinline__ float4 grid_from_pairs(const float2 (&u)[2]) {
    return R == 1 ? make_float4(u[0].x, u[1].x, u[0].y, u[1].y) : make_float4(u[0].x, u[0].y, u[1].x, u[1].y);
}

__device__ __forceinline__ float grid_load1(const GridParams& p, long long i) {
    if (p.dtype == DT_F32) return __ldg(static_cast<const float*>(p.in) + i);
    if (p.dtype == DT_BF16) return Storage<__nv_bfloat16>::load1(static_cast<const __nv_bfloat16*>(p.in) + i);
    return Storage<__half>::load1(static_cast<const __half*>(p.in) + i);
}
__device__ __forceinline__ float4 grid_load4(const GridParams& p, long long i) {
    if (p.dtype == DT_F32) return Storage<float>::load4(static_cast<const float*>(p.in) + i);
    if (p.dtype == DT_BF16) return Storage<__nv_bfloat16>::load4(static_cast<const __nv_bfloat16*>(p.in) + i);
    return Storage<__half>::load4(static_cast<const __half*>(p.in) + i);
}
__device__ __forceinline__ void grid_store(const GridParams& p, long long i, float4 v, int n, bool vec) {
    const float e[4] = {v.x, v.y, v.z, v.w};
    if (p.dtype == DT_F32) {
        float* o = static_cast<float*>(p.out) + i;
        if (vec) Storage<float>::store4(o, v);
        else
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (j < n) o[j] = e[j];
    } else if (p.dtype == DT_BF16) {
        __nv_bfloat16* o = static_cast<__nv_bfloat16*>(p.out) + i;
        if (vec) Storage<__nv_bfloat16>::store4(o, v);
        else
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (j < n) Storage<__nv_bfloat16>::store1(o + j, e[j]);
    } else {
        __half* o = static_cast<__half*>(p.out) + i;
        if (vec) Storage<__half>::store4(o, v);
        else
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (j < n) Storage<__half>::store1(o + j, e[j]);
    }
}

// (value, epoch) pairs: each pair is one 64-bit access (two per instruction).
__device__ __forceinline__ unsigned long long grid_pair(float v, unsigned epoch) {
    return (unsigned long long)__float_as_uint(v) | (unsigned long long)epoch << 32;
}
__device__ __forceinline__ void grid_put4(uint2* p, float4 v, unsigned epoch, bool on) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %6, 0;\n\t"
        "@p st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};\n\t"
        "@p st.relaxed.gpu.global.v2.b64 [%3], {%4, %5};\n\t}" ::"l"(p),
        "l"(grid_pair(v.x, epoch)), "l"(grid_pair(v.y, epoch)), "l"(p + 2), "l"(grid_pair(v.z, epoch)),
        "l"(grid_pair(v.w, epoch)), "r"((unsigned)on)
        : "memory");
}
__device__ __forceinline__ void grid_get4(const uint2* p, unsigned long long (&q)[4], bool on) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %6, 0;\n\t"
        "@p ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%4];\n\t"
        "@p ld.relaxed.gpu.global.v2.b64 {%2, %3}, [%5];\n\t}"
        : "+l"(q[0]), "+l"(q[1]), "+l"(q[2]), "+l"(q[3])
        : "l"(p), "l"(p + 2), "r"((unsigned)on)
        : "memory");
}
__device__ __forceinline__ void grid_get1(const uint2* p, unsigned long long& q, bool on) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %2, 0;\n\t"
        "@p ld.relaxed.gpu.global.b64 %0, [%1];\n\t}"
        : "+l"(q)
        : "l"(p), "r"((unsigned)on)
        : "memory");
}

__device__ __forceinline__ int grid_wrap(int i, int n) {
    return (unsigned)i < (unsigned)n ? i : ((i % n) + n) % n;
}

// Every 64th try of a wait: whether to give up (the limit ran out, or another
// CTA gave up).  The same answer on every lane of the warp.
static __device__ __noinline__ bool grid_wait_over(const GridParams& p, unsigned it, long long& t0) {
    int* const abort_flag = p.ctl + 2 * kGridCtlStride;
    const long long now = st_now();
    if (t0 == 0) t0 = now;
    bool over = *(volatile int*)abort_flag != 0;
    if (now - t0 > p.wait_ns || it > (1u << 26)) {
        atomicCAS(p.status, 0u, (unsigned)STENCIL_ERR_TIMEOUT);
        atomicExch(abort_flag, 1);
        over = true;
    }
    return __any_sync(0xffffffffu, over);
}

// STATES: every step's result is stored as well (a variant of its own: the branch
// in the step loop cost the plain runs 6 %, 5-point star 512^2 x 100 steps 52.4 ->
// 55.5 us).
template <int R, bool STAR, int RB, bool STATES = false, bool PLAIN = false>
__global__ void __launch_bounds__(grid_max_threads(R, RB), 1)
    sweep_grid_kernel(const __grid_constant__ GridParams p) {
    extern __shared__ float4 grid_rows[];  // [parity][warp][first rows, last rows][R][32], then R zero rows
    __shared__ unsigned s_base;
    const int warps = blockDim.x >> 5;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int strip = (int)blockIdx.x % p.strips, trow = (int)blockIdx.x / p.strips;
    const int ny = p.ny, nx = p.nx, H = p.H, Hy = p.Hy;
    const bool per = p.periodic != 0;
    // Owned points [xo0, xo1) x [yo0, yo1) and the first staged column and row.
    // Zero rule: every tile stages bx + 2H columns and by + 2Hy rows, and owns
    // the halo depth too at the grid's edges; the last tile row is staged so
    // that it ends with the grid's last row.
    int xs, xo0, xo1, ys, yo0, yo1;
    if (per) {
        xo0 = strip * p.bx;
        xo1 = min(xo0 + p.bx, nx);
        xs = xo0 - H;
        yo0 = trow * p.by;
        yo1 = min(yo0 + p.by, ny);
        ys = yo0 - Hy;
    } else {
        xs = strip * p.bx;
        xo0 = strip ? xs + H : 0;
        xo1 = strip == p.strips - 1 ? nx : xs + p.bx + H;
        ys = trow * p.by;
        yo0 = trow ? ys + Hy : 0;
        yo1 = trow == p.tiles_y - 1 ? ny : ys + p.by + Hy;
        if (trow == p.tiles_y - 1) ys = max(0, min(ys, ny - warps * RB));
    }
    const int c = xs + 4 * lane;    // grid column of the lane's chunk
    const int yr = ys + warp * RB;  // grid row of the warp's first row
    unsigned* const gen = reinterpret_cast<unsigned*>(p.ctl);
    int* const leave = p.ctl + kGridCtlStride;
    int* const abort_flag = p.ctl + 2 * kGridCtlStride;
    const GridWeights<R, STAR> ws(p);

    // The generation this launch counts from: read before any CTA can leave
    // (the last one to leave moves it on).
    // (No control words: one group of steps, nothing to count.)
    if (threadIdx.x == 0) s_base = p.ctl ? *(volatile unsigned*)gen : 0u;
    float4* const zero_rows = grid_rows + 4 * warps * R * 32;
    for (int i = threadIdx.x; i < R * 32; i += blockDim.x) zero_rows[i] = make_float4(0.f, 0.f, 0.f, 0.f);

    GridEdges ed;
    ed.zl = lane == 0;
    ed.zr = lane == 31 || (!per && c + 4 >= nx);
#pragma unroll
    for (int e = 0; e < 4; ++e) ed.m[e] = per || c + e < nx ? ~0u : 0u;
    ed.yrow0 = per ? 0 : yr;
    ed.ny = per ? RB : ny;
    // Masks where the grid's edge cuts a lane's chunk, or the warp's rows.
    const bool mask = !per && ((nx % 4 != 0 && xs + kGridCols > nx) || (yr < ny && yr + RB > ny));
    // A warp whose rows no owned point needs (staged beyond the halo or the grid) computes nothing.
    const bool idle = yr >= yo1 + Hy || (!per && yr >= ny);

    // The initial state, halo included.
    const int cw = per ? grid_wrap(c, nx) : c;
    float2 u[RB][2];
#pragma unroll
    for (int r = 0; r < RB; ++r) {
        int y = yr + r;
        if (per) y = grid_wrap(y, ny);
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (per || (y < ny && c < nx)) {
            const long long row = (long long)y * p.ld;
            if (p.vec) {
                v = grid_load4(p, row + cw);
            } else {
                float e4[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    int x = c + e;
                    if (per) x = grid_wrap(x, nx);
                    e4[e] = x < nx ? grid_load1(p, row + x) : 0.f;
                }
                v = make_float4(e4[0], e4[1], e4[2], e4[3]);
            }
        }
        grid_to_pairs<R>(v, u[r]);
    }

    // The lane's chunk: owned, or halo that an owned point needs.  (Periodic
    // ragged widths: a chunk that holds wrapped images beyond the last column
    // counts as halo too; its own columns come back from the exchange grid.)
    const bool col_own = c >= xo0 && c < xo1;
    const bool col_halo = per ? c < xo0 || c + 4 > xo1 : !col_own;
    const bool col_need = c + 4 > xo0 - H && c < xo1 + H && (per || c < nx);
    const bool col_border = c < xo0 + H || c + 4 > xo1 - H;  // other tiles may need it
    bool bad = false;   // this thread's wait ran out, or it saw the abort flag
    bool dead = false;  // some thread of the CTA is bad: all leave together
    unsigned epoch = 0;
    int par = 0;  // parity of the step's row buffers
    for (int t = 0;;) {
        const int kk = min(p.k, p.T - t);
        for (int s = 0; s < kk; ++s) {
            float4* mine = grid_rows + ((par * warps + warp) * 2) * R * 32;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                mine[r * 32 + lane] = make_float4(u[r][0].x, u[r][0].y, u[r][1].x, u[r][1].y);
                mine[(R + r) * 32 + lane] = make_float4(u[RB - R + r][0].x, u[RB - R + r][0].y, u[RB - R + r][1].x,
                                                        u[RB - R + r][1].y);
            }
            if (s == 0) {
                dead = __syncthreads_or(bad) != 0;
                if (dead) break;
            } else {
                __syncthreads();
            }
            // the last rows of the warp above and the first rows of the warp below
            const float4* top = warp > 0 ? mine - R * 32 : zero_rows;
            const float4* bot = warp + 1 < warps ? mine + 2 * R * 32 : zero_rows;
            if (!idle) {
                if (mask) grid_step<R, STAR, RB, true, PLAIN>(ws, u, top, bot, lane, ed);
                else grid_step<R, STAR, RB, false, PLAIN>(ws, u, top, bot, lane, ed);
            }
            par ^= 1;
            if (STATES && t + s + 1 < p.T && t + s + 1 >= p.state_first && col_own) {
                float* st = p.states + (long long)(t + s + 1 - p.state_first) * p.state_stride;
                const int n = min(4, nx - c);
#pragma unroll
                for (int r = 0; r < RB; ++r) {
                    const int y = yr + r;
                    if (y < yo0 || y >= yo1) continue;
                    const float4 v = grid_from_pairs<R>(u[r]);
                    float* o = st + (long long)y * p.ld + c;
                    if (p.vec) {
                        Storage<float>::store4(o, v);
                    } else {
                        const float e[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                        for (int k = 0; k < 4; ++k)
                            if (k < n) o[k] = e[k];
                    }
                }
            }
        }
        if (t == 0) epoch = s_base;
        t += kk;
        if (dead || t >= p.T) break;

        // Exchange: publish the border, read the halo back.
        ++epoch;
        uint2* const xb = p.xbuf[epoch & 1];
        // (Straight-line predicated code, and the warp retries as one: branches
        // per row and lane made this part 1400 instructions for 16 rows.)
        if (yr < yo1 && yr + RB > yo0) {
            const unsigned mark = p.withhold && blockIdx.x == 0 ? 0u : epoch;
            uint2* row = xb + (long long)yr * p.xld + c;  // columns of the chunk beyond nx: the pitch's padding
#pragma unroll
            for (int r = 0; r < RB; ++r, row += p.xld) {
                const int y = yr + r;
                const bool own = col_own && y >= yo0 && y < yo1;
                grid_put4(row, grid_from_pairs<R>(u[r]), mark, own && (col_border || y < yo0 + Hy || y >= yo1 - Hy));
            }
        }
        constexpr int B = RB < 4 ? RB : 4;  // rows whose loads are in flight together
#pragma unroll
        for (int r0 = 0; r0 < RB; r0 += B) {
            unsigned need = 0;
#pragma unroll
            for (int r = 0; r < B; ++r) {
                const int y = yr + r0 + r;
                const bool halo = col_halo || y < yo0 || y >= yo1;  // (the tile's own points stay)
                if (halo && col_need && y >= yo0 - Hy && y < yo1 + Hy && (per || (unsigned)y < (unsigned)ny))
                    need |= 1u << r;
            }
            unsigned it = 0;
            long long t_wait = 0;
            while (__any_sync(0xffffffffu, need)) {
                unsigned long long q[B][4];
#pragma unroll
                for (int r = 0; r < B; ++r) {
                    const bool on = need >> r & 1u;
                    int y = yr + r0 + r;
                    if (per) y = grid_wrap(y, ny);
                    const uint2* row = xb + (long long)y * p.xld;
#pragma unroll
                    for (int e = 0; e < 4; ++e) q[r][e] = 0;
                    if (!per || nx % 4 == 0) {
                        grid_get4(row + cw, q[r], on);
                    } else {
#pragma unroll
                        for (int e = 0; e < 4; ++e) {  // (columns beyond the halo depth have no owner to wait for)
                            const bool use = c + e < xo1 + H;
                            if (!use) q[r][e] = grid_pair(0.f, epoch);
                            grid_get1(row + grid_wrap(c + e, nx), q[r][e], on && use);
                        }
                    }
                }
#pragma unroll
                for (int r = 0; r < B; ++r) {
                    bool got = need >> r & 1u;
                    float v[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        got = got && (unsigned)(q[r][e] >> 32) == epoch;
                        v[e] = __uint_as_float((unsigned)q[r][e]);
                    }
                    float2 n[2];
                    grid_to_pairs<R>(make_float4(v[0], v[1], v[2], v[3]), n);
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        u[r0 + r][h].x = got ? n[h].x : u[r0 + r][h].x;
                        u[r0 + r][h].y = got ? n[h].y : u[r0 + r][h].y;
                    }
                    need &= got ? ~(1u << r) : ~0u;
                }
                if ((++it & 63u) == 0u && grid_wait_over(p, it, t_wait)) {
                    bad = true;
                    break;
                }
            }
        }
    }

    if (col_own && !dead) {
#pragma unroll
        for (int r = 0; r < RB; ++r) {
            const int y = yr + r;
            if (y < yo0 || y >= yo1) continue;
            const int n = min(4, nx - c);
            grid_store(p, (long long)y * p.ld + c, grid_from_pairs<R>(u[r]), n, p.vec && n == 4);
        }
    }
    // Leave: the last CTA moves the generation past this launch's epochs.
    __syncthreads();
    if (threadIdx.x == 0 && p.ctl) {
        const unsigned groups = (unsigned)((p.T + p.k - 1) / p.k);
        if (atomicAdd(leave, 1) == (int)gridDim.x - 1) {
            atomicExch(leave, 0);
            atomicExch(abort_flag, 0);
            atomicExch(gen, s_base + groups - 1);
        }
    }
}

struct GridKernelRef {
    const void* fn;
    int max_threads;
};

}  // namespace gbst
