// sweep_warp.cuh -- one warp per tile: the radius-1 Jacobi sweep streamed down a
// strip by a single warp, K steps per pass (sm_103a).
//
// The same pipeline as the CTA-wide kernel (sweep_stream.cuh): rows of the
// strip arrive through a cp.async ring, K time levels follow one another down
// the rows with 2R+1 = 3 partial sums per column and level in registers, and
// only level K is stored.  But the strip is one warp wide (32 lanes x NC
// columns, H >= K halo columns per side recomputed by its neighbours), so the
// columns next to a lane's come by shuffles: no shared-memory edge arrays and no
// barrier, K per row there.  A lane's NC columns are held as NC/2 pairs (c_q,
// c_{q + NC/2}) for packed FP32x2 FMAs; of the pairs a tap reads only the two
// that straddle a neighbour's column are assembled.  Products are added in the
// CTA-wide kernel's order, so the results have the same bits.
//
// Zero rule: a lane at the grid's left or right edge takes zeros instead of its
// neighbour's columns; rows outside the grid are zeroed as levels complete
// them, in the groups of rows that can hold one; only a strip whose last
// chunk the right edge cuts masks columns.  Periodic grids load wrapped rows
// and columns and mask nothing.
//
// What bounds it: the FMA pipe (packed FMAs reach 83 % of it at best) and, for
// the 9-point box, registers: at NC = 8 and K = 8 its unrolled row step also
// outgrows the instruction cache (1818 GStencil/s at 8192^2; NC = 4: 2517,
// CTA-wide 2357).  The 5-point star fits: NC = 8, K = 8 4179, NC = 4 3620,
// CTA-wide 3415.  Radius 3 unrolls 7 rows per step and loses (13-point star
// 1209 against 1271 at best), so this form is radius 1 only.
#pragma once

#include <type_traits>
#include <utility>

#include "common.cuh"
#include "sweep_stream.cuh"

namespace gbst {

constexpr int kWarpRing = 4;  // rows in flight (a power of 2)

// Taps are added in two ascending passes (own-chunk columns first, as the
// CTA-wide kernel does): even columns take dx = 0, 1 then -1, odd ones -1, 0
// then 1, i.e. all in the first pass.
__host__ __device__ constexpr int warp_pass(int q, int dx) { return (q & 1) == 0 && dx < 0 ? 1 : 0; }

template <int... I, class F>
__device__ __forceinline__ void warp_for(std::integer_sequence<int, I...>, F&& f) {
    (f(std::integral_constant<int, I>{}), ...);
}

// The (w, w) pairs in registers (opaque, so that they are not reloaded at each use).
template <bool STAR>
struct WarpWeights {
    float2 reg[9];
    static __host__ __device__ constexpr bool used(int i) { return !STAR || i / 3 == 1 || i % 3 == 1; }
    template <class F>
    __device__ __forceinline__ explicit WarpWeights(F&& get) {
#pragma unroll
        for (int i = 0; i < 9; ++i)
            if (used(i)) {
                float w = get(i);
                asm volatile("" : "+f"(w));
                reg[i] = make_float2(w, w);
            }
    }
};

// Adds one arriving row to a level's partial sums: pairs P, left column L (-1),
// right column Q (NC); J: the row's index mod 3.
template <bool STAR, int NP, int J>
__device__ __forceinline__ void warp_row(const WarpWeights<STAR>& ws, float2 (&acc)[3][NP], const float2 (&P)[NP],
                                         float L, float Q) {
    warp_for(std::make_integer_sequence<int, 3>{}, [&](auto mc) {
        constexpr int m = decltype(mc)::value;
        constexpr int slot = (J - m + 7) % 3;
        // by passes over the taps, so that one weight serves several outputs in a row
        warp_for(std::make_integer_sequence<int, 6>{}, [&](auto pc) {
            constexpr int dx = decltype(pc)::value % 3 - 1, pass = decltype(pc)::value / 3;
            if constexpr (!STAR || m == 1 || dx == 0) {
                warp_for(std::make_integer_sequence<int, NP>{}, [&](auto qc) {
                    constexpr int q = decltype(qc)::value;
                    if constexpr (warp_pass(q, dx) == pass) {
                        constexpr int s = q + dx, wi = 3 * m + dx + 1;
                        float2 v;
                        if constexpr (s < 0) v = make_float2(L, P[NP - 1].x);
                        else if constexpr (s >= NP) v = make_float2(P[0].y, Q);
                        else v = P[s];
                        constexpr bool first = m == 0 && (STAR || dx == (q & 1 ? -1 : 0));
                        if constexpr (first) acc[slot][q] = fmul2(ws.reg[wi], v);
                        else acc[slot][q] = ffma2(ws.reg[wi], v, acc[slot][q]);
                    }
                });
            }
        });
    });
}

// Bytes of a warp's ring.
template <typename TS, int NC>
__host__ __device__ constexpr int warp_ring_bytes() { return kWarpRing * 32 * NC * (int)sizeof(TS); }

// Rows a tile loads beyond its last output row: K for the halo, 2 for rounding
// the row loop up to its unroll.
__host__ __device__ constexpr int warp_rows_after(int K) { return K + 3; }

// One tile: outputs [y0, y0 + by) x [x0, x0 + bx).  EDGE: the tile loads rows or
// columns outside the grid; CUT: the right edge may cut a chunk; ALL: level l+1
// is also stored to p.lvl_out[l] where that is not null (l < K-1).  p.bx and p.H are multiples of NC.
template <bool STAR, int K, typename TS, int NC, bool EDGE, bool CUT = EDGE, bool ALL = false>
__device__ __forceinline__ void warp_tile(const StreamParams& p, const WarpWeights<STAR>& ws, char* ring, int lane,
                                          int x0, int y0) {
    constexpr int NP = NC / 2, PF = kWarpRing, NQ = NC / 4;
    constexpr int CB = NC * (int)sizeof(TS);  // bytes of a lane's chunk
    constexpr int PB = 4 * (int)sizeof(TS);   // bytes of a 4-column piece
    constexpr unsigned FULL = 0xffffffffu;
    const int ny = (int)p.ny, nx = (int)p.nx;
    const long long ld = p.ld;
    const int c = x0 - p.H + NC * lane;
    const int ybeg = y0 - K;
    const int ylast = min(y0 + p.by, ny);
    const bool per = EDGE && p.periodic != 0;
    const bool mask = EDGE && !per;
    const bool zl = mask && (lane == 0 || c <= 0), zr = mask && (lane == 31 || c + NC >= nx);
    const bool cut = CUT && mask && nx % NC != 0 && x0 - p.H + 32 * NC > nx;  // the right edge cuts a chunk
    const int nsteps = ((ylast - y0) + 2 * K + 2) / 3 * 3;
    const TS* gin = static_cast<const TS*>(p.in);
    char* my = ring + lane * CB;
    const TS* src = gin + (EDGE ? 0 : (long long)ybeg * ld + c);
    bool pin[NQ];  // piece j of the chunk holds columns of the grid
    int pc[NQ];
#pragma unroll
    for (int j = 0; j < NQ; ++j) {
        const int cj = c + 4 * j;
        pin[j] = per || (cj >= 0 && cj < nx);
        pc[j] = per ? (int)wrap_index(cj, nx) : cj;
    }
    auto issue = [&](int s) {
        char* dst = my + (s & (PF - 1)) * (32 * CB);
        bool ok = s < nsteps;
        if constexpr (EDGE) {
            int y = ybeg + s;
            if (per) y = (int)wrap_index(y, ny);
            else ok = ok && y >= 0 && y < ny;
#pragma unroll
            for (int j = 0; j < NQ; ++j) {
                const bool o = ok && pin[j];
                cp_async<PB>(dst + j * PB, o ? gin + (long long)y * ld + pc[j] : gin, o);
            }
        } else {
            const TS* g = ok ? src + (long long)s * ld : gin;  // (past the tile: zero bytes are copied)
#pragma unroll
            for (int j = 0; j < NQ; ++j) cp_async<PB>(dst + j * PB, g + 4 * j, ok);
        }
        cp_async_commit();
    };
#pragma unroll
    for (int s = 0; s < PF - 1; ++s) issue(s);

    float2 acc[K][3][NP];
#pragma unroll
    for (int l = 0; l < K; ++l)
#pragma unroll
        for (int m = 0; m < 3; ++m)
#pragma unroll
            for (int q = 0; q < NP; ++q) acc[l][m][q] = make_float2(0.f, 0.f);

    bool st[NQ];
#pragma unroll
    for (int j = 0; j < NQ; ++j) {
        const int cj = c + 4 * j;
        st[j] = cj >= x0 && cj < x0 + p.bx && cj < nx;
    }
    TS* out = static_cast<TS*>(p.out) + c;
    auto store_row = [&](TS* o, const float2 (&X)[NP]) {
#pragma unroll
        for (int j = 0; j < NQ; ++j) {
            float e[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) e[i] = 4 * j + i < NP ? X[(4 * j + i) % NP].x : X[(4 * j + i) % NP].y;
            if (st[j]) Storage<TS>::store4(o + 4 * j, make_float4(e[0], e[1], e[2], e[3]));
        }
    };

    auto group = [&](int s0, auto mr) {
        [[maybe_unused]] constexpr bool MR = decltype(mr)::value;
        warp_for(std::make_integer_sequence<int, 3>{}, [&](auto jc) {
            constexpr int J = decltype(jc)::value;
            const int s = s0 + J;
            issue(s + PF - 1);
            cp_async_wait<PF - 1>();
            const char* slot = my + (s & (PF - 1)) * (32 * CB);
            float v[NC];
#pragma unroll
            for (int j = 0; j < NQ; ++j) {
                float q4[4];
                smem_chunk_to_f32<TS>(slot + j * PB, q4);
#pragma unroll
                for (int e = 0; e < 4; ++e) v[4 * j + e] = q4[e];
            }
            float2 X[NP];
#pragma unroll
            for (int q = 0; q < NP; ++q) X[q] = make_float2(v[q], v[q + NP]);
#pragma unroll
            for (int l = 0; l < K; ++l) {
                float L = __shfl_up_sync(FULL, X[NP - 1].y, 1);
                float Q = __shfl_down_sync(FULL, X[0].x, 1);
                if constexpr (EDGE) {
                    L = zl ? 0.f : L;
                    Q = zr ? 0.f : Q;
                }
                warp_row<STAR, NP, J>(ws, acc[l], X, L, Q);
                constexpr int done = (J + 2) % 3;
#pragma unroll
                for (int q = 0; q < NP; ++q) X[q] = acc[l][done][q];
                if constexpr (EDGE) {
                    if constexpr (MR) {
                        if (mask && (unsigned)(ybeg - (l + 1) + s) >= (unsigned)ny) {
#pragma unroll
                            for (int q = 0; q < NP; ++q) X[q] = make_float2(0.f, 0.f);
                        }
                    }
                    if (CUT && cut) {
#pragma unroll
                        for (int q = 0; q < NP; ++q) {
                            X[q].x = c + q < nx ? X[q].x : 0.f;
                            X[q].y = c + q + NP < nx ? X[q].y : 0.f;
                        }
                    }
                }
                if constexpr (ALL) {
                    const int yl = ybeg - (l + 1) + s;
                    if (l < K - 1 && p.lvl_out[l] && yl >= y0 && yl < ylast)
                        store_row(static_cast<TS*>(p.lvl_out[l]) + c + (long long)yl * ld, X);
                }
            }
            const int yo = ybeg - K + s;
            if (yo >= y0 && yo < ylast) store_row(out + (long long)yo * ld, X);
        });
    };
    for (int s0 = 0; s0 < nsteps; s0 += 3) {
        if constexpr (EDGE) {
            // level rows completed in this group: ybeg + s0 - K .. ybeg + s0 + 1
            if (mask && (ybeg + s0 - K < 0 || ybeg + s0 + 3 > ny)) group(s0, std::true_type{});
            else group(s0, std::false_type{});
        } else {
            group(s0, std::false_type{});
        }
    }
    cp_async_wait<0>();
}

// Warps per SM the registers must allow: the 5-point star at NC = 8 takes 220
// registers (8 warps), the NC = 4 forms fit 128 (16).
__host__ __device__ constexpr int warp_min_blocks(int NC) { return NC == 8 ? 8 : 16; }

// A launch of one-warp CTAs over a whole grid: p.strips x tile rows, edge tiles first.
// (ALL and NC = 8 kernels take widths that are a multiple of NC.)
template <bool STAR, int K, typename TS, int NC, bool ALL = false>
__global__ void __launch_bounds__(32, warp_min_blocks(NC)) sweep_warp_kernel(const __grid_constant__ StreamParams p) {
    __shared__ __align__(16) char ring[warp_ring_bytes<TS, NC>()];
    const int lane = threadIdx.x;
    int strip, tile;
    stream_tile_of(blockIdx.x, p.strips, gridDim.x / p.strips, strip, tile);
    const int x0 = strip * p.bx, y0 = tile * p.by;
    const int ny = (int)p.ny, nx = (int)p.nx;
    const int ylast = min(y0 + p.by, ny);
    const bool interior = y0 - K >= 0 && ylast + warp_rows_after(K) <= ny && x0 - p.H >= 0 && x0 - p.H + 32 * NC <= nx;
    const WarpWeights<STAR> ws([&](int i) { return p.w.w[i]; });
    if (interior) warp_tile<STAR, K, TS, NC, false, false, ALL>(p, ws, ring, lane, x0, y0);
    else if (ALL || NC == 8 || nx % NC == 0) warp_tile<STAR, K, TS, NC, true, false, ALL>(p, ws, ring, lane, x0, y0);
    else warp_tile<STAR, K, TS, NC, true, true, ALL>(p, ws, ring, lane, x0, y0);
}

}  // namespace gbst
