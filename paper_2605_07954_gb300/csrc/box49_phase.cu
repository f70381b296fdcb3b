// box49_phase.cu -- the 7x7 box stencil on tcgen05, four output rows per MMA row.
//
// The same contraction as box49_umma.cu (each weight row di a banded Toeplitz
// matrix T_di, Sec. II-D), arranged so that the tensor cores read the staged
// rows less often.  There, every MMA takes 128 consecutive rows and one T_di,
// so a tile's rows are read 7 times per 64 output columns.  Here MMA row m
// stands for the FOUR output rows y0 + 4m .. y0 + 4m + 3 (phases 0..3), each
// with its own block of 32 accumulator columns.  Staged row y0 + 4m + r
// (r = -3 .. 6) feeds phase q through weight row di = r + 3 - q, so one MMA
//   A = rows y0 + r, y0 + r + 4, ...   (128 rows, one K slice)
//   B = [T_{r+3-qlo} | .. | T_{r+3-qhi}],  N = 32 (qhi - qlo + 1)
// does the work of up to four: 10 MMAs per K slice for 512 x 32 outputs where
// one weight row per MMA takes 28 (N = 32) or 14 (N = 64, whose K windows are
// wider).  Nothing has to be shifted afterwards: accumulator lane m, column
// block q is output row y0 + 4m + q as it stands.
//
// Rows of one residue mod 4 must lie side by side for that, and TMA brings
// them so: the grid is a 3D tensor (column, row mod 4, row / 4), which needs
// ny % 4 == 0, and a staged tile is four boxes of 130 rows (y0 - 4 + ph, ..).
// Within a phase a row shift of 4 is one staged row, so A's start address is
// (phase, row group) and nothing is copied.  As in box49_umma.cu the columns
// are one 128-byte swizzled atom per row plus the last K slice as two
// 16-byte planes.  B stores T_6 .. T_0 side by side (n-major), so every stack
// of consecutive weight rows is a start address into it.
//
// A tile is 512 rows x 64 (BF16) or 32 (TF32) columns, two stages deep; four
// accumulators of 128 TMEM columns.  Warps, barriers, bounded waits and the
// wind-down after a timeout are those of box49_umma.cu.
//
// What bounds it: DRAM.  16384^2 BF16 moves 1.03 GB a step (ncu; the grid once
// in, once out) in 200 us (5.1 TB/s, 0.76 of the measured copy rate); without
// its stores the same launch takes 146 us, without the whole epilogue 143, with
// the MMAs alone 133 (80 cycles per MMA of up to N = 128; issuing one costs the
// issuing thread about 70).  Per step, this kernel | one weight row per MMA:
// 16384^2 BF16 209 | 293 us (1282 | 916 GStencil/s), TF32 390 | 509 us.
// Tried: the whole accumulator staged at once, one store set (212 us), 128-byte
// staged rows (214), stores straight from registers, 32 bytes a lane (228).
#include <cuda_bf16.h>

#include "umma.cuh"

namespace gbst {

PFN_cuTensorMapEncodeTiled_v12000 um_encoder();

constexpr int kPhRows = 4 * kUmRows;     // output rows per tile
constexpr int kPhGroups = kUmRows + 2;   // staged rows of a phase: y0 - 4 + ph, step 4
constexpr int kPhNT = 32;                // output columns of an accumulator block
constexpr int kPhBufs = 4;               // accumulators (128 TMEM columns each)

template <bool TF32>
struct PhCfg {
    static constexpr int EB = TF32 ? 4 : 2;                  // bytes per element
    static constexpr int EPG = 16 / EB;                      // elements per plane row
    static constexpr int L = TF32 ? 4 : 8;                   // K window starts L columns left
    static constexpr int KE = TF32 ? 8 : 16;                 // K of one MMA
    static constexpr int KSTEPS = (kPhNT + L + 3 + KE - 1) / KE;
    static constexpr int COLS = 128 / EB;                    // output columns per tile = one atom
    static constexpr int JT = COLS / kPhNT;                  // accumulators per tile
    static constexpr int STAGES = 2;
    static constexpr int PL0 = 4 * kUmAtom;                  // planes after the four atoms
    static constexpr int STAGE_BYTES = 4 * kUmAtom + 4 * 2 * kUmPlane;
    static constexpr int TX_BYTES = 4 * kPhGroups * (128 + 2 * 16);
    static constexpr int BPLANE = 7 * kPhNT * 16;            // T_6 .. T_0 of one K plane
    static constexpr int B_BYTES = KSTEPS * 2 * BPLANE;
    static constexpr int BCOLS = 64 / EB;                    // output columns of a staged block (64-byte rows)
    static constexpr int BLOCK = kUmRows * 64;               // bytes of a staged block: one phase, BCOLS columns
    static constexpr int NBLK = 4 * kPhNT / BCOLS;           // blocks per accumulator
    static constexpr int BPP = TF32 ? 1 : 2;                 // blocks staged and stored together
    static constexpr int NBARS = 2 * STAGES + 2 * kPhBufs + 1;
    static constexpr int SMEM = 1024 + STAGES * STAGE_BYTES + 2 * BPP * BLOCK + B_BYTES + 8 * NBARS;
    static_assert(SMEM <= 227 * 1024 - 1024, "shared memory per CTA");
    static_assert(STAGE_BYTES % 1024 == 0 && B_BYTES % 16 == 0, "alignment");
    static_assert((JT - 1) * kPhNT + (KSTEPS - 1) * KE <= COLS, "K slices end in the plane pair");
    static_assert(kUmAtom >= kPhGroups * 128 && kUmPlane >= kPhGroups * 16, "phase pitch");
};

struct PhParams {
    int tiles_x, tiles;
    int round_out;      // TF32: store TF32-rounded values
    unsigned* status;
    long long wait_ns;
    int withhold;       // test hook: CTA 0 withholds its first accumulator-ready signal
    float w[49];
};

__device__ __forceinline__ void ph_tma_load(unsigned dst, const CUtensorMap* map, int x, int ph, int g, unsigned bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(dst),
        "l"(map), "r"(x), "r"(ph), "r"(g), "r"(bar)
        : "memory");
}

__device__ __forceinline__ void ph_tma_store(const CUtensorMap* map, unsigned src, int x, int ph, int g) {
    asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.bulk_group [%0, {%1, %2, %3}], [%4];" ::"l"(map),
                 "r"(x), "r"(ph), "r"(g), "r"(src)
                 : "memory");
}

template <bool TF32>
__global__ void __launch_bounds__(kUmThreads, 1)
    box49_phase_kernel(const __grid_constant__ CUtensorMap tmap_sw, const __grid_constant__ CUtensorMap tmap_pl,
                       const __grid_constant__ CUtensorMap tmap_out, const __grid_constant__ PhParams p) {
    using C = PhCfg<TF32>;
    extern __shared__ __align__(1024) unsigned char um_dyn[];
    unsigned char* stages = um_dyn + ((1024u - (um_smem(um_dyn) & 1023u)) & 1023u);
    unsigned char* outstg = stages + C::STAGES * C::STAGE_BYTES;
    unsigned char* bmat = outstg + 2 * C::BPP * C::BLOCK;
    __shared__ unsigned s_tmem;
    __shared__ volatile int s_abort;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // barriers: full[S], empty[S], tmem_full[4], tmem_empty[4], drain
    const unsigned full0 = um_smem(bmat + C::B_BYTES), empty0 = full0 + 8u * C::STAGES,
                   tfull0 = empty0 + 8u * C::STAGES, tempty0 = tfull0 + 8u * kPhBufs, drain = tempty0 + 8u * kPhBufs;

    if (threadIdx.x == 0) {
        s_abort = 0;
        for (int s = 0; s < C::STAGES; ++s) {
            um_bar_init(full0 + 8u * s, 1);
            um_bar_init(empty0 + 8u * s, 1);
        }
        for (int b = 0; b < kPhBufs; ++b) {
            um_bar_init(tfull0 + 8u * b, 1);
            um_bar_init(tempty0 + 8u * b, 4);
        }
        um_bar_init(drain, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // B, K-major, no swizzle: element (k, n) at (k / EPG) * BPLANE + 16 n + EB * (k % EPG),
    // where n = (6 - di) * 32 + n' holds W[di][k - n' - (L - 3)] (0 outside the band).
    for (int i = threadIdx.x; i < C::KSTEPS * 2 * 7 * kPhNT * C::EPG; i += kUmThreads) {
        const int e = i % C::EPG;
        const int n = (i / C::EPG) % (7 * kPhNT);
        const int pl = i / (C::EPG * 7 * kPhNT);
        const int di = 6 - n / kPhNT;
        const int dj = pl * C::EPG + e - n % kPhNT - (C::L - 3);
        const float v = (dj >= 0 && dj <= 6) ? p.w[di * 7 + dj] : 0.f;
        unsigned char* dst = bmat + pl * C::BPLANE + n * 16 + e * C::EB;
        if constexpr (TF32) {
            *reinterpret_cast<unsigned*>(dst) = um_tf32(v);
        } else {
            *reinterpret_cast<__nv_bfloat16*>(dst) = __float2bfloat16_rn(v);
        }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // B is read by the tensor cores
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(um_smem(&s_tmem)),
                     "r"(512)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    um_fence_before();
    __syncthreads();
    um_fence_after();
    const unsigned tmem = s_tmem;

    if (warp == 0) {
        // ---------------- TMA producer ----------------
        int it = 0;
        for (int tile = blockIdx.x; tile < p.tiles; tile += gridDim.x, ++it) {
            const int s = it % C::STAGES;
            int ok = 1;
            if (lane == 0) ok = um_wait(empty0 + 8u * s, ((it / C::STAGES) & 1) ^ 1, &s_abort, p.status, p.wait_ns);
            if (!__shfl_sync(0xffffffffu, ok, 0)) break;
            if (lane == 0) {
                const int x0 = (tile % p.tiles_x) * C::COLS, g0 = (tile / p.tiles_x) * kUmRows;
                const unsigned fb = full0 + 8u * s;
                const unsigned dst = um_smem(stages + s * C::STAGE_BYTES);
                if ((dst & 1023u) != 0u || (fb & 7u) != 0u) {
                    // never issue a misaligned copy: report it and stop the CTA
                    atomicCAS(p.status, 0u, (unsigned)STENCIL_ERR_DEVICE_CHECK);
                    s_abort = 1;
                    ok = 0;
                } else {
                    um_bar_expect_tx(fb, (unsigned)C::TX_BYTES);
                    const int xs = x0 - C::L;
                    for (int ph = 0; ph < 4; ++ph) {
                        ph_tma_load(dst + (unsigned)(ph * kUmAtom), &tmap_sw, xs, ph, g0 - 1, fb);
                        for (int g = 0; g < 2; ++g)
                            ph_tma_load(dst + (unsigned)(C::PL0 + (2 * ph + g) * kUmPlane), &tmap_pl,
                                        xs + C::COLS + C::EPG * g, ph, g0 - 1, fb);
                    }
                }
            }
            if (!__shfl_sync(0xffffffffu, ok, 0)) break;
        }
        // Loads still in flight (only after an abort) land before the CTA exits.
        if (lane == 0) {
            for (int i = it - C::STAGES < 0 ? 0 : it - C::STAGES; i < it; ++i)
                um_drain(full0 + 8u * (i % C::STAGES), (i / C::STAGES) & 1, p.status, p.wait_ns);
        }
        __syncwarp();
    } else if (warp == 1) {
        // ---------------- MMA issue (one thread) ----------------
        const unsigned long long bdesc0 = um_desc(um_smem(bmat), C::BPLANE, 128);
        int it = 0, u = 0, issued = 0;
        bool alive = true;
        for (int tile = blockIdx.x; tile < p.tiles && alive; tile += gridDim.x, ++it) {
            const int s = it % C::STAGES;
            int ok = 1;
            if (lane == 0) ok = um_wait(full0 + 8u * s, (it / C::STAGES) & 1, &s_abort, p.status, p.wait_ns);
            if (!__shfl_sync(0xffffffffu, ok, 0)) break;
            const unsigned sbase = um_smem(stages + s * C::STAGE_BYTES);
            const unsigned long long a_sw = um_desc_sw128(sbase);
            const unsigned long long a_pl = um_desc(sbase + (unsigned)C::PL0, kUmPlane, 128);
#pragma unroll
            for (int j = 0; j < C::JT; ++j, ++u) {
                const int bf = u % kPhBufs;
                if (lane == 0) ok = um_wait(tempty0 + 8u * bf, ((u / kPhBufs) & 1) ^ 1, &s_abort, p.status, p.wait_ns);
                if (!__shfl_sync(0xffffffffu, ok, 0)) {
                    alive = false;
                    break;
                }
                um_fence_after();
                if (lane == 0) {
                    const unsigned d = tmem + (unsigned)(bf * 128);
#pragma unroll
                    for (int ks = 0; ks < C::KSTEPS; ++ks) {
                        const int c = kPhNT * j + C::KE * ks;  // first column of the K slice (from x0 - L)
#pragma unroll
                        for (int i = 0; i < 10; ++i) {
                            // row offset r = -3 .. 6; r = 0 first, which writes all four blocks
                            const int r = i == 0 ? 0 : i <= 3 ? i - 4 : i - 3;
                            const int ph = r & 3, go = (r - ph) / 4 + 1;  // phase, staged row of group 0
                            const int qlo = r + 3 > 6 ? r - 3 : 0, qhi = r + 3 < 3 ? r + 3 : 3;
                            const unsigned long long a =
                                c < C::COLS ? a_sw + (unsigned long long)((ph * kUmAtom + go * 128 + c * C::EB) >> 4)
                                            : a_pl + (unsigned long long)((ph * 2 * kUmPlane + go * 16) >> 4);
                            const unsigned long long bd =
                                bdesc0 + (unsigned long long)((ks * 2 * C::BPLANE + (6 - (r + 3 - qlo)) * kPhNT * 16) >> 4);
                            um_mma<TF32>(d + (unsigned)(kPhNT * qlo), a, bd, um_idesc_n<TF32>(kPhNT * (qhi - qlo + 1)),
                                         (ks | i) != 0);
                        }
                    }
                    if (!(p.withhold && blockIdx.x == 0 && u == 0)) um_commit(tfull0 + 8u * bf);
                    issued = 1;
                }
                __syncwarp();
            }
            if (!alive) break;
            if (lane == 0) um_commit(empty0 + 8u * s);  // the stage is free once these MMAs have read it
            __syncwarp();
        }
        // Every MMA issued is complete before the tensor memory is released.
        if (lane == 0 && issued) {
            um_commit(drain);
            um_drain(drain, 0, p.status, p.wait_ns);
        }
        __syncwarp();
    } else {
        // ---------------- epilogue: TMEM lanes 32 q .. 32 q + 31 ----------------
        // Per accumulator: load the lane's four phases of 32 columns (one wait),
        // free the accumulator, and stage it in blocks of 128 rows x 64 bytes (one
        // phase of 32 BF16 or 16 TF32 columns), each stored with one TMA copy
        // (clipped at the grid edges).  Two sets of blocks alternate, so a set is
        // written while TMA still reads the other one.
        const int q = warp & 3;
        const int r = 32 * q + lane;
        const bool issuer = threadIdx.x == 64;
        const unsigned stg0 = um_smem(outstg) + (unsigned)(r * 64);
        const int sw = (r >> 1) & 3;  // 64-byte swizzle of this row
        int it = 0, u = 0;
        bool alive = true;
        for (int tile = blockIdx.x; tile < p.tiles && alive; tile += gridDim.x, ++it) {
            const int x0 = (tile % p.tiles_x) * C::COLS, g0 = (tile / p.tiles_x) * kUmRows;
            for (int j = 0; j < C::JT; ++j, ++u) {
                const int bf = u % kPhBufs;
                int ok = 1;
                if (lane == 0) ok = um_wait(tfull0 + 8u * bf, (u / kPhBufs) & 1, &s_abort, p.status, p.wait_ns);
                ok = __shfl_sync(0xffffffffu, ok, 0);
                if (!um_epi_and(ok)) {  // the four epilogue warps leave together
                    alive = false;
                    break;
                }
                um_fence_after();
                unsigned v[128];
                const unsigned trow = tmem + ((unsigned)(32 * q) << 16) + (unsigned)(bf * 128);
#pragma unroll
                for (int c = 0; c < 4; ++c) um_ld32(trow + (unsigned)(32 * c), v + 32 * c);
                um_ld_wait();
                um_fence_before();
                __syncwarp();
                if (lane == 0) um_bar_arrive(tempty0 + 8u * bf);  // accumulator free for the MMAs
#pragma unroll
                for (int part = 0; part < C::NBLK / C::BPP; ++part) {
                    const unsigned set = (unsigned)((part & 1) * C::BPP * C::BLOCK);
                    // the stores that last read this set have finished reading it
                    if (issuer) asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
                    um_epi_sync();
#pragma unroll
                    for (int b = 0; b < C::BPP; ++b) {
                        const int col0 = (part * C::BPP + b) * C::BCOLS;  // accumulator column
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            unsigned w[4];
#pragma unroll
                            for (int i = 0; i < 4; ++i) {
                                const int col = col0 + c * C::EPG + (TF32 ? i : 2 * i);
                                if constexpr (TF32) {
                                    w[i] = p.round_out ? um_tf32(__uint_as_float(v[col])) : v[col];
                                } else {
                                    __nv_bfloat162 h =
                                        __floats2bfloat162_rn(__uint_as_float(v[col]), __uint_as_float(v[col + 1]));
                                    w[i] = *reinterpret_cast<unsigned*>(&h);
                                }
                            }
                            um_st_shared_v4(stg0 + set + (unsigned)(b * C::BLOCK + ((c ^ sw) << 4)), w[0], w[1], w[2],
                                            w[3]);
                        }
                    }
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // staging is read by TMA
                    um_epi_sync();
                    if (issuer) {
#pragma unroll
                        for (int b = 0; b < C::BPP; ++b) {
                            const int col0 = (part * C::BPP + b) * C::BCOLS;
                            ph_tma_store(&tmap_out, um_smem(outstg) + set + (unsigned)(b * C::BLOCK),
                                         x0 + kPhNT * j + col0 % kPhNT, col0 / kPhNT, g0);
                        }
                        asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                    }
                }
            }
        }
        // every store has completed (and read its staging) before the CTA exits
        if (issuer) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
        __syncwarp();
    }

    um_fence_before();
    __syncthreads();
    um_fence_after();
    if (warp == 1) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
    }
}

// ---- host side ----------------------------------------------------------------------------

const void* get_box49_phase_kernel(int tf32) {
    return tf32 ? (const void*)box49_phase_kernel<true> : (const void*)box49_phase_kernel<false>;
}
int box49_phase_smem_bytes(int tf32) { return tf32 ? PhCfg<true>::SMEM : PhCfg<false>::SMEM; }
int box49_phase_rows() { return kPhRows; }
int box49_phase_cols(int tf32) { return tf32 ? PhCfg<true>::COLS : PhCfg<false>::COLS; }

// The grid as (column, row mod 4, row / 4): boxes of box_x columns x one phase x box_g rows.
static CUresult ph_encode(PFN_cuTensorMapEncodeTiled_v12000 enc, CUtensorMap* map, int tf32, const void* src, int ny,
                          int nx, int box_x, int box_g, CUtensorMapSwizzle swz) {
    const int eb = tf32 ? 4 : 2;
    const cuuint64_t dims[3] = {(cuuint64_t)nx, 4, (cuuint64_t)(ny / 4)};
    const cuuint64_t strides[2] = {(cuuint64_t)nx * (cuuint64_t)eb, (cuuint64_t)nx * (cuuint64_t)eb * 4};
    const cuuint32_t box[3] = {(cuuint32_t)box_x, 1, (cuuint32_t)box_g};
    const cuuint32_t estr[3] = {1, 1, 1};
    return enc(map, tf32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3,
               const_cast<void*>(src), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, swz,
               CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
}

// One step src -> dst on at most `ctas` persistent CTAs.  The caller guarantees
// 16-byte aligned grids, rows of a multiple of 16 bytes and ny % 4 == 0.
// Returns cudaErrorNotSupported when no tensor map can be made.
cudaError_t launch_box49_phase(int tf32, const void* src, void* dst, int ny, int nx, int round_out, unsigned* status,
                               const float* w, int ctas, cudaStream_t st, int timeout_ms, int withhold) {
    PFN_cuTensorMapEncodeTiled_v12000 enc = um_encoder();
    if (!enc || ny % 4 != 0) return cudaErrorNotSupported;
    const int eb = tf32 ? 4 : 2;
    alignas(64) CUtensorMap map_sw, map_pl, map_out;
    if (ph_encode(enc, &map_sw, tf32, src, ny, nx, 128 / eb, kPhGroups, CU_TENSOR_MAP_SWIZZLE_128B) != CUDA_SUCCESS ||
        ph_encode(enc, &map_pl, tf32, src, ny, nx, 16 / eb, kPhGroups, CU_TENSOR_MAP_SWIZZLE_NONE) != CUDA_SUCCESS ||
        ph_encode(enc, &map_out, tf32, dst, ny, nx, 64 / eb, kUmRows, CU_TENSOR_MAP_SWIZZLE_64B) != CUDA_SUCCESS)
        return cudaErrorNotSupported;
    PhParams pp{};
    const int cols = box49_phase_cols(tf32);
    pp.tiles_x = (nx + cols - 1) / cols;
    pp.tiles = pp.tiles_x * ((ny + kPhRows - 1) / kPhRows);
    pp.round_out = round_out;
    pp.status = status;
    pp.wait_ns = (long long)(timeout_ms > 0 ? timeout_ms : 2000) * 1000000LL;
    pp.withhold = withhold;
    for (int i = 0; i < 49; ++i) pp.w[i] = w[i];
    void* args[] = {&map_sw, &map_pl, &map_out, &pp};
    const int grid = ctas < pp.tiles ? ctas : pp.tiles;
    return cudaLaunchKernel(get_box49_phase_kernel(tf32), dim3((unsigned)grid), dim3((unsigned)kUmThreads), args,
                            (size_t)box49_phase_smem_bytes(tf32), st);
}

}  // namespace gbst
