// umma.cuh -- PTX helpers of the tcgen05 kernels: mbarriers with bounded waits,
// TMA copies, matrix descriptors, MMA issue, tensor-memory loads.
#pragma once

#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_runtime.h>

#include <cstdint>

#include "../../include/stencil.h"

namespace gbst {

constexpr int kUmRows = 128;            // M of one MMA
constexpr int kUmPlane = 2176;          // plane pitch: up to 136 rows x 16 B
constexpr int kUmAtom = 17408;          // swizzled atom pitch: up to 136 rows x 128 B
constexpr int kUmThreads = 192;         // 6 warps

// ---- PTX helpers ------------------------------------------------------------------------

__device__ __forceinline__ unsigned um_smem(const void* p) {
    return (unsigned)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ long long um_now() {
    long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ void um_bar_init(unsigned bar, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ void um_bar_arrive(unsigned bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void um_bar_expect_tx(unsigned bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

__device__ __forceinline__ bool um_bar_try(unsigned bar, unsigned parity) {
    unsigned ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

constexpr unsigned kUmWaitIters = 1u << 26;

// Wait for the phase of `parity` of `bar`.  Gives up when the CTA's abort flag
// is raised, or after `limit_ns` (then records a timeout and raises the flag).
__device__ __forceinline__ bool um_wait(unsigned bar, unsigned parity, volatile int* abort_flag,
                                        unsigned* status, long long limit_ns) {
    const long long t0 = um_now();
    for (unsigned it = 0;; ++it) {
        if (um_bar_try(bar, parity)) return true;
        if (*abort_flag) return false;
        if ((it & 63u) == 63u && (um_now() - t0 > limit_ns || it > kUmWaitIters)) {
            atomicCAS(status, 0u, (unsigned)STENCIL_ERR_TIMEOUT);
            *abort_flag = 1;
            return false;
        }
    }
}

// Bounded wait used while winding down (ignores the abort flag).
__device__ __forceinline__ void um_drain(unsigned bar, unsigned parity, unsigned* status, long long limit_ns) {
    const long long t0 = um_now();
    for (unsigned it = 0;; ++it) {
        if (um_bar_try(bar, parity)) return;
        if ((it & 63u) == 63u && (um_now() - t0 > limit_ns || it > kUmWaitIters)) {
            atomicCAS(status, 0u, (unsigned)STENCIL_ERR_TIMEOUT);
            return;
        }
    }
}

__device__ __forceinline__ void um_tma_2d(unsigned dst, const CUtensorMap* map, int x, int y, unsigned bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3}], [%4];" ::"r"(dst),
        "l"(map), "r"(x), "r"(y), "r"(bar)
        : "memory");
}

// Shared-memory matrix descriptor, K-major: start, LBO and SBO in 16-byte
// units; bits 46..48 hold the fixed value 0b001; no swizzle (layout 0).
__device__ __forceinline__ unsigned long long um_desc(unsigned saddr, unsigned lbo, unsigned sbo) {
    return (unsigned long long)((saddr >> 4) & 0x3FFFu) |
           ((unsigned long long)((lbo >> 4) & 0x3FFFu) << 16) |
           ((unsigned long long)((sbo >> 4) & 0x3FFFu) << 32) | (1ull << 46);
}

// The same for the 128-byte swizzle (layout type 2 in bits 61..63): SBO =
// 1024 B between 8-row groups, LBO unused within an atom (set to 16 B).  The
// tensor cores take the swizzle phase from the address bits, as the TMA unit
// does when it writes a 1024-byte aligned atom, so a start address moved by
// whole 128-byte rows (the row shift di) or by 32-byte K steps inside a row
// keeps base offset 0 (bits 49..51); the dyadic-exact tests fail with the
// start address's phase (start >> 7) & 7 in that field instead.
__device__ __forceinline__ unsigned long long um_desc_sw128(unsigned saddr) {
    return um_desc(saddr, 16, 1024) | (2ull << 61);
}

// Instruction descriptor: FP32 accumulator (bits 4-5 = 1), A/B format in bits
// 7-9 / 10-12 (BF16 = 1 under kind::f16, TF32 = 2 under kind::tf32), both
// operands K-major, N >> 3 in bits 17-22, M >> 4 in bits 24-28.
template <bool TF32>
__device__ __forceinline__ unsigned um_idesc_n(int n) {
    constexpr unsigned ab = TF32 ? 2u : 1u;
    return (1u << 4) | (ab << 7) | (ab << 10) | ((unsigned)(n >> 3) << 17) | ((unsigned)(kUmRows >> 4) << 24);
}

template <bool TF32, int NT>
__device__ __forceinline__ unsigned um_idesc() {
    return um_idesc_n<TF32>(NT);
}

template <bool TF32>
__device__ __forceinline__ void um_mma(unsigned tmem_d, unsigned long long adesc, unsigned long long bdesc,
                                       unsigned idesc, unsigned accumulate) {
    if constexpr (TF32) {
        asm volatile(
            "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
            "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
            : "memory");
    } else {
        asm volatile(
            "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
            "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
            : "memory");
    }
}

// Arrive on `bar` once every tcgen05 operation this thread issued so far is done.
__device__ __forceinline__ void um_commit(unsigned bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
                 : "memory");
}

// 32 consecutive FP32 accumulator columns of this thread's TMEM lane (no wait).
__device__ __forceinline__ void um_ld32(unsigned taddr, unsigned* r) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
}

__device__ __forceinline__ void um_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// Named barrier 1 over the NTH epilogue threads; returns the AND of `pred`.
template <int NTH = 128>
__device__ __forceinline__ int um_epi_and(int pred) {
    int r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\tsetp.ne.s32 p, %1, 0;\n\t"
        "bar.red.and.pred q, 1, %2, p;\n\tselp.s32 %0, 1, 0, q;\n\t}"
        : "=r"(r)
        : "r"(pred), "n"(NTH)
        : "memory");
    return r;
}

template <int NTH = 128>
__device__ __forceinline__ void um_epi_sync() { asm volatile("bar.sync 1, %0;" ::"n"(NTH) : "memory"); }

__device__ __forceinline__ void um_tma_store_2d(const CUtensorMap* map, unsigned src, int x, int y) {
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%1, %2}], [%3];" ::"l"(map),
                 "r"(x), "r"(y), "r"(src)
                 : "memory");
}

__device__ __forceinline__ void um_st_shared_v4(unsigned addr, unsigned a, unsigned b, unsigned c, unsigned d) {
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d)
                 : "memory");
}

__device__ __forceinline__ unsigned um_tf32(float x) {
    unsigned r;
    asm("cvt.rn.satfinite.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
    return r;
}

__device__ __forceinline__ void um_fence_before() {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void um_fence_after() {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

}  // namespace gbst
