// sweep_stream_pad_bf16.cu -- streaming kernels on padded rows (widths that are not a
// multiple of 4, zero rule): bf16 storage.
#include "sweep_stream.cuh"

namespace gbst {

template <int R, bool STAR, int K>
static StreamKernelRef pad_ref() {
    return {(const void*)sweep_stream_kernel<R, STAR, K, __nv_bfloat16, true, false, true>, K};
}

// Kernel advancing exactly k steps ({nullptr, 0} if not instantiated): the depths of the kernels on
// dense rows, so a run is cut into the same launches (16-bit storage rounds once per launch).
StreamKernelRef get_stream_pad_kernel_bf16(int R, int star, int k) {
    switch (100 * R + 10 * star + k) {
        case 101: return pad_ref<1, false, 1>();
        case 102: return pad_ref<1, false, 2>();
        case 103: return pad_ref<1, false, 3>();
        case 104: return pad_ref<1, false, 4>();
        case 106: return pad_ref<1, false, 6>();
        case 108: return pad_ref<1, false, 8>();
        case 111: return pad_ref<1, true, 1>();
        case 112: return pad_ref<1, true, 2>();
        case 113: return pad_ref<1, true, 3>();
        case 114: return pad_ref<1, true, 4>();
        case 116: return pad_ref<1, true, 6>();
        case 118: return pad_ref<1, true, 8>();
        case 211: return pad_ref<2, true, 1>();
        case 212: return pad_ref<2, true, 2>();
        case 214: return pad_ref<2, true, 4>();
        case 311: return pad_ref<3, true, 1>();
        case 312: return pad_ref<3, true, 2>();
        case 313: return pad_ref<3, true, 3>();
        case 314: return pad_ref<3, true, 4>();
        case 201: return pad_ref<2, false, 1>();
        case 202: return pad_ref<2, false, 2>();
        case 204: return pad_ref<2, false, 4>();
        default: return {nullptr, 0};
    }
}

}  // namespace gbst
