// D3Q19 + D3Q7 fused step, FP16 and BF16 offset storage (FP32 collision).
#include "dispatch.h"

namespace tlbm {
cudaError_t launch_step_3d_f16(int prec, int vec, bool trt, int rows, const void* src, void* dst, const KParams& p,
                        dim3 grid, dim3 block, cudaStream_t s) {
    if (prec == 2) {
        TLBM_STEP_CASE(3, __half, 4, true)
        TLBM_STEPCAP_CASE(3, __half, 2, true, 96)
        TLBM_STEPCAP_CASE(3, __half, 1, true, 64)
        TLBM_STEP_CASE(3, __half, 4, false)
        TLBM_ROWS_CASE(3, __half, 1, 2)
        TLBM_ROWSCAP_CASE(3, __half, 1, 4, 128)
        TLBM_AACAP_CASE(3, __half, 2, true, 96)
        TLBM_AACAP_CASE(3, __half, 1, true, 64)
        TLBM_AA_CASE(3, __half, 2, false)
    } else {
        TLBM_STEP_CASE(3, __nv_bfloat16, 4, true)
        TLBM_STEPCAP_CASE(3, __nv_bfloat16, 2, true, 96)
        TLBM_STEPCAP_CASE(3, __nv_bfloat16, 1, true, 64)
        TLBM_STEP_CASE(3, __nv_bfloat16, 4, false)
        TLBM_ROWS_CASE(3, __nv_bfloat16, 1, 2)
        TLBM_ROWSCAP_CASE(3, __nv_bfloat16, 1, 4, 128)
        TLBM_AACAP_CASE(3, __nv_bfloat16, 2, true, 96)
        TLBM_AACAP_CASE(3, __nv_bfloat16, 1, true, 64)
        TLBM_AA_CASE(3, __nv_bfloat16, 2, false)
    }
    return cudaErrorInvalidValue;
}

// Halves of an in-place pair with one thread per node, nodes in their order in
// memory: 64 registers, and no lane idle at a row's end.  us per step, warps of
// node pairs inside rows -> this kernel: 33^3 7.5 -> 5.0, 65^3 16.4 -> 11.3, 97^3
// 34 -> 28, 129^3 78 -> 64, 193^3 220 -> 201, 257^3 481 -> 465, 385^3 1504 and 1515.
template <class S>
static cudaError_t launch_flat_aa(int mode, const void* src, void* dst, const KParams& p, cudaStream_t s) {
    if (mode == AA_EVEN) return launch_flat_as<3, S, AA_EVEN>(src, dst, p, s);
    if (mode == AA_ODD) return launch_flat_as<3, S, AA_ODD>(src, dst, p, s);
    return cudaErrorInvalidValue;
}
cudaError_t launch_flat_3d_f16(int prec, int mode, const void* src, void* dst, const KParams& p, cudaStream_t s) {
    return prec == 2 ? launch_flat_aa<__half>(mode, src, dst, p, s) : launch_flat_aa<__nv_bfloat16>(mode, src, dst, p, s);
}

const void* func_step_3d_f16(int prec, int vec, bool trt, int rows) {
    if (prec == 2) {
        TLBM_STEP_FUNC(3, __half, 4, true)
        TLBM_STEPCAP_FUNC(3, __half, 2, true, 96)
        TLBM_STEPCAP_FUNC(3, __half, 1, true, 64)
        TLBM_STEP_FUNC(3, __half, 4, false)
        TLBM_ROWS_FUNC(3, __half, 1, 2)
        TLBM_ROWSCAP_FUNC(3, __half, 1, 4, 128)
        TLBM_AACAP_FUNC(3, __half, 2, true, 96)
        TLBM_AACAP_FUNC(3, __half, 1, true, 64)
        TLBM_AA_FUNC(3, __half, 2, false)
    } else {
        TLBM_STEP_FUNC(3, __nv_bfloat16, 4, true)
        TLBM_STEPCAP_FUNC(3, __nv_bfloat16, 2, true, 96)
        TLBM_STEPCAP_FUNC(3, __nv_bfloat16, 1, true, 64)
        TLBM_STEP_FUNC(3, __nv_bfloat16, 4, false)
        TLBM_ROWS_FUNC(3, __nv_bfloat16, 1, 2)
        TLBM_ROWSCAP_FUNC(3, __nv_bfloat16, 1, 4, 128)
        TLBM_AACAP_FUNC(3, __nv_bfloat16, 2, true, 96)
        TLBM_AACAP_FUNC(3, __nv_bfloat16, 1, true, 64)
        TLBM_AA_FUNC(3, __nv_bfloat16, 2, false)
    }
    return nullptr;
}
}  // namespace tlbm
